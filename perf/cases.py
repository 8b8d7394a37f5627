"""Measured cases of the DZS TreePM library: what its users have it do, through
its public entry points (include/dzs.h, the Python binding), at the sizes of
its configurations (32^3 .. 256^3 particles, meshes of one or two points per
particle and side).

Kinds of case:
  resume   one global KDK step of a halted run (paper Sec. 4.1.1): the state is
           restored from its checkpoint in pinned host memory, one full step
           runs (kick, drift, crossing, sort, DZS merge, tree, PM, walk), and
           the new checkpoint is written to pinned host memory.  Every pass
           starts from the same checkpoint, so every pass does the same work.
  batch    the same for several mocks stepped together by dzs_batch_step.
  accel    accelerations of a resident particle set (dzs_accel).
  pk       the time-slice power spectrum (dzs_power_spectrum).
  fof      the friends-of-friends catalogue of a clustered set (dzs_fof).
  alm      the harmonic analysis of a lightcone sky map (dzs_skymap_alm).
  sort     the allocation-free Morton sort of device positions.

Particle sets come from the seed alone: a Gaussian displacement field with the
library's spectrum shape on the particle lattice, growing with the expansion
factor of the case's step, and, as it grows, Lagrangian patches of 8, 64 and
512 particles collapsed to haloes.  The set is put in Morton order, as a step
leaves it, and with DZS on it is merged against the step's lightcone first (an
exact integer operation), as in a run that has reached that step.
"""
import ctypes
import math

import numpy as np
import torch

import paper_2005_05328_gb300 as dzs

DEV = "cuda:0"
TWO32 = 4294967296.0
OMEGA_M, OMEGA_L, HUBBLE, NS, Z_INIT = 0.3, 0.7, 0.7, 0.96, 49.0
LEAF, GROUP, THETA, RS_CELLS, RCUT_RS, SOFT = 8, 32, 0.5, 1.25, 4.5, 1.0 / 40.0
THETA_DZS, BUFFER_CELLS, ALPHA_DYN = 0.1, 2.0, 0.01
NSTEPS = 96
BOX_PER_N1D = 2.0  # L = 2 n1d Mpc/h in every configuration
BATCH_SIZES = (32, 48, 64, 96)


def _resume(n1d, mesh, step, **kw):
    case = dict(kind="resume", n1d=n1d, mesh=mesh, step=step, fp64=False, dzs=True, dynamical=False,
                physical=False, merge_level=3)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest call: the positions of a small plugin or tile, on a caller's stream
        dict(name="sort_20k", kind="sort", n=20011),
        # the plain FP64 configuration, 32^3 in 64 Mpc/h, mesh 64, at an ordinary early step
        dict(_resume(32, 64, 20, fp64=True, merge_level=2), name="resume_32_fp64"),
        # a late, clustered and half merged 48^3 mock of the batched mix (mesh 3 2^5), dynamical criterion
        dict(_resume(48, 96, 70, dynamical=True), name="resume_48_late"),
        # the batched configuration: mocks of 32^3 .. 96^3 advancing together, two of each size
        dict(name="batch_8", kind="batch", per_size=2, step=36),
        # the 128^3 / 256^3 configuration early in the run (z ~ 30): hardly clustered, nothing merged
        dict(_resume(128, 256, 12), name="resume_128_early"),
        # the same late in the run (z ~ 1): haloes, merged particles, a ragged particle count
        dict(_resume(128, 256, 78), name="resume_128_late"),
        # FP64 forces of a 64^3 set: the reference path users check FP32 against
        dict(name="accel_64_fp64", kind="accel", n1d=64, mesh=128, step=40, fp64=True),
        # the largest mock of the serving mix, 256^3 with mesh 512
        dict(_resume(256, 512, 8), name="resume_256"),
        # the regime of the 512^3 configuration (one mesh point per particle, merge level 4,
        # lightcone at the physical comoving distance) at 256^3
        dict(_resume(256, 256, 16, physical=True, merge_level=4), name="resume_256_mesh256"),
        # P(k) of a 256^3 set on mesh 512, every bin to the Nyquist frequency
        dict(name="pk_256", kind="pk", n1d=256, mesh=512, step=60, nbins=256),
        # halo catalogue of a clustered 128^3 output, the usual linking length
        dict(name="fof_128", kind="fof", n1d=128, mesh=256, step=90, link=0.2, nmin=20),
        # C_l of the Nside 256 sky map to l = 512
        dict(name="alm_256", kind="alm", nside=256, lmax=512, records=400000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sort", "resume", "resume", "resume", "accel", "pk", "fof", "alm"])
    if kind == "sort":
        return dict(kind="sort", n=_log_int(rng, 1000, dzs.NOALLOC_SORT_MAX_N))
    if kind == "alm":
        nside = rng.choice([32, 64, 128, 256])
        return dict(kind="alm", nside=nside, lmax=rng.randrange(nside // 2, 2 * nside + 1),
                    records=_log_int(rng, 1000, 400000))
    n1d = rng.choice([16, 24, 32, 48, 64, 96, 128, 192])
    step = rng.randrange(2, NSTEPS - 3)
    mesh = n1d * rng.choice([1, 2, 2])
    if kind == "resume":
        return _resume(n1d, mesh, step, fp64=n1d <= 64 and rng.random() < 0.3, dzs=rng.random() < 0.8,
                       dynamical=rng.random() < 0.3,
                       physical=n1d <= 128 and rng.random() < 0.3, merge_level=rng.choice([1, 2, 3, 4]))
    if kind == "accel":
        return dict(kind="accel", n1d=n1d, mesh=mesh, step=step, fp64=n1d <= 64 and rng.random() < 0.5)
    if kind == "pk":
        return dict(kind="pk", n1d=n1d, mesh=mesh, step=step, nbins=rng.randrange(mesh // 4, mesh // 2 + 1))
    return dict(kind="fof", n1d=max(32, n1d), mesh=2 * max(32, n1d), step=rng.randrange(64, NSTEPS), link=rng.choice([0.15, 0.17, 0.2, 0.25]),
                nmin=rng.choice([10, 20, 32]))


# ---------------------------------------------------------------- the run's tables, FP64


def _quad(f, lo, hi, panels):
    x, w = np.polynomial.legendre.leggauss(20)
    h = (hi - lo) / panels
    mid = lo + h * (np.arange(panels) + 0.5)
    return float((f(mid[:, None] + 0.5 * h * x[None, :]) * w[None, :]).sum() * 0.5 * h)


def _e_of(a):
    return np.sqrt(OMEGA_M / a ** 3 + (1.0 - OMEGA_M - OMEGA_L) / a ** 2 + OMEGA_L)


def _chi(a):
    return 2997.92458 * _quad(lambda s: np.exp(-s) / _e_of(np.exp(s)), math.log(a), 0.0, 256)


def _tables(box, step, physical):
    """a, drift, kick factors and lattice lightcone radii around one step"""
    lnai = -math.log1p(Z_INIT)
    dl = -lnai / NSTEPS
    a0, a1 = math.exp(lnai + step * dl), 1.0 if step + 1 == NSTEPS else math.exp(lnai + (step + 1) * dl)
    ah = math.exp(lnai + (step + 0.5) * dl)
    la, lh, lb = math.log(a0), math.log(ah), math.log(a1)

    def kick_f(s):
        return 1.0 / (np.exp(s) * _e_of(np.exp(s)))

    rmax = math.sqrt(3.0) * box / 2.0
    chi0 = _chi(math.exp(lnai))
    rlat = []
    for a in (a0, a1):
        r = min(_chi(a), rmax) if physical else rmax * _chi(a) / chi0
        rlat.append(int(math.floor(r / box * TWO32)))
    return dict(a0=a0, a1=a1, drift=_quad(lambda s: 1.0 / (np.exp(2 * s) * _e_of(np.exp(s))), la, lb, 8),
                kick1=_quad(kick_f, la, lh, 8), kick2=_quad(kick_f, lh, lb, 8), rlat0=rlat[0], rlat1=rlat[1])


# ---------------------------------------------------------------- particle sets


def _spread3(v):
    x = v & 0x1FFFFF
    for s, m in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                 (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        x = (x | (x << s)) & m
    return x


def _morton(u):
    """63-bit keys of lattice positions u [3][n] (int64)"""
    return (_spread3(u[0] >> 11) << 2) | (_spread3(u[1] >> 11) << 1) | _spread3(u[2] >> 11)


def _wrap(d):
    """signed minimum-image lattice difference"""
    return torch.remainder(d + 2 ** 31, 2 ** 32) - 2 ** 31


def _gauss_field(n1, gen):
    """displacement field [3][n1^3] with the BBKS shape, unit rms per axis"""
    w = torch.fft.rfftn(torch.randn((n1, n1, n1), generator=gen, device=DEV, dtype=torch.float64))
    kf = 2.0 * math.pi / (BOX_PER_N1D * n1)
    kx = torch.fft.fftfreq(n1, 1.0 / n1, device=DEV, dtype=torch.float64) * kf
    kz = torch.arange(n1 // 2 + 1, device=DEV, dtype=torch.float64) * kf
    k2 = kx[:, None, None] ** 2 + kx[None, :, None] ** 2 + kz[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    k = torch.sqrt(k2)
    q = k / (OMEGA_M * HUBBLE)
    t = torch.log(1.0 + 2.34 * q) / (2.34 * q) * (1.0 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3
                                                 + (6.71 * q) ** 4) ** -0.25
    w = w * torch.sqrt(k ** NS) * t / k2
    w[0, 0, 0] = 0.0
    out = []
    for ka in (kx[:, None, None], kx[None, :, None], kz[None, None, :]):
        f = torch.fft.irfftn(1j * ka * w, s=(n1, n1, n1))
        out.append((f / f.square().mean().sqrt()).reshape(-1))
    return torch.stack(out)


def _particles(n1, step, physical, seed):
    """state at a step of a run, in Morton order: u (int64), p, g (float64), id
    and crossed flags, on the GPU"""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) * 1000003 + 17 * n1 + step)
    box = BOX_PER_N1D * n1
    tab = _tables(box, step, physical)
    a = tab["a0"]
    n = n1 ** 3
    i = torch.arange(n, device=DEV)
    q = torch.stack([i // (n1 * n1), (i // n1) % n1, i % n1])
    psi = _gauss_field(n1, gen) * (1.75 * a)  # spacings
    x = q.to(torch.float64) + psi
    move = psi * 0.04  # displacement of one step, spacings
    collapsed = 0.5 * min(1.0, max(0.0, (a - 0.15) / 0.85))
    for s in (2, 4, 8):
        if collapsed == 0.0 or n1 % s:
            continue
        m = n1 // s
        patch = ((q[0] // s) * m + q[1] // s) * m + q[2] // s
        pick = torch.rand(m ** 3, generator=gen, device=DEV) < collapsed / 3.0
        centre = (q // s).to(torch.float64) * s + 0.5 * (s - 1)
        mean = torch.zeros((3, m ** 3), device=DEV, dtype=torch.float64)
        corner = ((q % s) == 0).all(0)  # one member's displacement moves the patch
        mean[:, patch[corner]] = psi[:, corner]
        r = 0.106 * s * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
        d = torch.randn((3, n), generator=gen, device=DEV, dtype=torch.float64)
        d = d / d.square().sum(0).sqrt()
        sel = pick[patch]
        x = torch.where(sel, centre + mean[:, patch] + r * d, x)
        kick = torch.randn((3, n), generator=gen, device=DEV, dtype=torch.float64) * (0.01 * s)
        move = torch.where(sel, mean[:, patch] * 0.04 + kick, move)
    u = torch.remainder(torch.round(x * (TWO32 / n1)).to(torch.int64), 2 ** 32)
    p = move * (BOX_PER_N1D / tab["drift"])
    g = p * (0.03 / tab["kick1"])
    order = torch.argsort(_morton(u), stable=True)
    u, p, g, ident = u[:, order], p[:, order], g[:, order], order
    crossed = _dist_far(u, tab["rlat0"])
    return dict(u=u, p=p, g=g, id=ident, fl=crossed.to(torch.uint8), tab=tab)


def _dist_far(u, rlat):
    """distance from the observer at 2^31 at least rlat"""
    d = (u - 2 ** 31).to(torch.float64)
    return d.square().sum(0) >= float(rlat) ** 2


def _context(n1, mesh, fp64=False, dzs_on=True, dynamical=False, physical=False, merge_level=3):
    return dzs.Context(n1d=n1, mesh=mesh, box=BOX_PER_N1D * n1, nsteps=NSTEPS, dzs_on=int(dzs_on),
                       merge_level=merge_level, precision=dzs.FP64 if fp64 else dzs.FP32,
                       rlc_mode=dzs.RLC_PHYSICAL if physical else dzs.RLC_SWEEP,
                       dzs_criterion=dzs.CRIT_DYNAMICAL if dynamical else dzs.CRIT_GEOMETRIC)


def _host_state(s, k=None):
    n = s["u"].shape[1]
    return dict(u=s["u"].to(torch.int32).cpu().numpy().view(np.uint32) if n else np.zeros((3, 0), np.uint32),
                p=s["p"].cpu().numpy(), g=s["g"].cpu().numpy(),
                k=np.ones(n, np.uint32) if k is None else k, id=s["id"].to(torch.int32).cpu().numpy().view(np.uint32),
                fl=s["fl"].cpu().numpy())


def _run_state(ctx, n1, step, physical, dynamical, dzs_on, seed):
    """load the state of a run that reached `step` into ctx; returns it as host arrays"""
    s = _particles(n1, step, physical, seed)
    st = _host_state(s)
    ctx.set_state(st, step)
    if dzs_on:
        ctx.merge_only(s["tab"]["rlat0"])
        got = ctx.state()
        of = torch.empty(n1 ** 3, dtype=torch.int64, device=DEV)
        of[s["id"]] = torch.arange(n1 ** 3, device=DEV)
        row = of[torch.from_numpy(got["id"].astype(np.int64)).to(DEV)]
        got["g"] = s["g"][:, row].cpu().numpy()  # the accelerations of the surviving particles
        st = got
        ctx.set_state(st, step)
    return st, s["tab"]


def _check(status, ctx):
    if status != dzs.DZS_OK:
        msg = dzs.load().dzs_last_error(ctx.h)
        raise dzs.DzsError(status, msg.decode() if msg else "")


class _Halted:
    """A context and the pinned checkpoint its run was halted with."""

    def __init__(self, case, seed):
        self.fp64 = case["fp64"]
        self.ctx = _context(case["n1d"], case["mesh"], case["fp64"], case["dzs"], case["dynamical"],
                            case["physical"], case["merge_level"])
        _run_state(self.ctx, case["n1d"], case["step"], case["physical"], case["dynamical"], case["dzs"], seed)
        lib, h, n0 = dzs.load(), self.ctx.h, case["n1d"] ** 3
        size = ctypes.c_size_t(0)
        _check(lib.dzs_checkpoint_bytes(h, ctypes.byref(size)), self.ctx)
        # a physical lightcone sweeps a small box in a few steps, the sweeping one a thin shell per step
        rec_room = n0 if case["physical"] and case["n1d"] <= 128 else n0 // 8
        self.blob = torch.empty(size.value, dtype=torch.uint8, pin_memory=True)
        self.new = torch.empty(size.value + rec_room * dzs.RECORD_DTYPE.itemsize, dtype=torch.uint8, pin_memory=True)
        self.written = ctypes.c_size_t(0)
        _check(lib.dzs_checkpoint(h, self.blob.data_ptr(), size.value, ctypes.byref(self.written)), self.ctx)
        # the program's own arrays, sized for the largest particle count of the run
        real = torch.float64 if self.fp64 else torch.float32
        self.state = {name: torch.zeros(rows * n0, dtype=kind) for name, kind, rows in (
            ("u", torch.int32, 3), ("p", real, 3), ("g", real, 3), ("k", torch.int32, 1), ("id", torch.int32, 1),
            ("fl", torch.uint8, 1))}
        self.records = np.zeros(rec_room, dzs.RECORD_DTYPE)

    def restore(self):
        _check(dzs.load().dzs_restore(self.ctx.h, self.blob.data_ptr(), self.blob.numel()), self.ctx)

    def checkpoint(self):
        _check(dzs.load().dzs_checkpoint(self.ctx.h, self.new.data_ptr(), self.new.numel(),
                                         ctypes.byref(self.written)), self.ctx)
        return self.unpack()

    def unpack(self):
        """the particles and lightcone records of the written checkpoint, in
        the run's own precision: the head, then u, p, g ([3][n] each), k, id,
        fl and the records not yet drained"""
        raw = self.new[:self.written.value]
        head = 16 + ctypes.sizeof(dzs.Params)
        n, _, pending, dropped, _ = (int(v) for v in raw[head:head + 40].numpy().view(np.uint64))
        at, state = head + 40, dict(self.state)
        for name, to in self.state.items():
            size = (3 if name in "upg" else 1) * n * to.element_size()
            if size == to.numel() * to.element_size():  # nothing merged yet: used where it lies
                state[name] = raw[at:at + size].view(to.dtype)
            else:
                to.view(torch.uint8)[:size].copy_(raw[at:at + size])
            at += size
        self.records[:pending] = np.frombuffer(raw.numpy().data, dzs.RECORD_DTYPE, pending, at)
        rec = self.records
        return dict(state, n=n, pending=pending, dropped=dropped, rec_id=rec["id"].view(np.int32),
                    rec_k=rec["k"].view(np.int32), rec_a_cross=rec["a_cross"], rec_x=rec["x"], rec_p=rec["p"])


def _batch_cases(case):
    return [_resume(n1, 2 * n1, case["step"]) for n1 in BATCH_SIZES for _ in range(case["per_size"])]


class _Mocks:
    """Halted mocks on streams of their own, and the batch that steps them."""

    def __init__(self, case, seed):
        self.runs = [_Halted(c, int(seed) * 100 + i) for i, c in enumerate(_batch_cases(case))]
        self.streams = [torch.cuda.Stream() for _ in self.runs]
        for r, s in zip(self.runs, self.streams):
            r.ctx.close()
            r.ctx = dzs.Context(r.ctx.params, stream=s.cuda_stream)
        self.batch = dzs.Batch([r.ctx for r in self.runs])

    def __del__(self):
        if hasattr(self, "batch"):
            self.batch.close()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sort":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed) * 7919 + case["n"])
        u = torch.randint(0, 2 ** 32, (3, case["n"]), generator=gen, device=DEV)
        return dict(kind=kind, u=u.to(torch.int32), perm=torch.empty(case["n"], dtype=torch.int32, device=DEV),
                    keys=torch.empty(case["n"], dtype=torch.int64, device=DEV))
    if kind == "resume":
        return dict(kind=kind, run=_Halted(case, seed))
    if kind == "batch":
        return dict(kind=kind, mocks=_Mocks(case, seed))
    if kind == "alm":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed) * 104729 + case["nside"])
        ctx = dzs.Context(n1d=32, mesh=32, box=64.0)
        ctx.observe(nside=case["nside"], a_lo=0.0, a_hi=2.0)
        ctx.observe_add_records(_sky_records(case, gen))
        return dict(kind=kind, ctx=ctx, lmax=case["lmax"])
    ctx = _context(case["n1d"], case["mesh"], case.get("fp64", False), dzs_on=False)
    _run_state(ctx, case["n1d"], case["step"], False, False, False, seed)
    s = dict(kind=kind, ctx=ctx, case=dict(case))
    if kind == "fof":
        s["halos"] = np.zeros(case["n1d"] ** 3 // case["nmin"], dzs.HALO_DTYPE)  # room for any catalogue
    if kind == "accel":
        s["fp64"] = case["fp64"]
        n = case["n1d"] ** 3
        s["g"] = torch.empty((3, n), dtype=torch.float64, pin_memory=True)
        s["g32"] = torch.empty((3, n), dtype=torch.float32, pin_memory=True)
    return s


def _sky_records(case, gen):
    """lightcone records around the observer of a 64 Mpc/h box: a smooth shell
    with clumps, masses 1 .. 8"""
    n = case["records"]
    d = torch.randn((n, 3), generator=gen, device=DEV, dtype=torch.float64)
    clump = torch.randint(0, n, (n,), generator=gen, device=DEV) % max(1, n // 50)
    near = torch.rand(n, generator=gen, device=DEV) < 0.5
    d = torch.where(near[:, None], d[clump] + 0.05 * d, d)
    d = d / d.square().sum(1, keepdim=True).sqrt()
    r = 10.0 + 20.0 * torch.rand((n, 1), generator=gen, device=DEV, dtype=torch.float64)
    rec = np.zeros(n, dzs.RECORD_DTYPE)
    rec["x"] = (32.0 + r * d).cpu().numpy()
    rec["k"] = (1 + torch.randint(0, 8, (n,), generator=gen, device=DEV)).cpu().numpy()
    rec["id"] = np.arange(n)
    rec["a_cross"] = 0.5
    return rec


def run(state):
    kind = state["kind"]
    if kind == "sort":
        u = state["u"]
        status = dzs.dzs_morton_sort_noalloc(u.data_ptr(), u.shape[1], state["perm"].data_ptr(),
                                             state["keys"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        if status != dzs.DZS_OK:
            raise RuntimeError("dzs_morton_sort_noalloc: status %d" % status)
        return dict(perm=state["perm"], keys=state["keys"])
    if kind == "resume":
        r = state["run"]
        r.restore()
        r.ctx.step(1)
        return r.checkpoint()
    if kind == "batch":
        mocks = state["mocks"]
        for r in mocks.runs:
            r.restore()
        mocks.batch.step(1, slice=1)
        mocks.batch.synchronize()
        out = [r.checkpoint() for r in mocks.runs]
        return dict(u=[o["u"] for o in out], p=[o["p"] for o in out], g=[o["g"] for o in out],
                    k=[o["k"] for o in out], id=[o["id"] for o in out], fl=[o["fl"] for o in out])
    ctx = state["ctx"]
    if kind == "accel":
        _check(dzs.load().dzs_accel(ctx.h, dzs.ACC_ALL, state["g"].data_ptr()), ctx)
        if state["fp64"]:
            return dict(g=state["g"])
        return dict(g=state["g32"].copy_(state["g"]))  # an FP32 context computes FP32 accelerations
    if kind == "pk":
        k, pk, modes = ctx.power_spectrum(state["case"]["nbins"])
        return dict(k=k, pk=pk.astype(np.float32), modes=modes.astype(np.int64))  # FP32 mesh arithmetic
    if kind == "fof":
        h, count = state["halos"], ctypes.c_size_t(0)
        _check(dzs.load().dzs_fof(ctx.h, state["case"]["link"], state["case"]["nmin"], h.ctypes.data, len(h),
                                  ctypes.byref(count), None), ctx)
        return dict(halos=count.value, first=h["first"], count=h["count"], mass=h["mass"].view(np.int64), x=h["x"],
                    rmax2=h["rmax2"].view(np.int64))
    cl, alm = ctx.skymap_alm(state["lmax"])
    return dict(cl=cl, alm=alm)


def work(case):
    kind = case["kind"]
    if kind == "sort":
        return dict(bytes=24.0 * case["n"], flops=0.0)
    if kind == "alm":
        nside, lmax = case["nside"], case["lmax"]
        # ring transforms (one FFT per ring) and the Legendre sums
        rings = 4 * nside - 1
        return dict(bytes=8.0 * 12 * nside ** 2 + 16.0 * (lmax + 1) * (lmax + 2) / 2,
                    flops=rings * (5.0 * 4 * nside * math.log2(4 * nside) + 4.0 * (lmax + 1) * (lmax + 2)))
    if kind == "batch":
        w = [work(c) for c in _batch_cases(case)]
        return dict(bytes=sum(v["bytes"] for v in w), flops=sum(v["flops"] for v in w))
    n, m = case["n1d"] ** 3, case["mesh"] ** 3
    real = 8 if case.get("fp64") else 4
    if kind == "fof":
        return dict(bytes=16.0 * n, flops=27.0 * 8 * n)
    fft = 2.5 * m * math.log2(m)
    if kind == "pk":
        return dict(bytes=12.0 * n, flops=fft + 50.0 * n)
    # particles within r_cut = 5.625 mesh cells of each other at the mean density
    pairs = n * (n / m) * 4.0 / 3.0 * math.pi * (RS_CELLS * RCUT_RS) ** 3
    flops = 45.0 * pairs + 2 * fft + 150.0 * n
    if kind == "accel":
        return dict(bytes=(12.0 + 8 * 3) * n, flops=flops)
    return dict(bytes=2.0 * n * (12 + 6 * real + 9), flops=flops)


# ---------------------------------------------------------------- plain FP64 values


def exact(case, seed):
    kind = case["kind"]
    if kind == "alm":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(int(seed) * 104729 + case["nside"])
        return _exact_alm(case, _sky_records(case, gen))
    if kind == "accel":
        n1 = case["n1d"]
        if n1 > 128 or (n1 == 128 and case["mesh"] == n1):
            return None
        s = _particles(n1, case["step"], False, seed)
        one = torch.ones(n1 ** 3, dtype=torch.int64, device=DEV)
        return dict(g=_forces(n1, case["mesh"], s["u"], one))  # the set is in Morton order already
    if kind == "pk":
        return _exact_pk(case, _particles(case["n1d"], case["step"], False, seed)["u"])
    if kind == "resume":
        n1 = case["n1d"]
        if n1 > 128 or (n1 == 128 and case["mesh"] == n1):
            return None
        return _exact_step(case, seed)
    if kind == "batch":
        out = [_exact_step(c, int(seed) * 100 + i) for i, c in enumerate(_batch_cases(case))]
        return dict(p=[o["p"] for o in out], g=[o["g"] for o in out])
    return None  # the sort and the halo catalogue are decided on integers


def _round_to(x, fp64):
    return x if fp64 else x.to(torch.float32).to(torch.float64)


def _exact_step(case, seed):
    """momenta and accelerations after one step, arithmetic in FP64; inputs as
    the run holds them (rounded to its precision)"""
    n1, fp64 = case["n1d"], case["fp64"]
    box = BOX_PER_N1D * n1
    s = _particles(n1, case["step"], case["physical"], seed)
    tab = s["tab"]
    u, ident = s["u"], s["id"]
    k = torch.ones_like(ident)
    p, g = _round_to(s["p"], fp64), _round_to(s["g"], fp64)
    crossed = s["fl"].to(torch.bool)
    if case["dzs"]:  # the merge that brought the run here; g stays with the surviving id
        amin2 = float(g[:, ~crossed].square().sum(0).min()) if bool((~crossed).any()) else math.inf
        u, p, k, ident, crossed, _ = _merge(case, u, p, k, ident, crossed, tab["rlat0"], amin2)
        of = torch.empty(n1 ** 3, dtype=torch.int64, device=DEV)
        of[s["id"]] = torch.arange(n1 ** 3, device=DEV)
        g = _round_to(s["g"], fp64)[:, of[ident]]
        p = _round_to(p, fp64)
    kick1 = tab["kick1"] if fp64 else float(np.float32(tab["kick1"]))
    p = _round_to(p + g * kick1, fp64)
    before = u
    u = torch.remainder(u + torch.round(p * (tab["drift"] * (TWO32 / box))).to(torch.int64), 2 ** 32)
    now = ~_dist_far(before, tab["rlat0"]) & _dist_far(u, tab["rlat1"])
    crossed = crossed | now
    amin2 = float(g[:, ~crossed].square().sum(0).min()) if bool((~crossed).any()) else math.inf
    order = torch.argsort(_morton(u), stable=True)
    u, p, k, ident, crossed = u[:, order], p[:, order], k[order], ident[order], crossed[order]
    if case["dzs"]:
        u, p, k, ident, crossed, _ = _merge(case, u, p, k, ident, crossed, tab["rlat1"], amin2)
        p = _round_to(p, fp64)
    g = _forces(n1, case["mesh"], u, k)
    p = p + g * tab["kick2"]
    return dict(p=_filled(p, n1), g=_filled(g, n1))


def _filled(v, n1):
    """[3][n] as the head of an array for n1^3 particles"""
    out = torch.zeros(3 * n1 ** 3, dtype=torch.float64, device=DEV)
    out[:v.numel()] = v.reshape(-1)
    return out


def _merge(case, u, p, k, ident, crossed, rlat, amin2):
    """DZS merge of a Morton-ordered set (Eq. 3, geometric or dynamical rule)"""
    n1 = case["n1d"]
    box = BOX_PER_N1D * n1
    jmin = 1
    while (1 << jmin) * (1 << (case["merge_level"] - 1)) < n1:
        jmin += 1
    n = u.shape[1]
    key = _morton(u)
    blat = int(math.floor(BUFFER_CELLS * TWO32 / case["mesh"]))
    head = torch.arange(n, device=DEV)  # first member of the particle's merged cell
    done = torch.zeros(n, dtype=torch.bool, device=DEV)
    gm0 = 1.5 * OMEGA_M * box ** 3 / (4.0 * math.pi * n1 ** 3)
    rhs = ALPHA_DYN * math.sqrt(amin2)
    for j in range(jmin, 22):
        cell = key >> (3 * (21 - j))
        _, inv, cnt = torch.unique_consecutive(cell, return_inverse=True, return_counts=True)
        if int(cnt.max()) < 2:
            break
        first = torch.cumsum(cnt, 0) - cnt
        mass = torch.zeros_like(cnt).index_add_(0, inv, k)
        d2 = torch.zeros(cnt.shape[0], dtype=torch.float64, device=DEV)
        for ax in range(3):
            sm = torch.zeros_like(cnt).index_add_(0, inv, k * u[ax])
            d2 += (((2 * sm + mass) // (2 * mass)) - 2 ** 31).to(torch.float64).square()
        if case["dynamical"]:
            dist = (torch.sqrt(d2) - float(rlat + blat)) * (box / TWO32)
            lhs = gm0 * mass.to(torch.float64) * (box * 2.0 ** -j) ** 2 / dist ** 4
            good = (dist > 0) & (lhs < rhs)
        else:
            lt = math.ceil(2.0 ** (32 - j) / THETA_DZS)
            good = d2 > (float(rlat + blat + lt) ** 2 if lt < 2 ** 32 else math.inf)
        take = (good & (cnt >= 2))[inv] & ~done
        head = torch.where(take, first[inv], head)
        done |= take
    heads, inv = torch.unique(head, return_inverse=True)
    m = heads.shape[0]
    mass = torch.zeros(m, dtype=torch.int64, device=DEV).index_add_(0, inv, k)
    merged = torch.zeros(m, dtype=torch.bool, device=DEV)
    merged[inv[done]] = True
    u2, p2 = u[:, heads].clone(), p[:, heads].clone()
    for ax in range(3):
        sm = torch.zeros(m, dtype=torch.int64, device=DEV).index_add_(0, inv, k * u[ax])
        sp = torch.zeros(m, dtype=torch.float64, device=DEV).index_add_(0, inv, k.to(torch.float64) * p[ax])
        u2[ax] = torch.where(merged, (2 * sm + mass) // (2 * mass), u2[ax])
        p2[ax] = torch.where(merged, sp / mass.to(torch.float64), p2[ax])
    ident2 = torch.full((m,), 2 ** 62, dtype=torch.int64, device=DEV).scatter_reduce_(0, inv, ident, "amin")
    return u2, p2, mass, ident2, crossed[heads] | merged, merged


def _forces(n1, mesh, u, k):
    return _pm(n1, mesh, u, k) + _tree(n1, mesh, u, k)


def _cic(mesh, u):
    """base cell and fraction per axis"""
    t = u * mesh
    return t >> 32, (t & 0xFFFFFFFF).to(torch.float64) / TWO32


def _delta(n1, mesh, u, k):
    c, f = _cic(mesh, u)
    rho = torch.zeros(mesh ** 3, dtype=torch.float64, device=DEV)
    for o in range(8):
        cell, w = torch.zeros_like(c[0]), k.to(torch.float64)
        for ax in range(3):
            bit = (o >> (2 - ax)) & 1
            cell = cell * mesh + (c[ax] + bit) % mesh
            w = w * (f[ax] if bit else 1.0 - f[ax])
        rho.index_add_(0, cell, w)
    return (rho * (mesh ** 3 / n1 ** 3) - 1.0).reshape(mesh, mesh, mesh)


def _axes(mesh, box):
    """wave numbers and CIC windows per axis"""
    m = torch.fft.fftfreq(mesh, 1.0 / mesh, device=DEV, dtype=torch.float64)
    half = torch.arange(mesh // 2 + 1, device=DEV, dtype=torch.float64)
    kf = 2.0 * math.pi / box
    return [(v * kf, torch.sinc(v / mesh) ** 2) for v in (m, m, half)]


def _pm(n1, mesh, u, k):
    box = BOX_PER_N1D * n1
    (kx, wx), (ky, wy), (kz, wz) = _axes(mesh, box)
    d = torch.fft.rfftn(_delta(n1, mesh, u, k))
    k2 = kx[:, None, None] ** 2 + ky[None, :, None] ** 2 + kz[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    win = wx[:, None, None] * wy[None, :, None] * wz[None, None, :]
    d *= -1.5 * OMEGA_M * torch.exp(-k2 * (RS_CELLS * box / mesh) ** 2) / (k2 * win ** 2)
    d[0, 0, 0] = 0.0
    phi = torch.fft.irfftn(d, s=(mesh, mesh, mesh))
    c, f = _cic(mesh, u)
    out = []
    for ax in range(3):
        gm = 8.0 * (torch.roll(phi, -1, ax) - torch.roll(phi, 1, ax)) - (torch.roll(phi, -2, ax)
                                                                        - torch.roll(phi, 2, ax))
        gm = (gm / (-12.0 * box / mesh)).reshape(-1)
        acc = torch.zeros(u.shape[1], dtype=torch.float64, device=DEV)
        for o in range(8):
            cell, w = torch.zeros_like(c[0]), torch.ones_like(f[0])
            for b in range(3):
                bit = (o >> (2 - b)) & 1
                cell = cell * mesh + (c[b] + bit) % mesh
                w = w * (f[b] if bit else 1.0 - f[b])
            acc += w * gm[cell]
        out.append(acc)
    return torch.stack(out)


def _build_tree(u, k):
    """oct-tree of a Morton-ordered set, depth by depth: node arrays and groups"""
    n = u.shape[1]
    key = _morton(u)
    names = ("level", "start", "count", "parent", "mass", "kmax", "cx", "cy", "cz", "mx", "my", "mz")
    nodes = {v: [] for v in names}
    internal, groups = [], []
    base = 0
    owner = torch.zeros(n, dtype=torch.int64, device=DEV)  # parent node of each particle, -1: below a leaf
    big = torch.tensor([True], device=DEV)                 # parents holding more than GROUP
    for j in range(22):
        live = torch.nonzero(owner >= 0).reshape(-1)
        if live.numel() == 0:
            break
        cell = key[live] >> (3 * (21 - j))
        _, inv, cnt = torch.unique_consecutive(cell, return_inverse=True, return_counts=True)
        start = live[torch.cumsum(cnt, 0) - cnt]
        mass = torch.zeros_like(cnt).index_add_(0, inv, k[live])
        nodes["level"].append(torch.full_like(cnt, j))
        nodes["start"].append(start)
        nodes["count"].append(cnt)
        parent = owner[start] if j else torch.full_like(cnt, -1)
        nodes["parent"].append(parent)
        nodes["mass"].append(mass)
        nodes["kmax"].append(torch.zeros_like(cnt).scatter_reduce_(0, inv, k[live], "amax"))
        half = 1 << (31 - j)
        for ax, cn, mn in ((0, "cx", "mx"), (1, "cy", "my"), (2, "cz", "mz")):
            sm = torch.zeros_like(cnt).index_add_(0, inv, k[live] * u[ax, live])
            nodes[mn].append((2 * sm + mass) // (2 * mass))
            nodes[cn].append((u[ax, start] // (2 * half)) * (2 * half) + half)
        inner = (cnt > LEAF) & (j < 21)
        internal.append(inner)
        parent_big = big[parent] if j else torch.ones_like(inner)
        groups.append(base + torch.nonzero(parent_big & ((cnt <= GROUP) | ~inner)).reshape(-1))
        big = torch.cat([big, cnt > GROUP]) if j else cnt > GROUP
        owner = torch.full_like(owner, -1)
        owner[live] = torch.where(inner[inv], base + inv, -1)
        base += cnt.shape[0]
    t = {v: torch.cat(nodes[v]) for v in names}
    t["inner"] = torch.cat(internal)
    t["nchild"] = torch.zeros_like(t["count"]).index_add_(0, t["parent"][1:], torch.ones_like(t["parent"][1:]))
    first = torch.full_like(t["count"], base)
    t["child"] = first.scatter_reduce_(0, t["parent"][1:], torch.arange(1, base, device=DEV), "amin")
    return t, torch.cat(groups)


def _expand(start, count):
    """(owner, member) of every item of the runs [start, start + count)"""
    owner = torch.repeat_interleave(torch.arange(count.shape[0], device=DEV), count)
    member = torch.arange(owner.shape[0], device=DEV) - (torch.cumsum(count, 0) - count)[owner] + start[owner]
    return owner, member


def _tree(n1, mesh, u, k):
    """short-range force of the group walk: skip, open (l >= theta d), accept"""
    box = BOX_PER_N1D * n1
    rs = RS_CELLS * box / mesh
    rcut2 = (RCUT_RS * rs / box * TWO32) ** 2
    scale = box / TWO32
    gm0 = 1.5 * OMEGA_M * box ** 3 / (4.0 * math.pi * n1 ** 3) / scale ** 2
    h0 = 2.8 * SOFT * box / n1 / scale
    t, groups = _build_tree(u, k)
    acc = torch.zeros((3, u.shape[1]), dtype=torch.float64, device=DEV)
    com, cen = (t["mx"], t["my"], t["mz"]), (t["cx"], t["cy"], t["cz"])
    kf, kmax = k.to(torch.float64), t["kmax"].to(torch.float64)

    def gap2(pos, half, grp):
        """squared distance of points (or cubes of half side `half`) from the groups' cubes"""
        hg = (2.0 ** 31) * torch.pow(2.0, -t["level"][grp].to(torch.float64)) + half
        s = torch.zeros(grp.shape[0], dtype=torch.float64, device=DEV)
        for ax in range(3):
            s += (_wrap(pos[ax] - cen[ax][grp]).abs().to(torch.float64) - hg).clamp(min=0.0).square()
        return s

    def evaluate(grp, pos, mass, big):
        """add the forces of entries (group, position, multiplicity, softening multiplicity)"""
        step = 1 << 17
        for e0 in range(0, grp.shape[0], step):
            ge = grp[e0:e0 + step]
            ent, i = _expand(t["start"][ge], t["count"][ge])
            ent = ent + e0
            d = [_wrap(pos[ax][ent] - u[ax][i]).to(torch.float64) for ax in range(3)]
            r2 = d[0].square() + d[1].square() + d[2].square()
            near = torch.nonzero((r2 > 0.0) & (r2 < rcut2)).reshape(-1)
            ent, i, r2 = ent[near], i[near], r2[near]
            r = torch.sqrt(r2)
            h = h0 * torch.pow(torch.maximum(big[ent], kf[i]), 1.0 / 3.0)
            q = (r / h).clamp(min=1e-300)
            inner = 32.0 / 3.0 - 38.4 * q.square() + 32.0 * q ** 3
            outer = 64.0 / 3.0 - 48.0 * q + 38.4 * q.square() - 32.0 / 3.0 * q ** 3 - 1.0 / 15.0 / q ** 3
            fac = torch.where(q >= 1.0, 1.0 / (r2 * r), torch.where(q < 0.5, inner, outer) / h ** 3)
            x = r * (scale / (2.0 * rs))
            f = gm0 * mass[ent] * fac * (torch.special.erfc(x) + 2.0 / math.sqrt(math.pi) * x * torch.exp(-x * x))
            for ax in range(3):
                acc[ax].index_add_(0, i, f * d[ax][near])

    for g0 in range(0, groups.shape[0], 8192):
        grp = groups[g0:g0 + 8192]
        node = torch.zeros_like(grp)
        while grp.numel():
            root = t["level"][node] == 0
            hn = (2.0 ** 31) * torch.pow(2.0, -t["level"][node].to(torch.float64))
            near = gap2([c[node] for c in cen], hn, grp)
            touch = root | (near == 0.0)
            keep = touch | (near <= rcut2)
            grp, node, touch, hn = grp[keep], node[keep], touch[keep], hn[keep]
            dist2 = gap2([c[node] for c in com], 0.0, grp)
            opened = touch | (2.0 * hn >= THETA * torch.sqrt(dist2))
            mono = ~opened & (dist2 <= rcut2)
            evaluate(grp[mono], [c[node[mono]] for c in com], t["mass"][node[mono]].to(torch.float64),
                     kmax[node[mono]])
            leaf = opened & ~t["inner"][node]
            own, part = _expand(t["start"][node[leaf]], t["count"][node[leaf]])
            lg = grp[leaf][own]
            close = gap2([u[ax][part] for ax in range(3)], 0.0, lg) <= rcut2
            lg, part = lg[close], part[close]
            evaluate(lg, [u[ax][part] for ax in range(3)], kf[part], kf[part])
            inner = opened & t["inner"][node]
            own, child = _expand(t["child"][node[inner]], t["nchild"][node[inner]])
            grp, node = grp[inner][own], child
    return acc


def _exact_pk(case, u):
    n1, mesh, nbins = case["n1d"], case["mesh"], case["nbins"]
    box = BOX_PER_N1D * n1
    d = torch.fft.rfftn(_delta(n1, mesh, u, torch.ones_like(u[0])))
    n = [torch.fft.fftfreq(mesh, 1.0 / mesh, device=DEV, dtype=torch.float64)] * 2
    n.append(torch.arange(mesh // 2 + 1, device=DEV, dtype=torch.float64))
    mag = torch.sqrt(n[0][:, None, None] ** 2 + n[1][None, :, None] ** 2 + n[2][None, None, :] ** 2)
    win = (torch.sinc(n[0] / mesh) ** 2)[:, None, None] * (torch.sinc(n[1] / mesh) ** 2)[None, :, None]
    win = win * (torch.sinc(n[2] / mesh) ** 2)[None, None, :]
    power = (d.real.square() + d.imag.square()) * (box ** 3 / float(mesh) ** 6) / win.square() - box ** 3 / n1 ** 3
    weight = torch.full((mesh // 2 + 1,), 2.0, dtype=torch.float64, device=DEV)
    weight[0] = weight[mesh // 2] = 1.0
    weight = weight.expand(mesh, mesh, -1).reshape(-1)
    b = torch.floor(mag + 0.5).to(torch.int64).reshape(-1)
    use = (b >= 1) & (b <= nbins)
    b, weight = b[use] - 1, weight[use]
    cnt, ks, ps = (torch.zeros(nbins, dtype=torch.float64, device=DEV).index_add_(0, b, v) for v in (
        weight, weight * mag.reshape(-1)[use] * (2.0 * math.pi / box), weight * power.reshape(-1)[use]))
    return dict(k=(ks / cnt).cpu(), pk=(ps / cnt).to(torch.float64).cpu(), modes=None)


def _exact_alm(case, rec):
    """a_lm of the RING map of the records, by direct sums over pixels and rings"""
    nside, lmax = case["nside"], case["lmax"]
    npix = 12 * nside * nside
    x = rec["x"] - 32.0
    sky = torch.zeros(npix, dtype=torch.float64, device=DEV)
    pix = torch.from_numpy(_ring_pixels(nside, x)).to(DEV)
    sky.index_add_(0, pix, torch.from_numpy(rec["k"].astype(np.float64)).to(DEV))
    m = torch.arange(lmax + 1, device=DEV, dtype=torch.float64)
    rings = 4 * nside - 1
    z = torch.empty(rings, dtype=torch.float64, device=DEV)
    f = torch.empty((rings, lmax + 1), dtype=torch.complex128, device=DEV)
    at = 0
    for r in range(1, rings + 1):
        cap = min(r, 4 * nside - r)
        if cap < nside:
            nphi, shift = 4 * cap, 0.5
            zr = 1.0 - cap * cap / (3.0 * nside * nside)
            zr = zr if r < nside else -zr
        else:
            nphi, shift = 4 * nside, 0.5 if (r + nside) % 2 == 0 else 0.0
            zr = (2 * nside - r) * 2.0 / (3.0 * nside)
        z[r - 1] = zr
        phase = (torch.arange(nphi, device=DEV, dtype=torch.float64) + shift) / nphi
        ang = -2.0 * math.pi * torch.remainder(m[:, None] * phase[None, :], 1.0)
        v = sky[at:at + nphi]
        f[r - 1] = torch.complex(torch.cos(ang) @ v, torch.sin(ang) @ v)
        at += nphi
    sin = torch.sqrt((1.0 - z) * (1.0 + z))[:, None]
    # lambda_mm, then the three-term recursion in l for all m at once
    lead = torch.cumprod(torch.cat([torch.tensor([0.28209479177387814], device=DEV, dtype=torch.float64),
                                    -torch.sqrt((2.0 * m[1:] + 1.0) / (2.0 * m[1:]))]), 0)
    mm = lead[None, :] * sin ** m[None, :]
    alm = torch.zeros((lmax + 1, lmax + 1), dtype=torch.complex128, device=DEV)
    prev2, prev = torch.zeros_like(mm), torch.zeros_like(mm)
    for el in range(lmax + 1):
        d = (el * el - m * m).clamp(min=1.0)
        a = torch.sqrt((4.0 * el * el - 1.0) / d) if el else torch.zeros_like(m)
        b = torch.sqrt(((2.0 * el + 1.0) * ((el - 1.0) ** 2 - m * m).clamp(min=0.0))
                       / (max(1.0, 2.0 * el - 3.0) * d))
        lam = a * z[:, None] * prev - b * prev2
        lam = torch.where(m[None, :] < el, lam, torch.zeros_like(lam))
        lam[:, el] = mm[:, el]
        alm[el] = (lam.to(torch.complex128) * f).sum(0)
        prev2, prev = prev, lam
    alm *= 4.0 * math.pi / npix
    p = alm.real.square() + alm.imag.square()
    el = torch.arange(lmax + 1, device=DEV, dtype=torch.float64)
    return dict(cl=((2.0 * p.sum(1) - p[:, 0]) / (2.0 * el + 1.0)).cpu(), alm=alm.cpu())


def _ring_pixels(nside, x):
    """RING pixels (Gorski et al. 2005) of directions x [n][3]"""
    r = np.sqrt((x ** 2).sum(1))
    z = x[:, 2] / r
    t = np.arctan2(x[:, 1], x[:, 0])
    t = np.where(t < 0, t + 2 * np.pi, t) / (0.5 * np.pi)
    t = np.where(t >= 4.0, t - 4.0, t)
    npix = 12 * nside * nside
    jp = np.floor(nside * (0.5 + t) - nside * 0.75 * z).astype(np.int64)
    jm = np.floor(nside * (0.5 + t) + nside * 0.75 * z).astype(np.int64)
    ir = nside + 1 + jp - jm
    shift = 1 - (ir & 1)
    ip = np.floor_divide(jp + jm - nside + shift, 2) % (4 * nside)
    belt = 2 * nside * (nside - 1) + (ir - 1) * 4 * nside + ip
    tp = t - np.floor(t)
    w = nside * np.sqrt(3.0 * (1.0 - np.abs(z)))
    ring = np.floor(tp * w).astype(np.int64) + np.floor((1.0 - tp) * w).astype(np.int64) + 1
    pos = np.floor(t * ring).astype(np.int64) % (4 * ring)
    polar = np.where(z > 0, 2 * ring * (ring - 1) + pos, npix - 2 * ring * (ring + 1) + pos)
    return np.where(np.abs(z) <= 2.0 / 3.0, belt, polar)
