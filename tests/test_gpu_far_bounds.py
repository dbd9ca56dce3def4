"""Where the far and split forms end (csrc/pc_far_f32.cuh): separations of a dipole's charges of more than one
sample c dt, planes whose tiles are wide against the distance of their sources, moments that grow during a run,
and devices without the memory for the forms' tables.  References: binary128 and the FP64 oracle."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2107_12437_gb300 as pc
import workloads as W
from test_gpu_far import OMEGA0, _cloud, _ed_binary128

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = pc.Context(0)
    yield c
    c.close()


def _norm(v):
    return np.abs(v) if v.ndim == 2 else np.linalg.norm(v, axis=-1)


# ------------------------------------------------------------------------------------------------
# separations of more than one sample: the float64 field sum
# ------------------------------------------------------------------------------------------------
# dt, separation of the charges, distance, extent of the sources, histories' end, frames: the separations are
# 0.33, 0.95, 1.05, 2, 6.7 and 3.3 samples; the last one's charges are slow enough only near their turning
# points, at which the frames look (sources within 20 nm, retarded by 17.5 um, and the quarter period)
_SPREAD = {
    "10 pm": (1e-19, 1e-11, 1.2e-6, 2e-7, 8e-15, (6.6e-15, 7.3e-15)),
    "28.4 pm": (1e-19, 2.84e-11, 1.2e-6, 2e-7, 8e-15, (6.6e-15, 7.3e-15)),
    "31.6 pm": (1e-19, 3.16e-11, 1.2e-6, 2e-7, 8e-15, (6.6e-15, 7.3e-15)),
    "60 pm": (1e-19, 6e-11, 1.2e-6, 2e-7, 8e-15, (6.6e-15, 7.3e-15)),
    "200 pm": (1e-19, 2e-10, 4.1e-6, 2e-8, 20e-15, tuple(4.09e-6 / W.C + (k + 0.5) * 2.5e-15 for k in (0, 1))),
    "1 nm": (1e-18, 1e-9, 17.5e-6, 2e-8, 80e-15, tuple(17.49e-6 / W.C + (k + 0.5) * 2.5e-15 for k in (2, 5))),
}


@pytest.mark.parametrize("kind", [pc.PC_TOTAL, pc.PC_COULOMB, pc.PC_RADIATION])
@pytest.mark.parametrize("case", sorted(_SPREAD))
def test_float64_fields_of_wide_dipoles(ctx, case, kind):
    # the bound of tests/test_gpu_far.py::test_split_fields_against_binary128, five sources at random places
    dt, amp, z, ext, t_end, times = _SPREAD[case]
    rng = np.random.default_rng(31)
    dp = W.sinusoidal_dipoles(rng.uniform(0.0, ext, (5, 3)), W.unit_vectors(rng, 5), OMEGA0, amp, dt, t_end)
    P = 11003
    pts = np.concatenate([rng.uniform(0.0, ext, (P, 2)), np.full((P, 1), z)], axis=1)
    out = pc.pc_fields(ctx, dipoles=pc.dipoles_to_device(dp), points=torch.as_tensor(pts, device="cuda"),
                       times=list(times), kind=kind)
    p = np.r_[0, P - 1, rng.integers(0, P, 60)]
    ref = oracle.fields_x(pts[p], times, dipoles=dp, kind=kind)
    scale = oracle.fields(pts[p], times, dipoles=dp, kind=kind)["scale_source"]
    assert ref["status"] == oracle.OK and not out["mask"].any()
    worst = {}
    for k in ("E", "B", "phi", "A"):
        g = out[k][:, torch.as_tensor(p, device="cuda")].cpu().numpy()
        sc = scale["E"] / W.C if k == "B" else scale[k]
        worst[k] = float(np.max(_norm(g - ref[k]) / np.maximum(_norm(ref[k]), 1e-3 * sc)))
    assert max(worst.values()) <= 1e-10, worst


# 600 pm at 0.1 as: 20 samples, so that a charge lies up to 10 from its centre; 12 um away, where every form's
# condition on separation over distance holds.  The moment rests, and all points are the same one.
_WIDE = dict(dt=1e-19, amp=6e-10, S=3001, R=12e-6)


def _resting(N):
    d = W.E_CHARGE * _WIDE["amp"] * np.ones((N, _WIDE["S"]))
    z = np.zeros((N, _WIDE["S"]))
    one = np.ones(N)
    axis = np.tile([0.0, 0.0, 1.0], (N, 1))
    return W.Dipoles(origin=np.zeros((N, 3)), axis=axis, q=W.E_CHARGE * one, m1=W.M_E * one, m2=W.M_E * one, d=d, d_dot=z,
                     d_ddot=z.copy(), t0=0.0, dt=_WIDE["dt"])


def _wide_call(ctx, form, time, r_excl=0.0):
    # enough (point, dipole) pairs for the form to be taken: 1e5, 2e6 and 1e8
    N, nu, nv = {"float64": (4, 160, 160), "list": (4, 710, 710), "plane": (64, 1300, 1300)}[form]
    dp = pc.dipoles_to_device(_resting(N))
    kw = dict(dipoles=dp, times=[time], r_excl=r_excl, precision=pc.PC_F64 if form == "float64" else pc.PC_MIXED)
    if form == "plane":
        return pc.pc_fields_plane(ctx, origin=(0.0, 0.0, _WIDE["R"]), eu=(1e-18, 0, 0), ev=(0, 1e-18, 0), nu=nu, nv=nv, **kw)
    pts = torch.zeros((nu * nv, 3), dtype=torch.float64, device="cuda")
    pts[:, 2] = _WIDE["R"]
    return pc.pc_fields(ctx, points=pts, **kw)


@pytest.mark.parametrize("form", ["float64", "list", "plane"])
def test_charge_beyond_the_end_of_its_history(ctx, form):
    # the centre's retarded time 9.5 samples inside the history, the nearer charge's half a sample past it
    pt = np.array([[0.0, 0.0, _WIDE["R"]]])
    for inside, status in ((9.5, oracle.ERR_HISTORY), (10.5, oracle.OK)):
        time = _WIDE["R"] / W.C + (_WIDE["S"] - 1 - inside) * _WIDE["dt"]
        assert oracle.fields(pt, [time], dipoles=_resting(1))["status"] == status
        if status == oracle.OK:
            assert not _wide_call(ctx, form, time)["mask"].any()
        else:
            with pytest.raises(pc.PcError, match="PC_ERR_HISTORY"):
                _wide_call(ctx, form, time)


@pytest.mark.parametrize("form", ["float64", "list", "plane"])
def test_charge_within_the_exclusion_radius(ctx, form):
    # the centre 9.5 samples outside r_excl, the nearer charge half a sample inside
    pt = np.array([[0.0, 0.0, _WIDE["R"]]])
    time = _WIDE["R"] / W.C + 1000 * _WIDE["dt"]
    for outside, masked in ((9.5, True), (10.5, False)):
        r_excl = _WIDE["R"] - outside * _WIDE["dt"] * W.C
        assert bool(oracle.fields(pt, [time], dipoles=_resting(1), r_excl=r_excl)["mask"].all()) == masked
        m = _wide_call(ctx, form, time, r_excl)["mask"]
        assert bool(m.all()) == masked and bool(m.any()) == masked


# ------------------------------------------------------------------------------------------------
# histories that are not smooth: the float64 field sum
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("kind", [pc.PC_TOTAL, pc.PC_COULOMB, pc.PC_RADIATION])
@pytest.mark.parametrize("case", ["d", "d_ddot", "all", "step", "mixture"])
def test_float64_fields_of_rough_histories(ctx, case, kind):
    # the fields are those of the piecewise linear samples, whatever these are: noise of a tenth of the moment
    # from sample to sample, one step of it, or noise in one dipole of five; bound as above
    rng = np.random.default_rng(17)
    dp = W.sinusoidal_dipoles(rng.uniform(0.0, 2e-7, (5, 3)), W.unit_vectors(rng, 5), OMEGA0, 1e-11, 1e-18, 9e-15)
    noise = rng.uniform(-0.1, 0.1, (3,) + dp.d.shape)
    if case == "mixture":
        noise[:, 1:] = 0.0
    if case in ("d", "all", "mixture"):
        dp.d += W.E_CHARGE * 1e-11 * noise[0]
    if case in ("all", "mixture"):
        dp.d_dot += W.E_CHARGE * 1e-11 * OMEGA0 * noise[1]
    if case in ("d_ddot", "all", "mixture"):
        dp.d_ddot += W.E_CHARGE * 1e-11 * OMEGA0 ** 2 * noise[2]
    if case == "step":
        dp.d[:, 6000:] += W.E_CHARGE * 1e-12
    times = [7.1e-15, 8.9e-15]
    P = 11003
    pts = np.concatenate([rng.uniform(0.0, 2e-7, (P, 2)), np.full((P, 1), 4.5e-7)], axis=1)
    out = pc.pc_fields(ctx, dipoles=pc.dipoles_to_device(dp), points=torch.as_tensor(pts, device="cuda"),
                       times=times, kind=kind)
    # points whose retarded samples of the first source lie around the step, and others
    late = np.linalg.norm(pts - dp.origin[0], axis=1) / (W.C * 1e-18)
    p = np.r_[np.argsort(np.abs(late - 1100.0))[:40], rng.integers(0, P, 160)]
    ref = oracle.fields_x(pts[p], times, dipoles=dp, kind=kind)
    scale = oracle.fields(pts[p], times, dipoles=dp, kind=kind)["scale_source"]
    assert ref["status"] == oracle.OK and not out["mask"].any()
    worst = {}
    for k in ("E", "B", "phi", "A"):
        g = out[k][:, torch.as_tensor(p, device="cuda")].cpu().numpy()
        sc = scale["E"] / W.C if k == "B" else scale[k]
        worst[k] = float(np.max(_norm(g - ref[k]) / np.maximum(_norm(ref[k]), 1e-3 * sc)))
    assert max(worst.values()) <= 1e-10, worst


@pytest.mark.parametrize("which", ["d", "d_dot", "d_ddot"])
@pytest.mark.parametrize("side", [0, 1])
def test_float64_fields_of_a_sample_that_is_no_number(ctx, which, side):
    # one NaN among the samples, at either end of a point's retarded segment: a call large enough for the split
    # form does what a small one does, which refuses the retarded times that do not converge
    rng = np.random.default_rng(23)
    dp = W.sinusoidal_dipoles(rng.uniform(0.0, 2e-7, (5, 3)), W.unit_vectors(rng, 5), OMEGA0, 1e-11, 1e-18, 9e-15)
    getattr(dp, which)[2, 6000 + side] = np.nan
    dev = pc.dipoles_to_device(dp)
    # the centre's retarded sample of source 2 at 7.1 fs is 6000.5, far from both knots
    direction = np.array([0.36, 0.48, 0.8])
    pt = dp.origin[2] + (7100 - 6000.5) * 1e-18 * W.C * direction

    def call(P):
        pts = torch.as_tensor(np.tile(pt, (P, 1)), device="cuda")
        try:
            out = pc.pc_fields(ctx, dipoles=dev, points=pts, times=[7.1e-15])
            return {k: bool(torch.isnan(out[k]).any()) for k in ("E", "B", "phi", "A")}
        except pc.PcError as e:
            return e.status

    small = call(500)
    assert small == call(40001)
    assert small == pc.capi.PC_ERR_NOCONV if which == "d" else True in small.values()


# ------------------------------------------------------------------------------------------------
# separations of more than one sample: the float64 run and its gradients
# ------------------------------------------------------------------------------------------------
def _wide_cloud(amp, dt, N=70, cell=1.6e-7, steps=9000):
    """_cloud() with steps of dt and charges amp apart; pairs from 1.1e-7 m on, most of them past one light
    crossing within the steps."""
    cfg = _cloud(N, cell=cell, seed=41)
    cfg.dt = dt
    cfg.d0[:] = W.E_CHARGE * amp
    cfg.n_steps = steps
    return cfg


@pytest.mark.parametrize("amp,dt,steps", [(1.8e-11, 1e-19, 9000), (4.5e-11, 1e-19, 9000), (4.5e-11, 2e-20, 45000)])
def test_float64_drive_of_wide_dipoles(ctx, amp, dt, steps):
    # 0.6, 1.5 and 7.5 samples: E_d on the run's own history within the float64 path's 1e-10 of its largest value
    cfg = _wide_cloud(amp, dt)
    f = pc.pc_dipoles_run(ctx, pc.lo_config_to_device(cfg), dt, steps, precision=pc.PC_F64, want_Ed=True)
    at = np.linspace(steps // 2, steps, 29).astype(int) - np.arange(29) % 7
    recv = [0, 33, 69]
    h = [f[k][0].cpu().numpy() for k in ("d", "d_dot", "d_ddot")]
    ref = _ed_binary128(cfg, h, 0.0, at * dt, recv)
    err = [float(np.max(np.abs(f["Ed"][0, i].cpu().numpy()[at] - e)) / np.max(np.abs(e))) for e, i in zip(ref, recv)]
    assert max(err) < 1e-10, err


@pytest.mark.parametrize("amp,dt,steps", [(1.8e-11, 1e-19, 9000), (4.5e-11, 1e-19, 9000)])
def test_float64_gradients_of_wide_dipoles(ctx, amp, dt, steps):
    # as tests/test_gpu_far.py::test_split_reverse_against_the_two_charge_form: masses one rounding apart keep
    # every pair in the two-charge form (a cloud of 0.15 um: its delays have to lie within some 9000 samples)
    cfg = _wide_cloud(amp, dt, cell=3e-8)
    w = torch.linspace(0.5, 1.5, cfg.N, dtype=torch.float64, device="cuda").view(1, cfg.N)
    got = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), dt, steps, w)
    cfg.m1 = np.nextafter(cfg.m1, np.inf)
    ref = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), dt, steps, w)
    err = [float((g - r).abs().max() / r.abs().max()) for g, r in zip(got, ref)]
    assert max(err) < 1e-10, err


@pytest.mark.parametrize("amp,dt,steps,cell", [(1.8e-11, 1e-19, 9000, 1.6e-7), (2.8e-11, 3e-20, 20000, 4e-8),
                                               (2e-11, 1e-20, 60000, 1e-7)])
def test_mixed_drive_of_wide_dipoles(ctx, amp, dt, steps, cell):
    # 0.6, 3.1 and 6.7 samples: E_d within 1e-5 of its largest value, the bound of
    # tests/test_gpu_far.py::test_far_drive_against_oracle, also in the steps in which the field of a source sets
    # in, its two charges' one after the other
    cfg = _wide_cloud(amp, dt, cell=cell)
    lod = pc.lo_config_to_device(cfg)
    f = pc.pc_dipoles_run(ctx, lod, dt, steps, precision=pc.PC_F64, want_Ed=True)
    m = pc.pc_dipoles_run(ctx, lod, dt, steps, precision=pc.PC_MIXED, want_Ed=True)
    e = float(((m["Ed"] - f["Ed"]).abs().amax(-1) / f["Ed"].abs().amax(-1)).max())
    assert e < 1e-5, e


# ------------------------------------------------------------------------------------------------
# planes whose tiles are wide against the distance of their sources
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("kind", [pc.PC_TOTAL, pc.PC_COULOMB, pc.PC_RADIATION])
@pytest.mark.parametrize("step", [1.6e-9, 1.9e-9, 1e-8, 2e-8, 2.2e-8, 4e-8, 1e-7, 3e-7, 1e-6])
def test_points_much_nearer_than_the_anchor_of_their_tile(ctx, step, kind):
    # sources straight beyond a corner of a tile (32 x 16 points), as near to it as the far form allows (400 c dt
    # and the tile's radius from the anchor); steps on both sides of far_fine's (5.8 c dt) and of kFarTile's (70).
    # The same frames in a call too small for the far kernel are fields_mixed_kernel's: the fields at those corners
    # are no further from the oracle than twice its (its tiles of 16 x 16 are 1.6 times smaller) and a few
    # float32 roundings of the source scale.
    dt, nu, nv, N = 1e-18, 160, 144, 12
    cdt = W.C * dt
    rng = np.random.default_rng(59)
    org = np.zeros((N, 3))
    for j in range(N):
        tu, tv = j % 5, (2 * j) % 9  # a tile of the 5 x 9, and a corner of it
        corner = step * np.array([tu * 32 + 31 * (j & 1), tv * 16 + 15 * (j >> 1 & 1)])
        out = corner - step * np.array([tu * 32 + 15.5, tv * 16 + 7.5])
        org[j, :2] = corner + out / np.linalg.norm(out) * (405.0 * cdt)
    S = int(math.hypot(nu, nv) * step / cdt) + 7000
    dp = W.sinusoidal_dipoles(org, W.unit_vectors(rng, N), OMEGA0, 1e-11, dt, (S - 1) * dt)
    times = [(S - 1900) * dt, (S - 1000.5) * dt]
    reps = int(1e8 / (N * nu * nv * len(times))) + 1
    iu, iv = np.meshgrid(np.arange(nu), np.arange(nv), indexing="ij")
    pts = np.stack([iu.ravel() * step, iv.ravel() * step, np.zeros(nu * nv)], axis=1)
    # of the points beyond 400 c dt of every source, the 12 nearest to each, and scattered ones
    r = np.linalg.norm(pts[:, None] - org[None], axis=2) / cdt
    r[r.min(axis=1) <= 400.0] = np.inf
    p = np.unique(np.concatenate([np.argsort(r[:, j])[:12] for j in range(N)] + [rng.integers(0, nu * nv, 60)]))
    p = p[np.isfinite(r[p, 0])]
    ref = oracle.fields(pts[p], times, dipoles=dp, kind=kind)
    assert ref["status"] == oracle.OK
    dev = pc.dipoles_to_device(dp)
    err = []
    for frames in (times * reps, times):
        out = pc.pc_fields_plane(ctx, dipoles=dev, origin=(0.0, 0.0, 0.0), eu=(step, 0, 0), ev=(0, step, 0), nu=nu, nv=nv,
                                 times=frames, kind=kind, precision=pc.PC_MIXED)
        err.append({})
        for k in ("E", "B", "phi", "A"):
            g = out[k][:len(times), torch.as_tensor(p, device="cuda")].cpu().numpy().astype(np.float64)
            sc = ref["scale_source"]["E"] / W.C if k == "B" else ref["scale_source"][k]
            err[-1][k] = float(np.max(_norm(g - ref[k]) / sc))
    assert all(err[0][k] <= 2.0 * err[1][k] + 3e-7 for k in err[0]), err


# ------------------------------------------------------------------------------------------------
# devices without the memory for a form's tables
# ------------------------------------------------------------------------------------------------
def _fill(leave):
    """All of the device's free memory but `leave` bytes, as one tensor."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def test_float64_fields_without_memory_for_the_mirror():
    # 64 histories of 10^6 samples: the split form's float32 mirror takes 1.07 GB, of which 0.6 are left
    N, S, P = 64, 1 << 20, 70000
    rng = np.random.default_rng(3)
    dp = W.sinusoidal_dipoles(rng.uniform(0.0, 1e-6, (N, 3)), W.unit_vectors(rng, N), OMEGA0, 1e-11, 1e-18, (S - 1) * 1e-18)
    dev = pc.dipoles_to_device(dp)
    pts = torch.as_tensor(np.concatenate([rng.uniform(0.0, 1e-6, (P, 2)), np.full((P, 1), 1.3e-6)], axis=1), device="cuda")
    c = pc.Context(0)
    ref = {k: v.clone() for k, v in pc.pc_fields(c, dipoles=dev, points=pts, times=[1e-12]).items()}
    c.close()
    c = pc.Context(0)
    pc.pc_fields(c, dipoles=dev, points=pts[:100], times=[1e-12])  # the two-charge form, loaded
    hold = _fill(600 << 20)
    try:
        out = pc.pc_fields(c, dipoles=dev, points=pts, times=[1e-12])
    finally:
        del hold
        c.close()
        torch.cuda.empty_cache()
    for k in ("E", "B", "phi", "A"):
        assert float((out[k] - ref[k]).abs().max() / ref[k].abs().max()) < 1e-10, k


def test_float64_run_without_memory_for_the_mirror():
    # 66 oscillators, 400 000 steps: a mirror of 422 MB next to outputs of 211 MB each; 250 MB are left for it
    steps = 400000
    lod = pc.lo_config_to_device(_cloud(66))
    c = pc.Context(0)
    ref = pc.pc_dipoles_run(c, lod, 1e-18, steps, precision=pc.PC_F64)
    c.close()
    size = sum(v.numel() * v.element_size() for v in ref.values() if torch.is_tensor(v))
    ref = ref["d"].cpu()
    c = pc.Context(0)
    pc.pc_dipoles_run(c, lod, 1e-18, 100, precision=pc.PC_MIXED)  # (the kernels loaded, and scratch for 100 steps)
    hold = _fill(size + (250 << 20))
    try:
        out = pc.pc_dipoles_run(c, lod, 1e-18, steps, precision=pc.PC_F64)
    finally:
        del hold
        c.close()
        torch.cuda.empty_cache()
    d = out["d"].cpu()
    # (both forms' E_d are within 1e-10, which 400 000 steps may add up)
    assert float((d - ref).abs().max() / ref.abs().max()) < 1e-7


@pytest.mark.parametrize("checkpoint", [0, 16000])
def test_float64_gradients_without_memory_for_the_mirror(checkpoint):
    # the whole adjoint's memory but half of its mirror's 42 MB (checkpointed: of a segment's 35)
    steps = 40000
    lod = pc.lo_config_to_device(_cloud(66))
    w = torch.linspace(0.5, 1.5, 66, dtype=torch.float64, device="cuda").view(1, 66)

    def run(c, n=steps):
        return pc.pc_dipoles_adjoint(c, lod, 1e-18, n, w, checkpoint_every=min(checkpoint, n // 2))

    c = pc.Context(0)
    run(c, 100)
    c.close()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    c = pc.Context(0)
    ref = [g.clone() for g in run(c)]
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    c.close()
    mirror = 66 * (32768 if checkpoint else steps + 1) * 16  # (a segment's store: 16000 steps and the depth, a power of 2)
    c = pc.Context(0)
    hold = _fill(used - mirror // 2)
    try:
        got = run(c)
    finally:
        del hold
        c.close()
        torch.cuda.empty_cache()
    # both forms' gradients agree to 1e-10 over 417 steps (tests/test_gpu_far.py)
    for g, r in zip(got, ref):
        assert float((g - r).abs().max() / r.abs().max()) < 1e-10 * steps / 417


# ------------------------------------------------------------------------------------------------
# moments that have grown
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("amp,cell,first", [(1e-11, 3.75e-8, 1600), (1.9e-11, 6e-8, 3200), (2.85e-11, 1e-7, 4800)])
def test_drive_of_grown_moments(ctx, amp, cell, first):
    # a run resumed with declared moments 1.45 times smaller than its samples' (the forms stay to 1.5), pairs around
    # both forms' least distance for these: E_d no further off than in the two-charge form, which declared moments
    # of a hundredth force, by the rms of the same samples (a fifth for their scatter)
    N, dt, n = 100, 1e-18, 400
    cfg = _cloud(N, cell=cell, seed=5)
    cfg.d0[:] = W.E_CHARGE * amp
    lod = pc.lo_config_to_device(cfg)
    state = torch.zeros(pc.pc_dipoles_state_size(ctx, lod, dt), dtype=torch.float64, device="cuda")
    pc.pc_dipoles_run(ctx, lod, dt, first, precision=pc.PC_F64, state_out=state)
    D = int(state[2])
    smp = state[4 + N:].view(N, D + 1, 3).cpu().numpy()
    at, recv = np.linspace(1, n, 40).astype(int), [0, 50, 99]
    rms = {}
    for precision in (pc.PC_F64, pc.PC_MIXED):
        for scale in (1 / 1.45, 0.01):
            decl = pc.lo_config_to_device(cfg)
            decl.d0 *= scale
            f = pc.pc_dipoles_run(ctx, decl, dt, n, precision=precision, state_in=state, want_Ed=True)
            # on the run's own samples
            hist = [np.concatenate([smp[:, :, c], f[k][0, :, 1:].cpu().numpy()], axis=1)
                    for c, k in enumerate(("d", "d_dot", "d_ddot"))]
            ref = _ed_binary128(cfg, hist, (first - D) * dt, (first + at) * dt, recv)
            rms[precision, scale] = float(np.sqrt(np.mean([((f["Ed"][0, i].cpu().numpy()[at] - e) / np.max(np.abs(e))) ** 2
                                                           for e, i in zip(ref, recv)])))
    assert rms[pc.PC_F64, 1 / 1.45] <= 1.2 * rms[pc.PC_F64, 0.01], rms
    assert rms[pc.PC_MIXED, 1 / 1.45] <= 1.2 * rms[pc.PC_MIXED, 0.01], rms


def test_gradients_of_configurations_of_very_unequal_weights(ctx):
    # each configuration's gradients are its own weights' alone, however small these are beside another's: the
    # split reverse's float32 terms (1e-7 of a gradient) keep their scale.  Scaling rounds at 1e-13 or so.
    cfg = _cloud(90, B=2, seed=90)
    w = torch.linspace(0.5, 1.5, 180, dtype=torch.float64, device="cuda").view(2, 90)
    ref = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), cfg.dt, 300, w)
    v = w.clone()
    v[1] *= 1e-40
    got = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), cfg.dt, 300, v)
    for g, r in zip(got, ref):
        assert float((g[0] - r[0]).abs().max() / r[0].abs().max()) < 1e-12
        assert float((g[1] / 1e-40 - r[1]).abs().max() / r[1].abs().max()) < 1e-12


@pytest.mark.parametrize("case", ["fast", "unequal masses", "dense", "not yet there"])
def test_float64_fields_of_mostly_near_pairs(ctx, case):
    # a large call whose pairs are nearly all near takes the general kernel, as a small one (below 1e5 pairs) does:
    # the same bits.  Then 32 frames, a launch's worth, before the field has left any source, and one after that.
    rng = np.random.default_rng(29)
    N, P, box = 20, 6000, 1e-7 if case == "dense" else 1e-6
    dp = W.sinusoidal_dipoles(rng.uniform(0.0, box, (N, 3)), W.unit_vectors(rng, N), OMEGA0, 1e-10 if case == "fast" else 1e-11,
                              1e-18, 9e-15)
    if case == "unequal masses":
        dp.m1 *= 2.0
    z = 4e-6 if case == "not yet there" else box / 2
    pts = torch.as_tensor(np.concatenate([rng.uniform(0.0, box, (P, 2)), np.full((P, 1), z)], axis=1), device="cuda")
    dev = pc.dipoles_to_device(dp)
    times = list(np.linspace(4e-15, 9e-15, 32)) if case == "not yet there" else [6.2e-15, 6.3e-15]
    late = [16e-15] if case == "not yet there" else []
    big = {k: v.clone() for k, v in pc.pc_fields(ctx, dipoles=dev, points=pts, times=times + late).items()}
    for q in range(0, 300, 100):
        small = pc.pc_fields(ctx, dipoles=dev, points=pts[q:q + 100], times=times)
        for k in ("E", "B", "phi", "A"):
            assert torch.equal(big[k][:len(times), q:q + 100], small[k]), k
    if late:
        small = pc.pc_fields(ctx, dipoles=dev, points=pts[:400], times=late)
        for k in ("E", "B", "phi", "A"):
            assert float((big[k][len(times), :400] - small[k][0]).abs().max() / small[k].abs().max()) < 1e-10, k
            assert not torch.equal(big[k][len(times), :400], small[k][0]), k  # the split form's


@pytest.mark.parametrize("dt,amp,omega,z", [(1e-20, 1.5e-12, 1e14, 3e-8), (2.6e-20, 1e-13, 2e13, 4e-9), (1e-18, 1e-11, OMEGA0, 3e-7)])
def test_float64_radiation_fields_of_slow_charges(ctx, dt, amp, omega, z):
    # the radiation field alone, a 1e-4 to 1e-8 part of the Coulomb field so close to slow charges (and as much in
    # the last case): plain errors within 1e-10 of it, at every phase of the moment
    S = 40001
    t0 = 0.25 * 2 * math.pi / omega
    rng = np.random.default_rng(37)
    s = int(t0 / dt) - S // 2  # samples around the moment's peak, and (shifted) around its zero
    for shift in (0, int(t0 / dt)):
        t = (s + shift + np.arange(S)) * dt
        d = W.E_CHARGE * amp * np.tile(np.sin(omega * t), (3, 1))
        one = np.ones(3)
        dp = W.Dipoles(origin=rng.uniform(0.0, z / 20, (3, 3)), axis=W.unit_vectors(rng, 3), q=W.E_CHARGE * one, m1=W.M_E * one,
                       m2=W.M_E * one, d=d, d_dot=W.E_CHARGE * amp * omega * np.tile(np.cos(omega * t), (3, 1)),
                       d_ddot=-omega * omega * d, t0=0.0, dt=dt)
        P = 40003
        pts = np.concatenate([rng.uniform(0.0, z / 4, (P, 2)), np.full((P, 1), z)], axis=1)
        times = [float((S // 2 + k) * dt + 1.05 * z / W.C) for k in (-3000, 4.3, 5000.5)]
        out = pc.pc_fields(ctx, dipoles=pc.dipoles_to_device(dp), points=torch.as_tensor(pts, device="cuda"), times=times,
                           kind=pc.PC_RADIATION)
        ref = oracle.fields_x(pts[:60], times, dipoles=dp, kind=pc.PC_RADIATION)
        scale = oracle.fields(pts[:60], times, dipoles=dp, kind=pc.PC_RADIATION)["scale_source"]["E"]
        for k, sc in (("E", scale), ("B", scale / W.C)):
            e = _norm(out[k][:, :60].cpu().numpy() - ref[k]) / np.maximum(_norm(ref[k]), 1e-3 * sc)
            assert float(np.max(e)) <= 1e-10, (k, shift, float(np.max(e)))


@pytest.mark.parametrize("steps", [60, 417])
@pytest.mark.parametrize("every", [2, 3, 66])
def test_split_reverse_of_some_unequal_masses(ctx, every, steps):
    # a pair is far by its source's masses, whatever the receiver's: gradients of configurations with both kinds as
    # in tests/test_gpu_far.py::test_split_reverse_against_the_two_charge_form
    cfg = _cloud(66, seed=47)
    cfg.m1[:, ::every] *= 1.5
    w = torch.linspace(0.5, 1.5, 66, dtype=torch.float64, device="cuda").view(1, 66)
    got = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), cfg.dt, steps, w)
    cfg.m1 = np.nextafter(cfg.m1, np.inf)
    ref = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), cfg.dt, steps, w)
    for g, r in zip(got, ref):
        assert float((g - r).abs().max() / r.abs().max()) < 1e-10
