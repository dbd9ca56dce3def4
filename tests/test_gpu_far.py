"""The first-order far form of the mixed path (csrc/pc_far_f32.cuh) against the FP64 oracle, at the edges of
what it accepts: whole plane calls large enough to be asked whether they are far, compared at scattered
points within the mixed path's bounds (tests/test_gpu_fields.py: 1e-5 over the source scale)."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2107_12437_gb300 as pc
import workloads as W
from test_gpu_fields import compare

pytestmark = pytest.mark.gpu

OMEGA0 = 2 * math.pi * 200e12


@pytest.fixture(scope="module")
def ctx():
    c = pc.Context(0)
    yield c
    c.close()


def _sources(N, seed=5, amp=1e-11, t_end=15e-15):
    rng = np.random.default_rng(seed)
    return W.sinusoidal_dipoles(rng.uniform(0.0, 1e-6, (N, 3)), W.unit_vectors(rng, N), OMEGA0, amp, 1e-18, t_end)


def _check(ctx, dp, nu, nv, times, kind=pc.PC_TOTAL, r_excl=0.0, step=0.5e-9, z=0.4e-6, origin=(0.1e-6, 0.2e-6),
           per_frame=150, nonempty_mask=False):
    # the frames an odd number of times over, so that the call is large enough (1e8 triples) for the far kernel
    times = list(times)
    reps = int(1e8 / (dp.origin.shape[0] * nu * nv * len(times))) + 1
    out = pc.pc_fields_plane(ctx, dipoles=pc.dipoles_to_device(dp), origin=(*origin, z), eu=(step, 0, 0),
                             ev=(0, step, 0), nu=nu, nv=nv, times=times * (reps | 1), kind=kind,
                             precision=pc.PC_MIXED, r_excl=r_excl)
    out = {k: v[:len(times)] for k, v in out.items()}
    rng = np.random.default_rng(3)
    # scattered points, the grid's corners among them
    p = np.unique(np.r_[0, nv - 1, (nu - 1) * nv, nu * nv - 1, rng.integers(0, nu * nv, per_frame)])
    pts = np.stack([origin[0] + (p // nv) * step, origin[1] + (p % nv) * step, np.full(p.size, z)], axis=1)
    ref = oracle.fields(pts, times, dipoles=dp, kind=kind, r_excl=r_excl)
    assert ref["status"] == oracle.OK
    if nonempty_mask:
        assert ref["mask"].any() and not ref["mask"].all()
    sub = {k: v[:, torch.as_tensor(p, device="cuda")].cpu().numpy() if k != "mask"
           else v[:, torch.as_tensor(p, device="cuda")].cpu() for k, v in out.items()}
    # where every source still rests with no moment the fields are zero: exactly so in both, and out of the
    # relative measures
    rest = ref["scale_source"]["E"] == 0.0
    for k in ("E", "B", "phi", "A"):
        assert not np.any(sub[k][rest]) and not np.any(ref[k][rest]), k
    sub["mask"], ref["mask"] = sub["mask"].clone(), ref["mask"].copy()
    sub["mask"][torch.as_tensor(rest)] = 1
    ref["mask"][rest] = 1
    compare(sub, ref, pc.PC_MIXED)


@pytest.mark.parametrize("kind", [pc.PC_TOTAL, pc.PC_COULOMB, pc.PC_RADIATION])
@pytest.mark.parametrize("nu,nv,frames", [(301, 517, 1), (517, 301, 2), (33, 2047, 5), (2047, 17, 3)])
def test_ragged_planes_and_frame_counts(ctx, nu, nv, frames, kind):
    # 70 sources (a second, partial chunk), partial tiles in both directions, odd and even frame counts
    _check(ctx, _sources(70), nu, nv, 10.3e-15 + 0.7e-15 * np.arange(frames), kind)


def test_more_frames_than_a_launch(ctx):
    _check(ctx, _sources(33), 160, 160, 10.1e-15 + 0.1e-15 * np.arange(35), per_frame=20)


@pytest.mark.parametrize("amp", [1e-13, 2.9e-11, 1e-10, 1e-9])
def test_amplitudes_around_the_limits(ctx, amp):
    # below 2.86e-11 m at 200 THz the charges stay under kFarV; above, every source is near
    _check(ctx, _sources(64, amp=amp), 401, 403, [10.4e-15])


def test_unequal_masses_stay_near(ctx):
    dp = _sources(64)
    dp.m1[::2] = 1836.0 * W.M_E
    dp.m2[1::4] = 1.0001 * W.M_E
    _check(ctx, dp, 401, 403, [11.4e-15])


def test_retarded_times_at_both_ends_of_the_history(ctx):
    # frames within the light-crossing time of the first sample (static sources) and at the last one
    dp = _sources(64, t_end=6e-15)
    _check(ctx, dp, 401, 403, [0.4e-15, 1.6e-15, 6e-15])


def test_exclusion_radius_beyond_the_far_distance(ctx):
    # charges within 200 nm are skipped and masked
    _check(ctx, _sources(64), 401, 403, [11.4e-15], r_excl=200e-9, nonempty_mask=True)


def test_coarse_grid_tiles_are_never_wholly_far(ctx):
    # grid steps of 40 nm: a tile spans more than a micrometre
    _check(ctx, _sources(64), 401, 403, [11.4e-15], step=4e-8)


@pytest.mark.parametrize("kind", [pc.PC_TOTAL, pc.PC_COULOMB, pc.PC_RADIATION])
@pytest.mark.parametrize("case", ["cube", "amplitude", "masses", "wide"])
def test_large_lists_take_the_far_form_by_pair(ctx, case, kind):
    # 28 801 points (a last CTA of one) around 70 sources (a partial group and chunk), two frames: points among
    # the sources and, "wide", micrometres away, where the anchor's and a point's delays differ by 10 000
    # samples; charges as fast as the limit; sources that are never far
    dp = _sources(70, amp=2.8e-11 if case == "amplitude" else 1e-11)
    if case == "masses":
        dp.m1[::3] = 1836.0 * W.M_E
    rng = np.random.default_rng(12)
    pts = rng.uniform(0.0, 1e-6, (28801, 3))
    if case == "wide":
        pts[::2] += rng.uniform(-1.5e-6, 1.5e-6, pts[::2].shape)
    times = [11.3e-15, 13.05e-15]
    out = pc.pc_fields(ctx, dipoles=pc.dipoles_to_device(dp), points=torch.as_tensor(pts, device="cuda"), times=times,
                       kind=kind, precision=pc.PC_MIXED)
    p = np.unique(np.r_[0, 28800, rng.integers(0, 28801, 200)])
    ref = oracle.fields(pts[p], times, dipoles=dp, kind=kind)
    assert ref["status"] == oracle.OK
    sub = {k: v[:, torch.as_tensor(p, device="cuda")].cpu() for k, v in out.items()}
    sub = {k: v if k == "mask" else v.numpy() for k, v in sub.items()}
    compare(sub, ref, pc.PC_MIXED)


# ------------------------------------------------------------------------------------------------
# the oscillator run's far drive (grid path, mixed)
# ------------------------------------------------------------------------------------------------
def _cloud(N, cell=37.5e-9, seed=11, ring=False, B=1):
    """N oscillators, one in each of N lattice cells (no two closer than 5 nm)."""
    rng = np.random.default_rng(seed)
    g = int(math.ceil(N ** (1 / 3) - 1e-9))
    org, ax = [], []
    for _ in range(B):
        c = np.stack(np.unravel_index(rng.permutation(g ** 3)[:N], (g, g, g)), axis=1)
        org.append(c * cell + rng.uniform(0.0, cell - 5e-9, (N, 3)))
        ax.append(W.unit_vectors(rng, N))
    return W.lo_batch(np.array(org), np.array(ax), OMEGA0, 1e-11, 1e-18, 0, 0)


def _err(a, b):
    return float(((a - b).abs().amax(-1) / b.abs().amax()).max())


@pytest.mark.parametrize("N,steps", [(65, 700), (96, 333), (130, 400), (257, 203)])
def test_far_drive_against_oracle(ctx, N, steps):
    # past the light-crossing time of the cloud, so that pairs have been static, crossing t = 0 and moving;
    # a last block of fewer than 16 steps; slices that do not divide the sources
    cfg = _cloud(N)
    cfg.n_steps = steps
    ref = oracle.dipoles_run(cfg)
    assert ref["status"] == oracle.OK
    out = pc.pc_dipoles_run(ctx, pc.lo_config_to_device(cfg), cfg.dt, steps, precision=pc.PC_MIXED, want_Ed=True)
    for k in ("d", "d_dot", "Ed"):
        g = out[k][0].cpu().numpy()
        assert np.max(np.abs(g - ref[k])) < 1e-5 * np.max(np.abs(ref[k])), k


@pytest.mark.parametrize("slices", [0, 1, 3, 12])
@pytest.mark.parametrize("spacing,near", [(1.0, 0.0), (0.5, 0.0), (1.0, 60e-9), (40.0, 0.0)])
def test_far_drive_against_float64(ctx, slices, spacing, near):
    # the float64 run's driving fields within 3e-6 of their largest value (float32 sums of some hundred
    # terms of 1e-7 each); blocks shorter than 16 steps (spacing 0.5: origins down to 2.5 nm, 7 steps),
    # near sources in float64, and a cloud that stays static for the whole run
    cfg = _cloud(100, B=2)
    cfg.origin *= spacing
    lod = pc.lo_config_to_device(cfg)
    f = pc.pc_dipoles_run(ctx, lod, cfg.dt, 450, precision=pc.PC_F64, want_Ed=True)
    try:
        pc.pc_set_run_tiling(ctx, slices)
        m = pc.pc_dipoles_run(ctx, lod, cfg.dt, 450, precision=pc.PC_MIXED, near_f64=near, want_Ed=True)
    finally:
        pc.pc_set_run_tiling(ctx, 0)
    assert _err(m["Ed"], f["Ed"]) < 3e-6
    assert _err(m["d"], f["d"]) < 1e-9


def test_far_drive_leaves_and_returns_where_moments_pass_its_limits(ctx):
    # a state whose oldest samples are three times the largest initial moment (beyond the limits): the
    # resumed run's first blocks take the two-charge form, the later ones the far form with its carried
    # sums formed anew; the float64 run resumed from the same state is the reference
    cfg = _cloud(80)
    lod = pc.lo_config_to_device(cfg)
    n = pc.pc_dipoles_state_size(ctx, lod, cfg.dt)
    state = torch.zeros(n, dtype=torch.float64, device="cuda")
    first = 960  # a whole number of blocks, beyond the state's depth
    pc.pc_dipoles_run(ctx, lod, cfg.dt, first, precision=pc.PC_F64, state_out=state)
    D = int(state[2])
    assert D < first
    state[4 + 80:].view(80, D + 1, 3)[:, :20] *= 3.0
    f = pc.pc_dipoles_run(ctx, lod, cfg.dt, 200, precision=pc.PC_F64, state_in=state, want_Ed=True)
    m = pc.pc_dipoles_run(ctx, lod, cfg.dt, 200, precision=pc.PC_MIXED, state_in=state, want_Ed=True)
    assert _err(m["Ed"], f["Ed"]) < 3e-6
    assert _err(m["d"], f["d"]) < 1e-9
    # and amplitudes that the limits of smaller declared moments forbid throughout
    small = pc.lo_config_to_device(cfg)
    small.d0 *= 0.1
    m = pc.pc_dipoles_run(ctx, small, cfg.dt, 200, precision=pc.PC_MIXED, state_in=state, want_Ed=True)
    assert _err(m["Ed"], f["Ed"]) < 3e-6


def test_far_drive_refuses_what_is_not_a_number(ctx):
    cfg = _cloud(80)
    cfg.omega0[0, 7] = np.nan
    with pytest.raises(pc.PcError):
        pc.pc_dipoles_run(ctx, pc.lo_config_to_device(cfg), cfg.dt, 400, precision=pc.PC_MIXED)


@pytest.mark.parametrize("amp,near", [(1e-12, 0.0), (1.9e-11, 0.0), (2.8e-11, 0.0), (2.8e-11, 20e-9)])
def test_mid_pairs_against_float64(ctx, amp, near):
    # pairs from 20 samples (6 nm) on with charges up to amp / 6 nm = 5e-3 of their distance apart, below
    # where the cubic form ends (1e-2) and where charges are too fast (2.86e-11 m); the bounds above
    cfg = _cloud(200, cell=10.2e-9, seed=7)
    cfg.d0[:] = W.E_CHARGE * amp
    cfg.m1[0, ::7] *= 1.5  # and sources that never are mid pairs
    lod = pc.lo_config_to_device(cfg)
    f = pc.pc_dipoles_run(ctx, lod, cfg.dt, 340, precision=pc.PC_F64, want_Ed=True)
    m = pc.pc_dipoles_run(ctx, lod, cfg.dt, 340, precision=pc.PC_MIXED, near_f64=near, want_Ed=True)
    assert _err(m["Ed"], f["Ed"]) < 3e-6
    assert _err(m["d"], f["d"]) < 1e-9


def test_mid_pairs_of_several_groups_of_a_slice(ctx):
    # one slice of 300 sources, staged 32 at a time, mid pairs in every group: each group's staged entries
    # have to be read before the next group's take their place, in both passes of a run's first block (the
    # resumed run starts with two).  The same run in slices of 25 differs by the order of its sums alone
    cfg = _cloud(300, cell=10.2e-9, seed=13)
    lod = pc.lo_config_to_device(cfg)
    state = torch.zeros(pc.pc_dipoles_state_size(ctx, lod, cfg.dt), dtype=torch.float64, device="cuda")
    f = pc.pc_dipoles_run(ctx, lod, cfg.dt, 203, precision=pc.PC_F64, state_out=state, want_Ed=True)
    g = pc.pc_dipoles_run(ctx, lod, cfg.dt, 100, precision=pc.PC_F64, state_in=state, want_Ed=True)
    try:
        for slices in (1, 12):
            pc.pc_set_run_tiling(ctx, slices)
            m = pc.pc_dipoles_run(ctx, lod, cfg.dt, 203, precision=pc.PC_MIXED, want_Ed=True)
            again = pc.pc_dipoles_run(ctx, lod, cfg.dt, 203, precision=pc.PC_MIXED, want_Ed=True)
            assert torch.equal(m["Ed"], again["Ed"])
            assert _err(m["Ed"], f["Ed"]) < 3e-6
            m = pc.pc_dipoles_run(ctx, lod, cfg.dt, 100, precision=pc.PC_MIXED, state_in=state, want_Ed=True)
            assert _err(m["Ed"], g["Ed"]) < 3e-6
    finally:
        pc.pc_set_run_tiling(ctx, 0)


# ------------------------------------------------------------------------------------------------
# the grid path's block loop in one cooperative launch
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("N,B,precision,near,steps", [
    (65, 1, "mixed", 0.0, 203), (153, 1, "mixed", 60e-9, 203), (90, 3, "mixed", 0.0, 333), (307, 1, "mixed", 0.0, 16),
    (2128, 1, "mixed", 0.0, 40), (65, 1, "f64", 0.0, 203), (304, 1, "f64", 0.0, 50), (90, 2, "f64", 0.0, 333)])
def test_cooperative_loop_is_the_loop_of_launches(ctx, monkeypatch, N, B, precision, near, steps):
    # one, two and up to fourteen receivers a CTA, a last CTA with fewer, receivers of two configurations in a
    # CTA, a single block, a partial last one; both stores; resumed from a state with samples beyond the
    # limits, which the blocks must notice at the same ones
    cfg = _cloud(N, B=B, seed=N)
    lod = pc.lo_config_to_device(cfg)
    kw = dict(precision=pc.PC_MIXED if precision == "mixed" else pc.PC_F64, near_f64=near)
    state = torch.zeros(pc.pc_dipoles_state_size(ctx, lod, cfg.dt), dtype=torch.float64, device="cuda")

    def runs():
        full = pc.pc_dipoles_run(ctx, lod, cfg.dt, steps, want_Ed=True, **kw)
        ring = pc.pc_dipoles_run(ctx, lod, cfg.dt, steps, want_history=False, state_out=state, **kw)
        D = int(state[2])
        state[4 + B * N:].view(B * N, D + 1, 3)[:3, -5:-3] *= 4.0
        back = pc.pc_dipoles_run(ctx, lod, cfg.dt, steps, state_in=state, want_Ed=True, **kw)
        return [r[k].clone() for r in (full, ring, back) for k in sorted(r) if torch.is_tensor(r[k])] + [state.clone()]

    got = runs()
    monkeypatch.setenv("PYCHARGE_GB300_HOST_LOOP", "1")
    for g, h in zip(got, runs()):
        assert torch.equal(g, h)


def test_cooperative_runs_on_two_streams(ctx):
    # two threads with a context and a stream each, at the same time
    import threading

    cfgs = [_cloud(180, seed=1), _cloud(250, seed=2)]
    lods = [pc.lo_config_to_device(c) for c in cfgs]
    ref = [pc.pc_dipoles_run(ctx, lo, 1e-18, 400, precision=pc.PC_MIXED)["d"].clone() for lo in lods]
    torch.cuda.synchronize()
    out = [None, None]

    def work(k):
        c, st = pc.Context(0), torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(5):
                out[k] = pc.pc_dipoles_run(c, lods[k], 1e-18, 400, precision=pc.PC_MIXED, stream=st)["d"]
        st.synchronize()
        c.close()

    t = [threading.Thread(target=work, args=(k,)) for k in (0, 1)]
    [x.start() for x in t]
    [x.join() for x in t]
    assert all(torch.equal(o, r) for o, r in zip(out, ref))


# ------------------------------------------------------------------------------------------------
# the oscillator run's split drive (grid path, float64)
# ------------------------------------------------------------------------------------------------
def _ed_binary128(cfg, hist, t0, times, receivers):
    """E_d of some receivers on a history (d, d', d'' [N][S] from time t0 on) in binary128."""
    out = []
    for i in receivers:
        o = np.arange(cfg.N) != i
        dps = W.Dipoles(origin=cfg.origin[0, o], axis=cfg.axis[0, o], q=cfg.q[0, o], m1=cfg.m1[0, o], m2=cfg.m2[0, o],
                        d=hist[0][o], d_dot=hist[1][o], d_ddot=hist[2][o], t0=t0, dt=cfg.dt)
        r = oracle.fields_x(cfg.origin[0, i][None], times, dipoles=dps)
        assert r["status"] == oracle.OK
        out.append(r["E"][:, 0] @ cfg.axis[0, i])
    return np.array(out)


@pytest.mark.parametrize("case", ["cloud", "dense", "unequal masses", "fast", "slices"])
def test_split_drive_against_binary128(ctx, case):
    # every receiver's E_d on the run's own history within 1e-10 of its largest value, the float64 path's
    # bound (two charges at 1e5 times their distance round to 1e-11 of their field)
    cfg = _cloud(90, seed=29)
    steps = 420
    if case == "dense":
        cfg.origin *= 0.45  # origins down to 2.3 nm, blocks of 7 steps
    if case == "unequal masses":
        cfg.m1[0, ::3] *= 1.5
    if case == "fast":
        cfg.omega0 *= 30.0  # charges beyond kSplitV: every pair in the two-charge form
    try:
        pc.pc_set_run_tiling(ctx, 7 if case == "slices" else 0)
        f = pc.pc_dipoles_run(ctx, pc.lo_config_to_device(cfg), cfg.dt, steps, precision=pc.PC_F64, want_Ed=True)
    finally:
        pc.pc_set_run_tiling(ctx, 0)
    h = {k: f[k][0].cpu().numpy() for k in ("d", "d_dot", "d_ddot", "Ed")}
    at = np.r_[np.arange(1, steps, 13), steps - 1, steps]
    recv = [0, 17, 44, 89]
    ref = _ed_binary128(cfg, (h["d"], h["d_dot"], h["d_ddot"]), 0.0, at * cfg.dt, recv)
    for e, i in zip(ref, recv):
        assert np.max(np.abs(h["Ed"][i, at] - e)) < 1e-10 * np.max(np.abs(e)), i


def test_split_drive_leaves_and_returns_where_moments_pass_its_limits(ctx):
    # as for the mixed drive: oldest samples of the resumed state beyond the limits
    cfg = _cloud(80)
    lod = pc.lo_config_to_device(cfg)
    first, n = 960, 200
    state = torch.zeros(pc.pc_dipoles_state_size(ctx, lod, cfg.dt), dtype=torch.float64, device="cuda")
    pc.pc_dipoles_run(ctx, lod, cfg.dt, first, precision=pc.PC_F64, state_out=state)
    D = int(state[2])
    smp = state[4 + 80:].view(80, D + 1, 3)
    smp[:, :20] *= 3.0
    f = pc.pc_dipoles_run(ctx, lod, cfg.dt, n, precision=pc.PC_F64, state_in=state, want_Ed=True)
    hist = [np.concatenate([smp[:, :, c].cpu().numpy(), f[k][0, :, 1:].cpu().numpy()], axis=1)
            for c, k in enumerate(("d", "d_dot", "d_ddot"))]
    at = np.arange(1, n + 1, 7)
    recv = [0, 33, 79]
    ref = _ed_binary128(cfg, hist, (first - D) * cfg.dt, (first + at) * cfg.dt, recv)
    for e, i in zip(ref, recv):
        assert np.max(np.abs(f["Ed"][0, i, at].cpu().numpy() - e)) < 1e-10 * np.max(np.abs(e)), i


# ------------------------------------------------------------------------------------------------
# the float64 field sum's split form
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("kind", [pc.PC_TOTAL, pc.PC_COULOMB, pc.PC_RADIATION])
@pytest.mark.parametrize("case", ["1 pm", "20 pm", "100 pm", "unequal masses", "list", "ends"])
def test_split_fields_against_binary128(ctx, case, kind):
    # plain relative errors of the float64 path within 1e-10 at every point that no cancellation between
    # the sources deeper than 1e3 affects (the bound of the two-charge form, tests/test_gpu_fields.py)
    amp = {"1 pm": 1e-12, "20 pm": 2e-11, "100 pm": 1e-10}.get(case, 1e-11)
    dp = _sources(41, amp=amp, t_end=6e-15 if case == "ends" else 15e-15)
    times = [3.5e-15, 6e-15] if case == "ends" else [10.4e-15, 12.5e-15]
    if case == "unequal masses":
        dp.m1[::2] *= 3.0
    nu, nv, step, z = 129, 257, 1.1e-9, 0.45e-6
    dev = pc.dipoles_to_device(dp)
    rng = np.random.default_rng(8)
    p = rng.integers(0, nu * nv, 90)
    pts = np.stack([0.3e-6 + (p // nv) * step, 0.2e-6 + (p % nv) * step, np.full(p.size, z)], axis=1)
    if case == "list":
        allp = rng.uniform(0.0, 1e-6, (nu * nv, 3))
        out = pc.pc_fields(ctx, dipoles=dev, points=torch.as_tensor(allp, device="cuda"), times=times, kind=kind)
        pts = allp[p]
    else:
        out = pc.pc_fields_plane(ctx, dipoles=dev, origin=(0.3e-6, 0.2e-6, z), eu=(step, 0, 0), ev=(0, step, 0), nu=nu,
                                 nv=nv, times=times, kind=kind)
    ref = oracle.fields_x(pts, times, dipoles=dp, kind=kind)
    scale = oracle.fields(pts, times, dipoles=dp, kind=kind)["scale_source"]
    assert ref["status"] == oracle.OK and not out["mask"].any()
    norm = lambda v: np.abs(v) if v.ndim == 2 else np.linalg.norm(v, axis=-1)  # noqa: E731
    for k in ("E", "B", "phi", "A"):
        g = out[k][:, torch.as_tensor(p, device="cuda")].cpu().numpy()
        sc = scale["E"] / W.C if k == "B" else scale[k]
        assert np.all(norm(g - ref[k]) <= 1e-10 * np.maximum(norm(ref[k]), 1e-3 * sc)), k


# ------------------------------------------------------------------------------------------------
# the adjoint's split reverse (grid path)
# ------------------------------------------------------------------------------------------------
@pytest.mark.parametrize("checkpoint", [0, 100])
@pytest.mark.parametrize("N,B,steps,scale", [(66, 1, 417, 1.0), (90, 2, 300, 1.0), (130, 1, 203, 0.6), (70, 1, 64, 30.0)])
def test_split_reverse_against_the_two_charge_form(ctx, N, B, steps, scale, checkpoint):
    # masses one rounding apart keep every pair in the two-charge form, forward and reverse, and move the
    # result by as much: gradients within 1e-10 of each group's largest (both forms round at 1e-12)
    cfg = _cloud(N, B=B, seed=N)
    cfg.origin *= scale
    w = torch.linspace(0.5, 1.5, B * N, dtype=torch.float64, device="cuda").view(B, N)
    got = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), cfg.dt, steps, w, checkpoint_every=checkpoint)
    cfg.m1 = np.nextafter(cfg.m1, np.inf)
    ref = pc.pc_dipoles_adjoint(ctx, pc.lo_config_to_device(cfg), cfg.dt, steps, w, checkpoint_every=checkpoint)
    for g, r, k in zip(got, ref, ("origin", "omega0", "d0")):
        assert float((g - r).abs().max()) < 1e-10 * float(r.abs().max()), k
