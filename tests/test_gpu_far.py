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
    out = pc.pc_fields_plane(ctx, dipoles=pc.dipoles_to_device(dp), origin=(*origin, z), eu=(step, 0, 0),
                             ev=(0, step, 0), nu=nu, nv=nv, times=list(times), kind=kind, precision=pc.PC_MIXED,
                             r_excl=r_excl)
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
