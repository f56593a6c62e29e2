"""The ways a pass can be organised: clusters of one to eight blocks for small
grids, one or two threads per lane, one to four column blocks in flight, rounds
whose copies start during the round before. Every one evaluates the same
butterflies and projections, so the phases of a run agree bit for bit whichever
way its grid, batch and block count select; the gaps agree to the rounding of
the block sums. The short form of the projections (all values normal) and the
long one (zeros) are compared with the oracle."""

import numpy as np
import pytest

import oracle.gs_oracle as O
from paper_1302_0120_gb300 import synthetic as S
from tests.gpu_util import GROUPING_RTOL, aligned_rel_err, gpu_gs
from tests.test_gpu_batch import make_batch, run_batched

pytestmark = pytest.mark.gpu


def _same(a, b):
    assert a[3] == 0 and b[3] == 0
    assert np.array_equal(a[0], b[0]), np.max(np.abs(a[0] - b[0]))
    np.testing.assert_allclose(a[1], b[1], rtol=GROUPING_RTOL, atol=0)
    np.testing.assert_allclose(a[2], b[2], rtol=GROUPING_RTOL, atol=0)


# masks of a batch: the cluster shrinks as the batch grows (64 x 64: four blocks
# for one mask, two for 64; 128 x 128: eight, four, then the persistent kernel)
@pytest.mark.parametrize("ny,nx,masks", [
    (32, 32, 1), (32, 32, 64), (64, 64, 64), (256, 32, 20), (64, 256, 2), (128, 128, 1), (128, 128, 30),
    (128, 128, 60), (128, 256, 1), (256, 128, 12), (256, 128, 40),
])
def test_clusters_match_persistent_kernel(ny, nx, masks):
    I, P = make_batch(masks, ny, nx, nspots=4)
    got = run_batched(I, P, 5)
    ref = run_batched(I, P, 5, grid=5)
    _same(got, ref)


# few blocks make every pass several rounds, the last one ragged; None is the
# grid that a run chooses (one round for these masks)
@pytest.mark.parametrize("ny,nx,grid", [
    (1024, 1024, 9), (1024, 1024, 41), (512, 512, 7), (256, 256, 3), (512, 1024, 11), (1024, 256, 6),
    (2048, 1024, 23), (64, 2048, 3), (128, 512, 1),
])
def test_rounds_match_one_round(ny, nx, grid):
    I = S.spot_target(41, ny, nx, 9, (0.5, 1.0))
    phi0 = S.random_phase(42, ny, nx)
    _same(gpu_gs(I, phi0, 4), gpu_gs(I, phi0, 4, grid=grid))


# batches of one grid and of single runs, on the grid of the whole batch
@pytest.mark.parametrize("masks,ny,nx", [(9, 1024, 1024), (11, 512, 512), (17, 256, 256), (3, 2048, 1024),
                                         (5, 600, 800), (4, 250, 360), (3, 1024, 1280)])
def test_batches_match_single_runs(masks, ny, nx):
    I, P = make_batch(masks, ny, nx, nspots=8)
    ph, r, g, st = run_batched(I, P, 3)
    for k in (0, masks // 2, masks - 1):
        _same((ph[k], r[k], g[k], st), gpu_gs(I[k], P[k], 3))


# A constant start transforms to a single frequency: the other values of F u are
# exact zeros on these grids, which take phase 0 (zero rule of the projections).
@pytest.mark.parametrize("n,grid", [(64, None), (64, 2), (128, None), (256, None), (512, None), (1024, None)])
def test_exact_zeros_take_phase_zero(n, grid):
    I = S.spot_target(51, n, n, 7, (0.5, 1.0))
    phi0 = np.zeros((n, n), np.float32)
    ph, r, g, st = gpu_gs(I, phi0, 1, grid=grid)
    assert st == 0
    # the oracle's transform leaves residues of 1e-16 where the exact one has
    # zeros: the step from the exact spectrum instead, F u0 = N at DC only
    m = O.target_amplitude(I)
    v = np.fft.ifft2(m) * n
    # v is real, so that the phase of its smallest values is all rounding: with
    # an FP32 error of 5e-7 rms in v, the pixels above 0.05 rms are off by 2e-6
    # in the root mean square (E[1/v^2] = 16 there)
    keep = np.abs(v) > 0.05 * np.sqrt(np.mean(np.abs(v) ** 2))
    assert aligned_rel_err(ph[keep], (v / np.abs(v))[keep]) <= 1e-5
    r0 = np.sqrt(((np.where(np.arange(n * n).reshape(n, n) == 0, float(n), 0.0) - m) ** 2).sum()) / n
    assert abs(r[0] - r0) <= 1e-5 * r0


@pytest.mark.parametrize("ny,nx", [(1024, 1280), (480, 640), (1500, 1500), (9, 1536)])
def test_general_teams_parity(ny, nx):
    I = S.spot_target(61, ny, nx, 6, (0.5, 1.0)) if min(ny, nx) > 20 else np.eye(ny, nx, 5, dtype=np.float32)
    phi0 = S.random_phase(62, ny, nx)
    ph, r, g, st = gpu_gs(I, phi0, 2)
    assert st == 0
    ref = O.gs_run(I, phi0, 2)
    np.testing.assert_allclose(r, ref["r"], rtol=1e-3)
    one = gpu_gs(I, phi0, 1)[0]
    u, _, _ = O.gs_step(np.exp(1j * phi0.astype(np.float64)), O.target_amplitude(I))
    assert aligned_rel_err(one, u) <= 1e-5


def _laser_with_dark_pixels(ny, nx):
    """A beam profile with some pixels switched off (p = 0)."""
    p = S.laser_amplitude(ny, nx)
    p[::7, ::5] = 0.0
    return p


def _laser_run(I, P, p, iters, grid=None, masks=1):
    import torch

    from paper_1302_0120_gb300 import GerchbergSaxton, build_lib
    from paper_1302_0120_gb300 import _binding as B

    build_lib.build()
    ny, nx = I.shape[-2:]
    It, Pt, pt = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (I, P, p))
    with GerchbergSaxton(nx, ny, max_batch=masks) as gs:
        gs.set_slm_amplitude(pt)
        if grid:
            gs.set_grid(grid)
        out = gs.run(It, Pt, iters) if masks == 1 else gs.run_batched(It, Pt, iters)
        st = gs.status()
        assert B.gs_check_workspace(gs.handle) == B.GS_OK
        return tuple(x.cpu().numpy() for x in out) + (st,)


# Under a laser amplitude a row pass stages the row's amplitude in shared memory
# beside the fetched rows or in their place: rounds after the first, for two
# threads a lane, one, and the grids with a kernel of their own (nx = 4096 and
# ny >= 2048, 2048 x 4096; several rounds on any grid).
@pytest.mark.parametrize("ny,nx,grid", [(64, 64, 1), (512, 512, 7), (1024, 1024, 9), (2048, 1024, 23), (600, 800, 11),
                                        (2048, 4096, 37), (4096, 2048, 41)])
def test_laser_rounds_match_one_round(ny, nx, grid):
    I = S.spot_target(71, ny, nx, 9, (0.5, 1.0))
    phi0 = S.random_phase(72, ny, nx)
    p = _laser_with_dark_pixels(ny, nx)
    _same(_laser_run(I, phi0, p, 3), _laser_run(I, phi0, p, 3, grid=grid))


@pytest.mark.parametrize("masks,ny,nx", [(9, 1024, 1024), (11, 512, 512), (3, 600, 800)])
def test_laser_batches_match_single_runs(masks, ny, nx):
    I, P = make_batch(masks, ny, nx, nspots=8)
    p = _laser_with_dark_pixels(ny, nx)
    ph, r, g, st = _laser_run(I, P, p, 3, masks=masks)
    for k in (0, masks // 2, masks - 1):
        _same((ph[k], r[k], g[k], st), _laser_run(I[k], P[k], p, 3))


# One step in FP64 (torch.fft) on the grids whose laser runs have a kernel of
# their own, and their neighbours on the common one. The FP32 step's error there
# is some 1e-6 in the root mean square (as for p = 1, test_gpu_parity.py).
@pytest.mark.parametrize("ny,nx", [(4096, 4096), (2048, 4096), (4096, 2048), (1024, 4096), (2048, 2048)])
def test_laser_step_on_long_rows(ny, nx):
    import torch

    I = S.spot_target(73, ny, nx, 20, (0.5, 1.0))
    phi0 = S.random_phase(74, ny, nx)
    p = _laser_with_dark_pixels(ny, nx)
    ph, r, g, st = _laser_run(I, phi0, p, 1)
    assert st == 0
    I64, phi64, p64 = (torch.from_numpy(x).cuda().double() for x in (I, phi0, p))
    energy = (p64 * p64).sum()
    m = torch.sqrt(I64 * (energy / I64.sum()))
    Y = torch.fft.fft2(torch.polar(p64, phi64)) / (ny * nx) ** 0.5
    v = torch.fft.ifft2(torch.polar(m, torch.angle(Y))) * (ny * nx) ** 0.5
    r0 = float(torch.sqrt(((Y.abs() - m) ** 2).sum() / energy))
    g0 = float(torch.sqrt(((v.abs() - p64) ** 2).sum() / energy))
    assert abs(r[0] - r0) <= 1e-5 * r0 and abs(g[0] - g0) <= 1e-5 * g0
    a = torch.polar(p64, torch.from_numpy(ph).cuda().double())
    b = torch.polar(p64, torch.angle(v))
    c = (a.conj() * b).sum()
    assert float(torch.linalg.norm(a * (c / c.abs()) - b) / torch.linalg.norm(b)) <= 1e-5


# The target start: a column pass that transforms the amplitude itself, without
# copies ahead, then a row pass, each in several rounds on a small grid.
@pytest.mark.parametrize("ny,nx,grid", [(256, 256, 3), (512, 512, 7), (1024, 1024, 9), (2048, 1024, 23), (600, 800, 11),
                                        (480, 640, 9)])
def test_target_start_rounds_match_one_round(ny, nx, grid):
    import torch

    from paper_1302_0120_gb300 import GerchbergSaxton, build_lib

    build_lib.build()
    I = torch.from_numpy(S.spot_target(75, ny, nx, 9, (0.5, 1.0))).cuda()
    out = []
    for g in (0, grid):
        with GerchbergSaxton(nx, ny, init_from_target=True) as gs:
            gs.set_grid(g)
            res = gs.run(I, None, 3)
            out.append(tuple(x.cpu().numpy() for x in res) + (gs.status(),))
    _same(*out)


# |z|^2 below the smallest normal number takes the long form of the projections.
# A laser amplitude of a power of two 2^-k everywhere scales every field of the
# run by it and changes no mask, but for the rounding of subnormal |z|^2: an
# error of 2^-150 in |z|^2, which is exponentially distributed about 2^-122 here
# (6 % of it below 2^-126, in nearly every thread), is one of
# 2^-150 sqrt(N) / 2^-121 (2e-6 at 1024^2) in the root mean square of a field.
@pytest.mark.parametrize("ny,nx", [(64, 64), (256, 256), (1024, 1024), (600, 800), (480, 640)])
def test_subnormal_fields_give_the_same_mask(ny, nx):
    k = round((122 + np.log2(ny * nx)) / 2)  # |z|^2 about N 4^-k
    I = S.spot_target(76, ny, nx, 9, (0.5, 1.0))
    phi0 = S.random_phase(77, ny, nx)
    one = _laser_run(I, phi0, np.ones((ny, nx), np.float32), 1)
    tiny = _laser_run(I, phi0, np.full((ny, nx), 2.0 ** -k, np.float32), 1)
    assert one[3] == 0 and tiny[3] == 0
    assert aligned_rel_err(tiny[0], np.exp(1j * one[0].astype(np.float64))) <= 1e-5
    # the gaps: terms of some 4^-k, rounded to 2^-149 where they are subnormal
    np.testing.assert_allclose(tiny[1], one[1], rtol=1e-3)
    np.testing.assert_allclose(tiny[2], one[2], rtol=1e-3)


# Sides up to 4096 beside short ones: as long as the lines fit shared memory.
@pytest.mark.parametrize("ny,nx", [(100, 2048), (2048, 100), (320, 320), (50, 600)])
def test_general_long_sides_parity(ny, nx):
    I = S.spot_target(78, ny, nx, 6, (0.5, 1.0))
    phi0 = S.random_phase(79, ny, nx)
    ph, r, g, st = gpu_gs(I, phi0, 1)
    assert st == 0
    u, r0, g0 = O.gs_step(np.exp(1j * phi0.astype(np.float64)), O.target_amplitude(I))
    assert aligned_rel_err(ph, u) <= 1e-5
    assert abs(r[0] - r0) <= 1e-5 * r0 and abs(g[0] - g0) <= 1e-5 * g0
