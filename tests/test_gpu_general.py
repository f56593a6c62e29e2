"""Grids whose sides are not powers of two (the 800 x 600 SLM of Sec. V and
other 5-smooth sides up to 1536) against the FP64 oracle, with the
tolerances of tests/test_gpu_parity.py: one step <= 1e-5, r and g <= 1e-3,
the final residual within 0.1%, the chain to a slack of 1e-6."""

import numpy as np
import pytest

import oracle.gs_oracle as O
from paper_1302_0120_gb300 import synthetic as S
from tests.gpu_util import aligned_rel_err, GROUPING_RTOL
from tests.test_gpu_parity import check_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize(
    "ny,nx,iters,nspots",
    [
        (600, 800, 25, 50),   # the paper's SLM and iteration count (register-resident kernel)
        (800, 600, 10, 30),   # the other sides of the register-resident kernel
        (800, 800, 8, 30),
        (600, 600, 8, 30),
        (768, 1024, 10, 30),  # the XGA SLM (1024 x 768), and 768 x 1024
        (1024, 768, 8, 30),
        (768, 768, 6, 20),
        (1024, 600, 6, 20),
        (160, 96, 20, 10),
        (36, 75, 15, 4),      # 75 columns: a ragged last group of 3
        (512, 800, 10, 30),   # one side a power of two
        (1536, 45, 6, 10),    # the largest side
        (45, 1536, 6, 10),
        (243, 250, 8, 20),    # radices 3 and 5 only
        (8, 8, 6, 1),         # small sides (below 32) on the general kernel
        (16, 16, 10, 2),
        (16, 64, 8, 2),
        (64, 8, 8, 2),
        (12, 10, 5, 1),
        (40, 48, 130, 3),     # two launches (128 iterations each at most)
    ],
)
def test_parity(ny, nx, iters, nspots):
    if min(ny, nx) < 10:  # no spot fits 7 px away from DC: a random positive target
        I = np.random.default_rng(ny + nx).random((ny, nx)).astype(np.float32)
    else:
        I = S.spot_target(ny + nx, ny, nx, nspots, (0.5, 1.0))
    phi0 = S.random_phase(ny + nx, ny, nx)
    check_run(I, phi0, iters, one_step_at=(0, iters - 1))


@pytest.mark.parametrize("grid", [1, 7, 200])
def test_parity_grid_shares(grid):
    """Ragged shares of rows and column groups over the blocks."""
    I = S.spot_target(3, 90, 120, 12, (0.5, 1.0))
    phi0 = S.random_phase(3, 90, 120)
    check_run(I, phi0, 6, grid=grid, one_step_at=(0,))


@pytest.mark.parametrize("ny,nx,grid", [(600, 800, 1), (600, 800, 7), (600, 800, 151), (768, 1024, 7)])
def test_register_kernel_grid_shares(ny, nx, grid):
    """The register-resident kernel with ragged shares of rows and column
    blocks over the blocks, several rounds per block."""
    I = S.spot_target(5, ny, nx, 30, (0.5, 1.0))
    phi0 = S.random_phase(5, ny, nx)
    check_run(I, phi0, 4, grid=grid, one_step_at=(0, 3))


def test_800x600_paper_variants():
    """The 800 x 600 experiment of Sec. V with the start P_S(F^{-1} m) and a
    Gaussian laser amplitude on the SLM."""
    import torch

    from paper_1302_0120_gb300 import GerchbergSaxton, build_lib

    build_lib.build()
    ny, nx, iters = 600, 800, 25
    I = S.spot_target(11, ny, nx, 50, (0.5, 1.0))
    p = S.laser_amplitude(ny, nx)
    with GerchbergSaxton(nx, ny, init_from_target=True) as gs:
        pt = torch.from_numpy(p).cuda()
        gs.set_slm_amplitude(pt)
        ph, r, g = gs.run(torch.from_numpy(I).cuda(), None, iters)
        st = gs.status()
        ph, r, g = ph.cpu().numpy(), r.cpu().numpy(), g.cpu().numpy()
    assert st == 0
    ref = O.gs_run(I, None, iters, p=p, init="target")
    # the conjugate-symmetric start is unstable under rounding (see
    # tests/test_gpu_variants.py): trajectories are compared over two steps
    assert np.max(np.abs(r[:2] - ref["r"][:2]) / ref["r"][:2]) <= 1e-3
    assert np.all(r[:-1] - g >= -1e-6) and np.all(g - r[1:] >= -1e-6)
    # one step from the GPU's own iterate
    with GerchbergSaxton(nx, ny) as gs:
        gs.set_slm_amplitude(pt)
        ph1, _, _ = gs.run(torch.from_numpy(I).cuda(), torch.from_numpy(ph).cuda(), 1)
        assert gs.status() == 0
        ph1 = ph1.cpu().numpy()
    m = O.target_amplitude(I, energy=float(np.sum(p.astype(np.float64) ** 2)))
    u1, _, _ = O.gs_step(p.astype(np.float64) * np.exp(1j * ph.astype(np.float64)), m, p.astype(np.float64))
    assert aligned_rel_err(ph1, u1 / np.abs(u1)) <= 1e-5


def test_batch_matches_single_runs():
    import torch

    from paper_1302_0120_gb300 import GerchbergSaxton, build_lib
    from tests.gpu_util import gpu_gs

    build_lib.build()
    ny, nx, nb, iters = 600, 800, 3, 5
    masks = [(S.spot_target(20 + k, ny, nx, 30, (0.5, 1.0)), S.random_phase(20 + k, ny, nx)) for k in range(nb)]
    with GerchbergSaxton(nx, ny, max_batch=nb) as gs:
        ph, r, g = gs.run_batched(torch.from_numpy(np.stack([m[0] for m in masks])).cuda(),
                                  torch.from_numpy(np.stack([m[1] for m in masks])).cuda(), iters)
        assert gs.status() == 0
        ph, r = ph.cpu().numpy(), r.cpu().numpy()
    for k, (I, phi0) in enumerate(masks):
        ph1, r1, _, st = gpu_gs(I, phi0, iters)
        assert st == 0 and np.array_equal(ph[k], ph1) and np.allclose(r[k], r1, rtol=GROUPING_RTOL, atol=0)


def test_loss_rejects_general_grids():
    import torch

    from paper_1302_0120_gb300 import GS_EINVAL
    from paper_1302_0120_gb300 import _binding as B
    from paper_1302_0120_gb300 import build_lib

    build_lib.build()
    h = B.gs_create(800, 800)
    try:
        x = torch.zeros(800, 800, device="cuda")
        out = torch.zeros(2, dtype=torch.float64, device="cuda")
        assert B.gs_loss_grad(h, x.data_ptr(), x.data_ptr(), out.data_ptr(), 0) == GS_EINVAL
        assert B.gs_physical_error(h, x.data_ptr(), x.data_ptr(), out.data_ptr()) == GS_EINVAL
    finally:
        B.gs_destroy(h)


@pytest.mark.parametrize("ny,nx", [(480, 640), (90, 120), (9, 1536)])
def test_fixed_grids_of_several_blocks_per_sm(ny, nx):
    """gs_set_grid is clamped to what the device keeps resident, which on these
    sides is more than one block of the general kernel per SM; the masks do not
    depend on it."""
    import torch

    from paper_1302_0120_gb300 import GerchbergSaxton, build_lib
    from paper_1302_0120_gb300 import _binding as B

    build_lib.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    I = torch.from_numpy(np.random.default_rng(5).random((ny, nx), dtype=np.float32)).cuda()
    P = torch.from_numpy(S.random_phase(6, ny, nx)).cuda()
    with GerchbergSaxton(nx, ny) as gs:
        ref, _, _ = gs.run(I, P, 4)
        for ctas in (sms - 1, sms + 20, 100000):
            gs.set_grid(ctas)
            assert B.gs_set_trace(gs.handle, True) == 0
            ph, _, _ = gs.run(I, P, 4)
            assert gs.status() == 0
            assert torch.equal(ph, ref)
            assert B.gs_get_trace(gs.handle).shape[1] == gs.grid
            assert gs.grid == ctas or (ctas == 100000 and gs.grid > sms), gs.grid
        assert B.gs_check_workspace(gs.handle) == B.GS_OK


@pytest.mark.parametrize("masks,ny,nx,laser", [(2, 16, 512, False), (4, 9, 1536, True), (16, 24, 1024, False),
                                               (12, 40, 1200, True), (5, 8, 1500, False), (3, 40, 1536, False)])
def test_batches_of_short_columns(masks, ny, nx, laser):
    """Batches of long rows and short columns may take several small blocks per
    SM: every mask of the batch equals its single run bit for bit, and the launch
    has the grid that is reported."""
    import torch

    from paper_1302_0120_gb300 import GerchbergSaxton, build_lib
    from paper_1302_0120_gb300 import _binding as B

    build_lib.build()
    rng = np.random.default_rng(nx + ny)
    I = torch.from_numpy(rng.random((masks, ny, nx), dtype=np.float32)).cuda()
    P = torch.from_numpy((2 * np.pi * rng.random((masks, ny, nx))).astype(np.float32)).cuda()
    p = torch.from_numpy(S.laser_amplitude(ny, nx)).cuda() if laser else None
    with GerchbergSaxton(nx, ny, max_batch=masks) as gs:
        gs.set_slm_amplitude(p)
        assert B.gs_set_trace(gs.handle, True) == 0
        ph, r, g = gs.run_batched(I, P, 4)
        assert gs.status() == 0 and B.gs_check_workspace(gs.handle) == B.GS_OK
        assert B.gs_get_trace(gs.handle).shape[1] == gs.grid
        for k in range(masks):
            ph1, r1, g1 = gs.run(I[k], P[k], 4)
            assert gs.status() == 0
            assert torch.equal(ph[k], ph1)
            np.testing.assert_allclose(r[k].cpu(), r1.cpu(), rtol=GROUPING_RTOL, atol=0)
            np.testing.assert_allclose(g[k].cpu(), g1.cpu(), rtol=GROUPING_RTOL, atol=0)
