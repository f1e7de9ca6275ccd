"""The block preconditioner reads no entry that the factored format leaves
undefined: band rows past the last full column, wrapped offsets of the first
rows, the strict upper corner of the border, gaps between blocks."""
import numpy as np
import pytest

from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# band widths 0 .. 20 at l_max = 70, dense polar rings
RADII = np.array([0.01, 0.03, 0.05, 0.07, 0.095, 0.12, 0.145, 0.17, 0.2, 0.23, 0.26, 0.29, 0.33, 0.38, 0.42])


def _defined(n, w):
    """Mask of the n (2w+1) values of a factored periodic-band block that hold L."""
    m = n - w
    i, d = np.arange(n)[:, None], np.arange(w + 1)[None, :]
    border = np.arange(n)[None, :] <= m + np.arange(w)[:, None]
    return np.concatenate([((i < m) & (d <= i)).reshape(-1), border.reshape(-1)])


@pytest.mark.parametrize("reps", [1, 12])  # one block per warp; full warps
@pytest.mark.parametrize("stage", ["sampled", "factored"])
@pytest.mark.parametrize("fill", [np.nan, np.inf])
def test_apply_reads_defined_entries_only(reps, stage, fill):
    """The buffer holds NaN or infinity wherever the sampled (the factored)
    format defines nothing; y = L^-T L^-1 x as in a buffer of zeros.  Blocks
    with cond(L L^T) below about 1e3: 1e-10 as in the test of every width."""
    import torch
    from scipy.linalg import solve_triangular
    from paper_1504_04653_gb300 import sympix as S
    lmax = 70
    radii = np.tile(RADII, reps)
    nops = len(radii)
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii)
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    ninv = np.stack([W.ninv_map(o, colat, 5.0 * (o % 4)) for o in range(nops)])
    bl = np.tile(W.gaussian_beam(lmax, 600.0), (nops, 1))
    S.sympix_kernel_table(plan, torch.tensor(bl).cuda(), torch.ones(nops, lmax + 1, dtype=torch.float64).cuda())
    nbytes, _ = plan.blocks_size("pband")
    blocks = torch.full((nbytes // 8,), fill, dtype=torch.float64, device="cuda")
    S.sympix_sample_blocks(plan, torch.tensor(ninv).cuda(), precision="fp64", out=blocks)
    host = blocks.cpu().numpy()
    layout = {(o, j): plan.block_layout("pband", o, j) for o in range(nops) for j in range(grid.nrings)}
    for off, n, w, fmt in layout.values():  # the diagonal raised by the largest row sum
        step, width = (w + 1, w + 1) if fmt == S.BLOCK_PBAND else (n + 1, n)
        rows = host[off:off + n * width].reshape(n, width)
        assert np.all(np.isfinite(rows))
        host[off:off + n * width:step] += 0.1 * np.max(np.abs(rows)) * (2 * min(w, n) + 1)
    blocks.copy_(torch.tensor(host))
    info = S.sympix_factor_blocks(plan, blocks, precision="fp64")
    assert int((info != 0).sum()) == 0
    host = blocks.cpu().numpy()
    if stage == "factored":
        keep = np.zeros(len(host), dtype=bool)
        for off, n, w, fmt in layout.values():
            keep[off:off + n * (2 * w + 1 if fmt == S.BLOCK_PBAND else n)] = (
                _defined(n, w) if fmt == S.BLOCK_PBAND else np.tri(n, dtype=bool).reshape(-1))
        host[~keep] = fill
        blocks.copy_(torch.tensor(host))
    x = torch.randn(nops, int(grid.npix), dtype=torch.float64, device="cuda")
    y, X = S.sympix_apply(plan, blocks, info, x).cpu().numpy(), x.cpu().numpy()
    for o in range(nops):
        if o >= len(RADII) and o % 11:
            continue
        for j in range(grid.nrings):
            off, n, w, fmt = layout[o, j]
            px = grid.ring_offset[j] + grid.ring_stride[j] * np.arange(n)
            L = S.unpack_block(host, plan, "pband", o, j, factored=True)
            assert np.all(np.isfinite(L)), (o, j, n, w, fmt)
            ref = solve_triangular(L.T, solve_triangular(L, X[o, px], lower=True), lower=False)
            assert np.max(np.abs(y[o, px] - ref)) <= 1e-10 * np.max(np.abs(ref)), (o, j, n, w, fmt)
