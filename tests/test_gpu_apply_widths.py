"""The block preconditioner on periodic bands of every width, in both lane
layouts, against dense solves; failed blocks; the alignment of the buffer."""
import numpy as np
import pytest

from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# band widths 0 .. 20 at l_max = 70, dense polar rings
RADII = np.array([0.01, 0.03, 0.05, 0.07, 0.095, 0.12, 0.145, 0.17, 0.2, 0.23, 0.26, 0.29, 0.33, 0.38, 0.42])


def _solve(L, x):
    from scipy.linalg import solve_triangular
    z = solve_triangular(L, x, lower=True)
    return solve_triangular(L.T, z, lower=False)


@pytest.mark.parametrize("reps", [1, 12])  # 1065 blocks: one per warp; 12780: full warps
@pytest.mark.parametrize("aligned", [True, False])
def test_apply_every_width(reps, aligned):
    """y = L^-T L^-1 x block by block.  Two substitutions and their reference
    each have a relative error below (n eps) cond(L)^2; the blocks here have
    cond(L L^T) below about 1e3, so 1e-10 leaves two digits."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    if reps > 1 and not aligned:
        pytest.skip("one layout is enough for the unaligned buffer")
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
    buf = torch.zeros(nbytes // 8 + 1, dtype=torch.float64, device="cuda")
    blocks = S.sympix_sample_blocks(plan, torch.tensor(ninv).cuda(), precision="fp64", out=buf[:-1])
    # well conditioned: the diagonal of every block raised by its largest row sum
    host = blocks.cpu().numpy()
    for o in range(nops):
        for j in range(grid.nrings):
            off, n, w, fmt = plan.block_layout("pband", o, j)
            step, width = (w + 1, w + 1) if fmt == S.BLOCK_PBAND else (n + 1, n)
            rows = host[off:off + n * width].reshape(n, width)
            host[off:off + n * width:step] += 0.1 * np.max(np.abs(rows)) * (2 * min(w, n) + 1)
    buf[:-1].copy_(torch.tensor(host))
    info = S.sympix_factor_blocks(plan, blocks, precision="fp64")
    assert int((info != 0).sum()) == 0
    fail = info.clone()
    fail[7::grid.nrings] = 3  # a failed block of every operator passes x through
    x = torch.randn(nops, int(grid.npix), dtype=torch.float64, device="cuda")
    if not aligned:
        odd = torch.zeros_like(buf)
        odd[1:] = buf[:-1]
        blocks = odd[1:]
    y = S.sympix_apply(plan, blocks, fail, x).cpu().numpy()
    L0, X = blocks.cpu().numpy(), x.cpu().numpy()
    seen = set()
    for o in range(nops):
        if o >= len(RADII) and o % 11:
            continue
        for j in range(grid.nrings):
            _, n, w, fmt = plan.block_layout("pband", o, j)
            px = grid.ring_offset[j] + grid.ring_stride[j] * np.arange(n)
            if j == 7:
                assert np.array_equal(y[o, px], X[o, px])
                continue
            L = S.unpack_block(L0, plan, "pband", o, j, factored=True)
            ref = _solve(L, X[o, px])
            assert np.max(np.abs(y[o, px] - ref)) <= 1e-10 * np.max(np.abs(ref)), (o, j, n, w, fmt)
            seen.add((int(fmt), int(w)) if fmt == S.BLOCK_PBAND else (int(fmt), n > 32))
    widths = {w for f, w in seen if f == S.BLOCK_PBAND}
    assert {2, 4, 6, 8, 10, 12, 14, 16} <= widths and max(widths) > 16, sorted(widths)
    assert (S.BLOCK_DENSE, False) in seen and (S.BLOCK_DENSE, True) in seen
