"""The sliding-window factor (w <= 12) over the range of its arithmetic: blocks
scaled as a whole and row by row, against the backward error of Cholesky."""
import numpy as np
import pytest

from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# band widths 0 .. 12 at l_max = 60
RADII = np.array([0.01, 0.03, 0.055, 0.08, 0.11, 0.14, 0.17, 0.2, 0.235, 0.27, 0.3, 0.33])


def _blocks(S, reps):
    import torch
    lmax, radii = 60, np.tile(RADII, reps)
    nops = len(radii)
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii)
    wl = W.Workload("widths", lmax, [600.0] * nops, [5.0 * (o % 4) for o in range(nops)], list(range(nops)))
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    S.sympix_kernel_table(plan, torch.tensor(wl.beams()).cuda(),
                          torch.ones(nops, lmax + 1, dtype=torch.float64).cuda())
    blocks = S.sympix_sample_blocks(plan, torch.tensor(wl.ninv(colat)).cuda(), precision="fp64")
    return grid, plan, blocks.cpu().numpy()


@pytest.mark.parametrize("reps", [1, 3])  # one block per warp; as many as fit
@pytest.mark.parametrize("rows", [False, True])
@pytest.mark.parametrize("top", [-96, -66, -62, 62, 66, 100, 112, 120, 125, 126])
def test_scaled_blocks(reps, rows, top):
    """Every block's largest diagonal entry brought to 2^(top-1) .. 2^(top+1) by
    a power of four; with `rows` each row and column then by its own power of
    two down to 2^-24 (the diagonal by 2^-48; 2^-12 for small values, so that
    all stay normal numbers).  Split FP32 keeps about 44
    bits, and of its input nothing of a low word below 2^-98 (a value below
    2^-74 is its high word) nor of a value below 2^-126:
    |L L^T - M|_ij <= 8 (2w + 2) (2^-44 s_ij + min(2^-24 s_ij, 2^-98) + 2^-126),
    s_ij = sqrt(M_ii M_jj)."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    grid, plan, host = _blocks(S, reps)
    rng = np.random.default_rng(top + 200)
    picked = {}
    for o in range(plan.nops):
        for j in range(grid.nrings):
            off, n, w, fmt = plan.block_layout("pband", o, j)
            if fmt != S.BLOCK_PBAND or w > 12:
                continue
            rowsview = host[off:off + n * (w + 1)].reshape(n, w + 1)
            big = int(np.floor(np.log2(rowsview[:, 0].max())))
            rowsview *= 2.0 ** (2 * ((top - big) // 2))
            # definite by a margin, so that the verdict is not in question
            rowsview[:, 0] *= 1.0 if w == 0 else 1.001
            if rows:
                k = rng.integers(-24 if top > 0 else -12, 1, n)
                q, d = np.arange(n)[:, None], np.arange(w + 1)[None, :]
                rowsview *= 2.0 ** (k[q] + k[(q - d) % n]).astype(float)
            if not (o >= len(RADII) and (o + j) % 5) and j % 2 == 0:
                picked[o, j] = (n, w)
    blocks = torch.tensor(host).cuda()
    info = S.sympix_factor_blocks(plan, blocks, precision="fp32x2").cpu().numpy()
    got, widths, worst = blocks.cpu().numpy(), set(), 0.0
    for (o, j), (n, w) in picked.items():
        M = S.unpack_block(host, plan, "pband", o, j)
        diag = np.sqrt(np.diag(M))
        if np.linalg.eigvalsh(M / diag / diag[:, None])[0] < 1e-3:
            continue  # either verdict may be right once low words are lost
        assert info[o * grid.nrings + j] == 0, (o, j, n, w, int(info[o * grid.nrings + j]))
        L = S.unpack_block(got, plan, "pband", o, j, factored=True)
        s = diag * diag[:, None]
        bound = 8 * (2 * w + 2) * (2.0 ** -44 * s + np.minimum(2.0 ** -24 * s, 2.0 ** -98) + 2.0 ** -126)
        err = np.max(np.abs(L @ L.T - M) / bound)
        worst = max(worst, err)
        assert err <= 1.0, (o, j, n, w, err)
        widths.add(int(w))
    print(f"top {top} rows {rows}: worst error / bound {worst:.3g}")
    assert len(widths) >= 6 and {2, 4, 8} <= widths and max(widths) >= 10, sorted(widths)


@pytest.mark.parametrize("reps", [1, 3])
@pytest.mark.parametrize("top", [-1040, -1000, 0, 1000, 1022])
def test_scaled_blocks_fp64(reps, top):
    """The same in FP64, down into the subnormal numbers, which lose what lies
    below 2^-1074: |L L^T - M|_ij <= 8 (2w + 2) (2^-53 s_ij + 2^-1074).  Every
    well-conditioned block factors, in every width from 0 to 12."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    grid, plan, host = _blocks(S, reps)
    picked = {}
    for o in range(plan.nops):
        for j in range(grid.nrings):
            off, n, w, fmt = plan.block_layout("pband", o, j)
            if fmt != S.BLOCK_PBAND or w > 12:
                continue
            rowsview = host[off:off + n * (w + 1)].reshape(n, w + 1)
            big = int(np.floor(np.log2(rowsview[:, 0].max())))
            half = (top - big) // 2
            rowsview *= 2.0 ** half
            rowsview *= 2.0 ** half
            if not (o >= len(RADII) and (o + j) % 5) and j % 2 == 0:
                picked[o, j] = (n, w)
    blocks = torch.tensor(host).cuda()
    info = S.sympix_factor_blocks(plan, blocks, precision="fp64").cpu().numpy()
    got, widths = blocks.cpu().numpy(), set()
    up = 2.0 ** (-(top // 2))  # both sides back to where numpy's products are normal numbers
    for (o, j), (n, w) in picked.items():
        M = S.unpack_block(host, plan, "pband", o, j) * up * up
        diag = np.sqrt(np.diag(M))
        if np.linalg.eigvalsh(M / diag / diag[:, None])[0] < 1e-3:
            continue
        assert info[o * grid.nrings + j] == 0, (o, j, n, w, int(info[o * grid.nrings + j]))
        L = S.unpack_block(got, plan, "pband", o, j, factored=True) * up
        bound = 8 * (2 * w + 2) * (2.0 ** -53 * diag * diag[:, None] + 2.0 ** -1074 * up * up)
        assert np.max(np.abs(L @ L.T - M) / bound) <= 1.0, (o, j, n, w, np.max(np.abs(L @ L.T - M) / bound))
        widths.add(int(w))
    print(sorted(widths))
    assert {0, 2, 4, 6, 8, 10, 12} <= widths, sorted(widths)
