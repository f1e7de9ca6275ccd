"""FP32 sampling of bands wider than 16 (register-tiled) against the dense
storage's kernel, which sums the same terms in the same order one element at a
time: equal bit for bit."""
import numpy as np
import pytest

from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax,radii,special", [
    (150, [0.08, 0.11, 0.15, 0.2], False),         # w up to 24, remainders of the 64-column tiles
    (150, [0.26, 0.33, 0.45, 0.55], False),        # up to w 64 and spans beyond the staging
    (61, [0.2, 0.4], False),
    (150, [0.1, 0.16, 0.3], True),                 # N^-1 with infinities, NaN, huge and tiny values
])
def test_equals_dense_storage(lmax, radii, special):
    import torch
    from paper_1504_04653_gb300 import sympix as S
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii)
    nops = len(radii)
    bl = np.tile(W.gaussian_beam(lmax, 200.0), (nops, 1))
    dl = np.tile(W.prior(lmax), (nops, 1))
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    ninv = np.stack([W.ninv_map(50 + o, colat, 10.0) for o in range(nops)])
    if special:
        p = np.random.default_rng(3).choice(int(grid.npix), 60, replace=False)
        for i, v in enumerate((np.inf, -np.inf, np.nan, 3e38, -1e30, 1e-44)):
            ninv[:, p[i::6]] = v
    S.sympix_kernel_table(plan, torch.tensor(bl).cuda(), torch.tensor(dl).cuda())
    nv = torch.tensor(ninv).cuda()
    band = S.sympix_sample_blocks(plan, nv, precision="fp32", storage="pband").cpu().numpy()
    full = S.sympix_sample_blocks(plan, nv, precision="fp32", storage="dense").cpu().numpy()
    seen = set()
    for o in range(nops):
        for j in range(grid.nrings):
            off, n, w, fmt = plan.block_layout("pband", o, j)
            if fmt != S.BLOCK_PBAND or w <= 8:
                continue
            A = band[off:off + n * (w + 1)].reshape(n, w + 1)
            offd = plan.block_layout("dense", o, j)[0]
            D = full[offd:offd + n * n].reshape(n, n)
            q = np.arange(n)
            for d in range(w + 1):
                assert np.array_equal(A[:, d], D[q, (q - d) % n], equal_nan=True), (o, j, n, w, d)
            seen.add((w - 1) // 16)
    assert len(seen) >= 1
