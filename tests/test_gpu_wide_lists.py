"""FP32 sampling of bands wider than 16: each of the plan's three work lists
(w of 17 .. 31, 32 .. 47, 48 .. 64) against the dense storage's kernel, which
sums the same terms in the same order: equal bit for bit."""
import numpy as np
import pytest

from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi,radii", [(17, 31, [0.17, 0.22, 0.27]), (32, 47, [0.3, 0.36, 0.42]),
                                         (48, 64, [0.46, 0.52, 0.58])])
def test_list_equals_dense_storage(lo, hi, radii):
    import torch
    from paper_1504_04653_gb300 import sympix as S
    lmax, nops = 150, len(radii)
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii)
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    ninv = torch.tensor(np.stack([W.ninv_map(20 + o, colat, 10.0) for o in range(nops)])).cuda()
    bl = torch.tensor(np.tile(W.gaussian_beam(lmax, 200.0), (nops, 1))).cuda()
    S.sympix_kernel_table(plan, bl, torch.tensor(np.tile(W.prior(lmax), (nops, 1))).cuda())
    band = S.sympix_sample_blocks(plan, ninv, precision="fp32", storage="pband").cpu().numpy()
    full = S.sympix_sample_blocks(plan, ninv, precision="fp32", storage="dense").cpu().numpy()
    widths = set()
    for o in range(nops):
        for j in range(grid.nrings):
            off, n, w, fmt = plan.block_layout("pband", o, j)
            if fmt != S.BLOCK_PBAND or not lo <= w <= hi:
                continue
            A = band[off:off + n * (w + 1)].reshape(n, w + 1)
            offd = plan.block_layout("dense", o, j)[0]
            D = full[offd:offd + n * n].reshape(n, n)
            q, d = np.arange(n)[:, None], np.arange(w + 1)[None, :]
            assert np.array_equal(A, D[q, (q - d) % n]), (o, j, n, w)
            widths.add(int(w))
    print(sorted(widths))
    assert len(widths) >= 4, sorted(widths)
