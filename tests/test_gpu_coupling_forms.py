"""Blocks between rings over the forms the arc kernel and the general kernel
divide between them: narrow to full support, several column tiles, arcs longer
than one staged chunk, ring ranges, operators of different radii."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax,radii,delta,ring0,ring1", [
    (40, [0.02, 0.2], 1, 0, 41),        # from no coupled pair to a few columns
    (97, [0.5, 0.12], 3, 10, 60),       # more than 32 stored columns
    (150, [0.9], 1, 60, 70),            # arcs of more than 64 pixels, three and more column tiles
    (33, [1.6, 3.2], 2, 0, 34),         # around the ring, the whole sphere
])
def test_forms_match_oracle(lmax, radii, delta, ring0, ring1):
    """Sums of n products of FP64 values: 1e-10 normwise, the tolerance of
    every FP64 block (the kernel values dominate the error)."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii, ring0, ring1)
    nops = len(radii)
    bl = np.tile(W.gaussian_beam(lmax, 300.0), (nops, 1))
    dl = np.tile(W.prior(lmax), (nops, 1))
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    ninv = np.stack([W.ninv_map(90 + o, colat, 10.0) for o in range(nops)])
    nbytes, _ = plan.coupling_size(delta)
    S.sympix_kernel_table(plan, torch.tensor(bl).cuda(), torch.tensor(dl).cuda())
    out = torch.full((nbytes // 8,), np.nan, dtype=torch.float64, device="cuda")  # every entry is written
    buf = S.sympix_sample_coupling(plan, torch.tensor(ninv).cuda(), delta, out=out).cpu().numpy()
    assert np.all(np.isfinite(buf))
    og = O.grid(lmax)
    for o in range(nops):
        r_s, _ = plan.radius(o)
        rings = range(ring0, ring1 - delta)
        for j in list(rings)[:: max(1, len(rings) // 12)]:
            M = S.unpack_coupling(buf, plan, delta, o, j)
            ref, _ = O.block_pair(og, bl[o], dl[o], r_s, ninv[o], j, j + delta)
            assert np.max(np.abs(M - ref)) <= 1e-10 * max(np.max(np.abs(ref)), 1e-300), (o, j)
