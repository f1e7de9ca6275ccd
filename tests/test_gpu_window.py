"""The sliding-window factor (FP64 and split FP32, w <= 12): every width in both
lane layouts against numpy's Cholesky, and scaling by powers of four."""
import numpy as np
import pytest

from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# band widths 0 .. 12 at l_max = 60
RADII = np.array([0.01, 0.03, 0.055, 0.08, 0.11, 0.14, 0.17, 0.2, 0.235, 0.27, 0.3, 0.33])


def _sampled(S, reps, lmax=60):
    import torch
    radii = np.tile(RADII, reps)
    nops = len(radii)
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii)
    wl = W.Workload("widths", lmax, [600.0] * nops, [5.0 * (o % 4) for o in range(nops)], list(range(nops)))
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    # a diagonal prior keeps every block definite whatever the radius cuts off
    dl = np.ones((nops, lmax + 1))
    S.sympix_kernel_table(plan, torch.tensor(wl.beams()).cuda(), torch.tensor(dl).cuda())
    return grid, plan, S.sympix_sample_blocks(plan, torch.tensor(wl.ninv(colat)).cuda(), precision="fp64")


@pytest.mark.parametrize("fprec", ["fp64", "fp32x2"])
@pytest.mark.parametrize("reps", [1, 3])  # one block per warp; with the 2196 blocks of 3 as many as fit
def test_every_width_matches_cholesky(fprec, reps):
    """Backward error of Cholesky: |L L^T - M| <= (2w + 2) eps |M| row by row;
    eps 2^-53 in FP64 and about 2^-44 in split FP32, and a factor of 8 for
    products and sums rounded separately.  The pivot verdict is numpy's."""
    from paper_1504_04653_gb300 import sympix as S
    grid, plan, blocks = _sampled(S, reps)
    M0 = blocks.cpu().numpy()
    info = S.sympix_factor_blocks(plan, blocks, precision=fprec).cpu().numpy()
    L0 = blocks.cpu().numpy()
    eps = 2.0 ** -53 if fprec == "fp64" else 2.0 ** -44
    seen, good = set(), 0
    for o in range(plan.nops):
        for j in range(grid.nrings):
            _, n, w, fmt = plan.block_layout("pband", o, j)
            if fmt != S.BLOCK_PBAND or w > 12 or (o >= len(RADII) and (o + j) % 5):
                continue
            M = S.unpack_block(M0, plan, "pband", o, j)
            ev = np.linalg.eigvalsh(M)
            if abs(ev[0]) < 1e-9 * ev[-1]:
                continue  # either verdict is right
            assert (info[o * grid.nrings + j] == 0) == (ev[0] > 0), (o, j, n, w)
            if ev[0] > 0:
                L = S.unpack_block(L0, plan, "pband", o, j, factored=True)
                assert np.max(np.abs(L @ L.T - M)) <= 8 * (2 * w + 2) * eps * np.max(np.abs(M)), (o, j, n, w)
                seen.add(int(w))
                good += 1
    assert good > 100 and {2, 4, 6, 8} <= seen and max(seen) >= 9, sorted(seen)


@pytest.mark.parametrize("power", [-1000, 960, -1060])
def test_scaled_blocks(power):
    """Blocks scaled by 2^power have factors scaled by 2^(power / 2), bit for
    bit while the blocks and their reciprocals are normal numbers; scaled
    into the subnormals they still factor, to the precision that is left."""
    from paper_1504_04653_gb300 import sympix as S
    grid, plan, blocks = _sampled(S, 1)
    # split the scaling: 2^power itself may not be a normal number
    scaled = blocks * 2.0 ** (power // 2) * 2.0 ** (power - power // 2)
    ia = S.sympix_factor_blocks(plan, blocks).cpu().numpy()
    ib = S.sympix_factor_blocks(plan, scaled).cpu().numpy()
    a, b = blocks.cpu().numpy(), scaled.cpu().numpy()
    checked = 0
    for j in range(0, grid.nrings, 3):
        for o in range(plan.nops):
            _, n, w, fmt = plan.block_layout("pband", o, j)
            if fmt != S.BLOCK_PBAND or w > 12 or ia[o * grid.nrings + j] != 0:
                continue
            La = S.unpack_block(a, plan, "pband", o, j, factored=True) * 2.0 ** (power // 2)
            Lb = S.unpack_block(b, plan, "pband", o, j, factored=True)
            if power > -1060:
                assert ib[o * grid.nrings + j] == 0
                # entries whose products fall below the normal range may differ by what is lost there
                assert np.max(np.abs(La - Lb)) <= 1e-15 * np.max(np.abs(La)), (o, j)
            elif ib[o * grid.nrings + j] == 0:
                assert np.all(np.isfinite(Lb)) and np.max(np.abs(La - Lb)) <= 1e-2 * np.max(np.abs(La)), (o, j)
            checked += 1
    assert checked > 50
