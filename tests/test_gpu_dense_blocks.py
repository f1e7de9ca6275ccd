"""Dense-format ring blocks (polar or fully coupled rings): sampling over row
tiles, and the factor of up to 32 rows inside the sliding-window launch."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lmax,radii", [(40, [0.9, 3.2]), (75, [0.25, 3.2])])
@pytest.mark.parametrize("storage", ["pband", "dense"])
def test_dense_sampling_matches_oracle(lmax, radii, storage):
    """Up to 160 pixels a ring: one to three tiles of 64 columns, arcs and whole
    rings; 1e-10 normwise, the tolerance of every FP64 block, and symmetric."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii)
    nops = len(radii)
    bl = np.tile(W.gaussian_beam(lmax, 400.0), (nops, 1))
    dl = np.tile(W.prior(lmax), (nops, 1))
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    ninv = np.stack([W.ninv_map(70 + o, colat, 15.0) for o in range(nops)])
    S.sympix_kernel_table(plan, torch.tensor(bl).cuda(), torch.tensor(dl).cuda())
    buf = S.sympix_sample_blocks(plan, torch.tensor(ninv).cuda(), precision="fp64", storage=storage).cpu().numpy()
    og, sizes = O.grid(lmax), set()
    for o in range(nops):
        r_s, _ = plan.radius(o)
        for j in list(range(0, grid.nrings, 5)) + [1, 2, grid.nrings // 2]:
            _, n, _, fmt = plan.block_layout("pband", o, j)
            if fmt != S.BLOCK_DENSE:
                continue
            M = S.unpack_block(buf, plan, storage, o, j)
            ref, _ = O.block(og, bl[o], dl[o], r_s, ninv[o], j)
            assert np.array_equal(M, M.T)
            assert np.max(np.abs(M - ref)) <= 1e-10 * np.max(np.abs(ref)), (o, j, n)
            sizes.add((n + 63) // 64)
    assert {1, 2} <= sizes


@pytest.mark.parametrize("fprec", ["fp64", "fp32x2"])
def test_small_dense_factor(fprec):
    """Blocks of 8 to 32 rows and just above: L against numpy's Cholesky with
    the backward error n eps of FP64 (times 8), the pivot of an indefinite
    block, the strict upper triangle untouched."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    lmax = 30
    grid = S.Grid(lmax)
    plan = S.Plan(grid, [3.2, 0.6])
    rng = np.random.default_rng(8)
    nbytes, _ = plan.blocks_size("pband")
    host = np.zeros(nbytes // 8)
    want, seen = {}, set()
    for o in range(2):
        for j in range(grid.nrings):
            off, n, w, fmt = plan.block_layout("pband", o, j)
            if fmt == S.BLOCK_DENSE:
                B = rng.standard_normal((n, n))
                M = B @ B.T + n * np.eye(n)
                bad = (j % 4 == 1) * (1 + (5 * j) % n)
                if bad:
                    M[bad - 1, bad - 1] = -1.0
                host[off:off + n * n] = M.reshape(-1)
                want[(o, j)] = (M, bad)
                seen.add(n)
            else:
                host[off:off + n * (w + 1)].reshape(n, w + 1)[:, 0] = 1.0
    blocks = torch.tensor(host).cuda()
    info = S.sympix_factor_blocks(plan, blocks, precision=fprec).cpu().numpy()
    got = blocks.cpu().numpy()
    for (o, j), (M, bad) in want.items():
        off, n, _, _ = plan.block_layout("pband", o, j)
        assert info[o * grid.nrings + j] == bad, (o, j, n)
        if bad:
            continue
        A = got[off:off + n * n].reshape(n, n)
        L = np.tril(A)
        assert np.array_equal(np.triu(A, 1), np.triu(M, 1))
        assert np.max(np.abs(L @ L.T - M)) <= 8 * n * 2.0 ** -53 * np.max(np.abs(M)), (o, j, n)
    assert min(seen) <= 12 and any(n > 32 for n in seen) and any(24 <= n <= 32 for n in seen), sorted(seen)


def test_table_of_several_radii():
    """The kernel values of several operators with their own radii equal those
    of plans with one operator, bit for bit, wherever they are coupled."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    lmax, radii = 60, [0.1, 0.45, 0.02, 0.3, 0.3, 0.07, 0.6, 0.15, 0.25, 0.01, 0.5]
    grid = S.Grid(lmax)
    bl = np.stack([W.gaussian_beam(lmax, 60.0 + 30 * o) for o in range(len(radii))])
    dl = np.stack([W.prior(lmax) * (1 + o) for o in range(len(radii))])
    many = S.Plan(grid, radii)
    S.sympix_kernel_table(many, torch.tensor(bl).cuda(), torch.tensor(dl).cuda())
    for o, r in enumerate(radii):
        one = S.Plan(grid, [r])
        S.sympix_kernel_table(one, torch.tensor(bl[o:o + 1]).cuda(), torch.tensor(dl[o:o + 1]).cuda())
        for j in (0, 7, 30, 44):
            m = one.support(0, j, 12)
            for rho in range(max(0, j - 12), min(grid.nrings, j + 13)):
                if m[rho - j + 12] < 0:
                    continue
                count = int(m[rho - j + 12]) // 2 + 1
                for a, b in zip(many.table(o, j, rho, count), one.table(0, j, rho, count)):
                    assert a is None and b is None or np.array_equal(a, b), (o, j, rho)
