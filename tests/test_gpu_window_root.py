"""The root and the reciprocal that the sliding-window factor and the block
preconditioner apply form from an FP32 estimate, seen through diagonal blocks
(w = 0): L = sqrt(M) and y = x / L^2, over exponents and significands."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _diagonal_plan(S):
    grid = S.Grid(60)
    plan = S.Plan(grid, [0.005, 0.005])
    spans = [plan.block_layout("pband", o, j) for o in range(2) for j in range(grid.nrings)]
    assert all(fmt == S.BLOCK_PBAND and w == 0 for _, _, w, fmt in spans)
    at = np.concatenate([np.arange(off, off + n) for off, n, _, _ in spans])
    return grid, plan, at


def _values(count, lo, hi):
    """Values of every exponent lo .. hi - 1: random significands, and those at
    both ends of the binade."""
    rng = np.random.default_rng(5)
    f = 1.0 + rng.random(count)
    f[::7], f[3::7], f[5::14] = 1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -52
    return np.ldexp(np.minimum(f, 2.0 - 2.0 ** -52), lo + np.arange(count) % (hi - lo))


def _factor(S, precision, lo, hi):
    import torch
    grid, plan, at = _diagonal_plan(S)
    nbytes, _ = plan.blocks_size("pband")
    host = np.zeros(nbytes // 8)
    host[at] = d = _values(len(at), lo, hi)
    blocks = torch.tensor(host).cuda()
    info = S.sympix_factor_blocks(plan, blocks, precision=precision)
    assert int((info != 0).sum()) == 0
    return blocks.cpu().numpy()[at], d


def test_root_fp64():
    """y (1 + e/2 + 3 e^2/8): half an ulp in the residual e, one rounding of the
    sum, one of d y: within 2.5 x 2^-53, 3 x 2^-53 allowed; all exponents."""
    from paper_1504_04653_gb300 import sympix as S
    L, d = _factor(S, "fp64", -1022, 1024)
    assert np.max(np.abs(L / np.sqrt(d) - 1.0)) <= 3 * 2.0 ** -53 + 2.0 ** -53


@pytest.mark.parametrize("lo,hi", [(-64, 64), (64, 127)])
def test_root_split_fp32(lo, hi):
    """Split FP32: products and sums of about 2^-47 each, within 2^-45 together.
    Their roundings go either way, so over thousands of values they leave
    nothing of 2^-49 in the mean, which a series cut after its first term
    (3 r^2 / 8 with r of about 2^-23) does."""
    from paper_1504_04653_gb300 import sympix as S
    L, d = _factor(S, "fp32x2", lo, hi)
    err = L / np.sqrt(d) - 1.0
    print(f"{lo} .. {hi}: {len(err)} values, largest {np.max(np.abs(err)):.3g}, mean {np.mean(err):.3g}")
    assert np.max(np.abs(err)) <= 2.0 ** -45
    assert abs(np.mean(err)) <= 2.0 ** -49


def test_reciprocal_fp64():
    """1/L within 2 x 2^-53, squared and times x with two roundings: 6 x 2^-53."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    grid, plan, at = _diagonal_plan(S)
    nbytes, _ = plan.blocks_size("pband")
    host = np.zeros(nbytes // 8)
    host[at] = _values(len(at), -500, 500)
    info = torch.zeros(plan.nblocks, dtype=torch.int32, device="cuda")
    x = np.random.default_rng(6).standard_normal((2, int(grid.npix)))
    y = S.sympix_apply(plan, torch.tensor(host).cuda(), info, torch.tensor(x).cuda()).cpu().numpy()
    for o in range(2):
        for j in range(grid.nrings):
            off, n, _, _ = plan.block_layout("pband", o, j)
            px = grid.ring_offset[j] + grid.ring_stride[j] * np.arange(n)
            ref = x[o, px] / host[off:off + n] / host[off:off + n]
            assert np.max(np.abs(y[o, px] / ref - 1.0)) <= 8 * 2.0 ** -53, (o, j)
