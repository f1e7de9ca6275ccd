"""Plans of different band widths side by side: calls from two threads, and a
captured step replayed after another plan's calls (the shared-memory limit
belongs to a kernel, not to a launch)."""
import threading

import numpy as np
import pytest

from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _plan(S, lmax, radii):
    import torch
    nops = len(radii)
    grid = S.Grid(lmax)
    plan = S.Plan(grid, radii)
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    ninv = torch.tensor(np.stack([W.ninv_map(o, colat, 10.0) for o in range(nops)])).cuda()
    bl = torch.tensor(np.tile(W.gaussian_beam(lmax, 400.0), (nops, 1))).cuda()
    dl = torch.ones(nops, lmax + 1, dtype=torch.float64, device="cuda")
    S.sympix_kernel_table(plan, bl, dl)
    nbytes, _ = plan.blocks_size("pband")
    return grid, plan, bl, dl, ninv, torch.zeros(nbytes // 8, dtype=torch.float64, device="cuda")


def _widths(S, grid, plan):
    return {w for o in range(plan.nops) for j in range(grid.nrings)
            for _, _, w, fmt in [plan.block_layout("pband", o, j)] if fmt == S.BLOCK_PBAND}


@pytest.mark.parametrize("kind", ["sample", "factor", "apply"])
def test_two_threads(kind):
    """Each thread's calls succeed and give what they give alone.  (A launch met
    another plan's lower limit about once in some thousand calls.)"""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    # sample: different widths of 17 .. 31, one launch's; apply and factor: w <= 8
    # and w <= 16, full warps in both
    radii = {"sample": ([0.25] * 2, [0.38] * 2)}.get(kind, ([0.05, 0.08] * 12, [0.1, 0.2] * 12))
    sides = []
    for r in radii:
        grid, plan, bl, dl, ninv, blocks = _plan(S, 110, r)
        info = torch.zeros(plan.nblocks, dtype=torch.int32, device="cuda")
        x = torch.randn(plan.nops, int(grid.npix), dtype=torch.float64, device="cuda")
        y = torch.zeros_like(x)
        S.sympix_sample_blocks(plan, ninv, precision="fp64", out=blocks)
        if kind == "apply":
            S.sympix_factor_blocks(plan, blocks, precision="fp64", info=info)

        def call(plan=plan, ninv=ninv, blocks=blocks, info=info, x=x, y=y):
            if kind == "sample":
                return S.sympix_sample_blocks(plan, ninv, precision="fp32", out=blocks)
            if kind == "factor":
                S.sympix_sample_blocks(plan, ninv, precision="fp64", out=blocks)
                return S.sympix_factor_blocks(plan, blocks, precision="fp64", info=info)
            return S.sympix_apply(plan, blocks, info, x, out=y)

        sides.append((call, _widths(S, grid, plan)))
    top = [max(w for w in s[1] if w <= 31) for s in sides]
    assert top[0] < top[1] and (kind != "sample" or top[0] > 16), [sorted(s[1]) for s in sides]
    refs = [c().clone() for c, _ in sides]
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(2)

    def work(call):
        start.wait()
        try:
            for _ in range(4000):
                call()
        except Exception as e:  # reported below, in the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c, _ in sides]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]
    for (c, _), ref in zip(sides, refs):
        assert torch.equal(c().nan_to_num(), ref.nan_to_num())


def test_captured_step_beside_another_plan():
    """A step captured on a plan with bands of about w = 28, replayed after a plan
    of narrower bands has sampled."""
    import torch
    from paper_1504_04653_gb300 import sympix as S
    _, plan, bl, dl, ninv, blocks = _plan(S, 110, [0.38, 0.3])
    info = torch.zeros(plan.nblocks, dtype=torch.int32, device="cuda")
    step = S.Step(plan, bl, dl, ninv, blocks, info, "pband", "fp32", "fp32")
    step.launch()
    torch.cuda.synchronize()
    ref = blocks.clone()
    _, other, _, _, ninv2, out2 = _plan(S, 110, [0.25])
    S.sympix_sample_blocks(other, ninv2, precision="fp32", out=out2)
    blocks.zero_()
    step.launch()
    torch.cuda.synchronize()
    assert torch.equal(blocks.nan_to_num(), ref.nan_to_num())
