"""The w <= 12 factor kernel as a plan option in FP64 and split FP32: the number
a plan reports selects the kernel it runs, and pivot verdicts of the sliding
window (2, the default) and the chunked border (3)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1504_04653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _sampled(S, name, ninv_of=lambda grid, ninv: ninv):
    import torch
    wl = W.WORKLOADS[name]
    grid = S.Grid(wl.lmax)
    plan = S.Plan(grid, wl.radii())
    colat = W.pixel_colatitude(grid.theta, grid.nring, grid.ring_offset, grid.ring_stride, grid.npix)
    ninv = ninv_of(grid, wl.ninv(colat))
    S.sympix_kernel_table(plan, torch.tensor(wl.beams()).cuda(), torch.tensor(wl.priors()).cuda())
    return wl, grid, plan, ninv, S.sympix_sample_blocks(plan, torch.tensor(ninv).cuda(), precision="fp64")


@pytest.mark.parametrize("fprec,window,chunked", [("fp64", "k_f64_window", "k_f64_band_pass"),
                                                  ("fp32x2", "k_df_window", "k_df_band_pass")])
def test_reported_number_selects_the_kernel(fprec, window, chunked):
    import torch
    from paper_1504_04653_gb300 import sympix as S
    wl, grid, plan, ninv, blocks = _sampled(S, "lmax64")
    plan.set_trace(True)

    def factor():
        plan.trace_read()
        b = blocks.clone()
        S.sympix_factor_blocks(plan, b, precision=fprec)
        return [n for n, _ in plan.trace_read()], b.cpu().numpy()

    plan.set_narrow_factor(-1)
    names, ref = factor()
    assert window in names
    plan.set_narrow_factor(plan.narrow_kernels()[fprec])  # what a program stored
    again, got = factor()
    assert again == names and np.array_equal(got, ref)
    for k in range(4):
        plan.set_narrow_factor(k)
        assert plan.narrow_kernels()[fprec] == k
        names = factor()[0]
        assert (window in names) == (k == 2) and (chunked in names) == (k == 3), (k, names)
    info = torch.empty(plan.nblocks, dtype=torch.int32, device="cuda")
    bl, dl = torch.tensor(wl.beams()).cuda(), torch.tensor(wl.priors()).cuda()
    plan.autotune(bl, dl, torch.tensor(ninv).cuda(), blocks.clone(), info, sample_precision="fp64",
                  factor_precision=fprec)
    k = plan.narrow_kernels()[fprec]
    names = factor()[0]
    assert (window in names) == (k == 2) and (chunked in names) == (k == 3), (k, names)


@pytest.mark.parametrize("fprec", ["fp64", "fp32x2"])
@pytest.mark.parametrize("narrow", [-1, 3])
@pytest.mark.parametrize("where", ["third", "near the end"])
def test_indefinite_pivot(fprec, narrow, where):
    """info is the oracle's pivot index: negative inverse noise over a third of
    the sphere (pivots anywhere), and single pixels near a ring's end, which
    leave the band's minors positive (pivots in the corner and the last rows)."""
    from paper_1504_04653_gb300 import sympix as S

    def negative(grid, ninv):
        if where == "third":
            ninv[0, : grid.npix // 3] *= -40.0
        else:
            for j, back in ((40, 3), (20, 9), (55, 1)):
                n = int(grid.nring[j])
                ninv[0, int(grid.ring_offset[j]) + (n - back) * int(grid.ring_stride[j])] *= -3.0
        return ninv

    wl, grid, plan, ninv, blocks = _sampled(S, "lmax64", negative)
    plan.set_narrow_factor(narrow)
    info = S.sympix_factor_blocks(plan, blocks, precision=fprec).cpu().numpy()
    og = O.grid(64)
    corner = band = 0
    for j in range(grid.nrings):
        ref, _ = O.block(og, wl.beams()[0], wl.priors()[0], wl.radii()[0], ninv[0], j)
        _, want = O.cholesky(ref)
        assert info[j] == want, (j, int(info[j]), want)
        _, n, w, fmt = plan.block_layout("pband", 0, j)
        if want > 0 and fmt == S.BLOCK_PBAND:
            corner += want > n - w
            band += want <= n - w
    assert band >= 1 and (corner >= 2 or where == "third"), (corner, band)


@pytest.mark.parametrize("fprec,tol", [("fp64", 1e-12), ("fp32x2", 1e-10)])
def test_window_against_chunked_lmax3000(fprec, tol):
    """Rings of up to 6075 pixels: the two kernels' factors of the same blocks.
    Backward errors of (2w + 2) 2^-53 and 2^-44 for w <= 10, times conditions of
    up to a few hundred."""
    from paper_1504_04653_gb300 import sympix as S
    wl, grid, plan, ninv, blocks = _sampled(S, "lmax3000")
    out = {}
    for k in (2, 3):
        b = blocks.clone()
        plan.set_narrow_factor(k)
        assert int((S.sympix_factor_blocks(plan, b, precision=fprec) != 0).sum()) == 0
        out[k] = b
    for j in (5, 300, 901, 902, 1500, 2098, 2700):
        off, n, w, fmt = plan.block_layout("pband", 0, j)
        assert fmt == S.BLOCK_PBAND
        m = n - w
        band = [b[off:off + m * (w + 1)].cpu().numpy().reshape(m, w + 1) for b in out.values()]
        live = np.arange(w + 1)[None, :] <= np.arange(m)[:, None]
        bord = [b[off + n * (w + 1):off + n * (2 * w + 1)].cpu().numpy().reshape(w, n) for b in out.values()]
        lower = np.arange(n)[None, :] <= m + np.arange(w)[:, None]
        top = np.max(np.abs(band[1][live]))
        assert np.max(np.abs(band[0] - band[1])[live]) <= tol * top, (j, n, w)
        assert np.max(np.abs(bord[0] - bord[1])[lower]) <= tol * top, (j, n, w)
