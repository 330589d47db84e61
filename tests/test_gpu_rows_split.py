"""Galerkin rows split over warps and the one-launch colour relaxation (k_stencil_split.cu) against one thread per row."""
import pytest
import torch

from paper_1806_11277_gb300 import ehs, synth

pytestmark = pytest.mark.gpu


def _vec(shp, dt, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(shp, dtype=torch.complex128, device="cuda", generator=gen)
    d = len(shp) - 2
    for k in range(d):
        v[:, k].select(d - k, 0).zero_()
    return v.to(dt)


# fine cells (n_y, n_x) / (n_z, n_y, n_x), items: the smallest level, rows that do not fill a block of 32 cells, a
# colour whose cells end inside a block, the largest 2D level of the rule (128^2), items of one and of several media
@pytest.mark.parametrize("half", [0, 1, 2])
@pytest.mark.parametrize("shape,levels,media,nrhs", [((8, 8), 3, 1, 1), ((40, 24), 3, 2, 1), ((56, 88), 4, 1, 3),
                                                      ((256, 256), 3, 1, 1), ((8, 16, 8), 3, 1, 2),
                                                      ((24, 8, 16), 3, 1, 1), ((16, 16, 32), 3, 1, 2)])
def test_split_rows_equal_whole_rows(shape, levels, media, nrhs, half, monkeypatch):
    d = len(shape)
    if d == 2:
        meds = [synth.random_2d(n=shape[0], nx=shape[1], sigma=0.3, seed=k, corr=4.0, abl=2) for k in range(media)]
    else:
        m = synth.layered_3d(n=max(shape), abl=2, corr=3.0)
        cut = tuple(slice(0, s) for s in shape)
        meds = [synth.Medium(m.lam[cut], m.mu[cut], m.rho[cut], m.omega, m.h, 2)]
    got = []
    for fixed in (None, "0"):
        if fixed is not None:
            monkeypatch.setenv("EHS_ROWS_VARIANT", fixed)
        out = []
        with ehs.solver_for(meds, levels=levels, alpha=0.4, nrhs=nrhs, coef_half=half) as S:
            for dt in (torch.complex64, torch.complex128):
                for l in range(1, levels):
                    x, b = _vec(S.level_shape(l), dt, l), _vec(S.level_shape(l), dt, 10 + l)
                    y = torch.empty_like(x)
                    S.op_apply(x, y, level=l)
                    out.append(y)
                    if l < levels - 1:
                        S.smooth(b, x, level=l, nsweeps=2)
                        out.append(x)
        got.append(out)
    # the same sums in another order: a row has at most 285 products and its rounding is bounded by 285 units of the
    # largest of them; the parity bars of the operator and of a sweep (1e-5 and 2e-5) hold that against FP64
    for a, b in zip(*got):
        tol = 2e-5 if a.dtype == torch.complex64 else 1e-12
        assert float((a - b).abs().max() / b.abs().max()) <= tol


# MG-DD colour residuals: a row over two warps above 200 K box unknowns, over four below (a right-hand side alone);
# boxes whose unknowns end inside a block, and unequal ones
@pytest.mark.parametrize("shape,split", [((128, 160), (4, 4, 1)), ((160, 152), (4, 3, 1))])
@pytest.mark.parametrize("fmt", [0, 2])
def test_gather_of_a_large_batch_equals_single_ones(shape, split, fmt):
    n = 32
    med = [synth.random_2d(n=shape[0], nx=shape[1], sigma=0.3, seed=7, corr=4.0, abl=2)]
    kw = dict(levels=3, alpha=0.4, coarse_dd=split, coarse_dd_overlap=3, coarse_fmt=fmt, coef_half=1 if fmt else 0)
    with ehs.solver_for(med, nrhs=n, **kw) as S, ehs.solver_for(med, nrhs=1, **kw) as S1:
        for dt in (torch.complex64, torch.complex128):
            b = _vec(S.level_shape(0), dt, 3)
            x = torch.empty_like(b)
            S.vcycle(b, x)
            # twice the bar of one cycle against the FP64 oracle
            tol = 1e-4 if dt == torch.complex64 else 2e-10
            for i in (0, n - 1):
                x1 = torch.empty_like(b[i:i + 1])
                S1.vcycle(b[i:i + 1].contiguous(), x1)
                assert float((x[i] - x1[0]).abs().max() / x1.abs().max()) <= tol
