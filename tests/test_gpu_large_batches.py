"""Batches large enough for the launch forms of large problems: every item gets what it gets alone."""
import pytest
import torch

from paper_1806_11277_gb300 import ehs, synth

pytestmark = pytest.mark.gpu


def _medium(shape):
    if len(shape) == 2:
        return synth.random_2d(n=shape[0], nx=shape[1], sigma=0.3, seed=7, corr=4.0, abl=2)
    m = synth.layered_3d(n=max(shape), abl=2, corr=3.0)
    cut = tuple(slice(0, s) for s in shape)
    return synth.Medium(m.lam[cut], m.mu[cut], m.rho[cut], m.omega, m.h, 2)


def _vec(shp, dt, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(shp, dtype=torch.complex128, device="cuda", generator=gen)
    d = len(shp) - 2
    for k in range(d):
        v[:, k].select(d - k, 0).zero_()
    return v.to(dt)


def _compare(shape, nrhs, levels, dt, run, tol, **kw):
    """run(S, n): outputs of the call under test on the first n sources; items 0, 1 and the last against one source."""
    med = _medium(shape)
    kw = dict(levels=levels, alpha=0.4, restart=1, **kw)
    with ehs.solver_for(med, nrhs=nrhs, **kw) as S, ehs.solver_for(med, nrhs=1, **kw) as S1:
        outs = run(S, lambda l, seed: _vec(S.level_shape(l), dt, seed))
        for i in (0, 1, nrhs - 1):
            ones = run(S1, lambda l, seed: _vec(S.level_shape(l), dt, seed)[i:i + 1].contiguous())
            for a, b in zip(outs, ones):
                assert float((a[i] - b[0]).abs().max() / b.abs().max()) <= tol, i


# residual passes of Galerkin levels, every launch shape: ragged rows, more than one block an item, an odd batch
@pytest.mark.parametrize("variant", ["0", "1", "2", "3"])
@pytest.mark.parametrize("shape,nrhs,half", [((72, 104), 5, 0), ((72, 104), 5, 2), ((24, 16, 20), 3, 0),
                                             ((24, 16, 20), 3, 1)])
def test_galerkin_rows(shape, nrhs, half, variant, monkeypatch):
    monkeypatch.setenv("EHS_ROWS_VARIANT", variant)

    def run(S, vec):
        out = []
        for l in (1, 2):
            x, b = vec(l, l), vec(l, 10 + l)
            y = torch.empty_like(x)
            S.op_apply(x, y, level=l)
            out.append(y)
            if l == 1:
                S.smooth(b, x, level=l, nsweeps=2)
                out.append(x)
        return out

    for dt, tol in ((torch.complex64, 2e-5), (torch.complex128, 1e-12)):   # the bars of an operator and a sweep
        _compare(shape, nrhs, 3, dt, run, tol, coef_half=half)


# 3D rows split over warps, two items a block: a last block with one item, pairs that straddle two media, sizes on both
# sides of the limits of the split form (FP64 4096 cells of the batch, FP16 tables 16384, an odd batch 32768)
@pytest.mark.parametrize("half", [0, 1])
@pytest.mark.parametrize("shape,media,nrhs", [((16, 16, 8), 1, 3), ((16, 16, 8), 2, 3), ((32, 16, 32), 1, 3),
                                              ((48, 40, 48), 1, 3)])
def test_split_rows_of_odd_batches(shape, media, nrhs, half, monkeypatch):
    m = _medium(shape)
    meds = [synth.Medium(m.lam * (1 + 0.2 * k), m.mu, m.rho * (1 - 0.1 * k), m.omega, m.h, 2) for k in range(media)]
    got = []
    for fixed in (None, "0"):
        if fixed is not None:
            monkeypatch.setenv("EHS_ROWS_VARIANT", fixed)
        out = []
        with ehs.solver_for(meds, levels=3, alpha=0.4, nrhs=nrhs, coef_half=half, restart=1) as S:
            for dt in (torch.complex64, torch.complex128):
                for l in (1, 2):
                    x = _vec(S.level_shape(l), dt, l)
                    y = torch.empty_like(x)
                    S.op_apply(x, y, level=l)
                    out.append(y)
        got.append(out)
    for a, b in zip(*got):                    # the same sums in another order: the bars of the operator
        tol = 1e-5 if a.dtype == torch.complex64 else 1e-12
        assert float((a - b).abs().max() / b.abs().max()) <= tol


# complex64 prolongations above 400 K cells of the batch run a thread per cell instead of per component
@pytest.mark.parametrize("shape,nrhs", [((136, 120), 25), ((24, 16, 20), 55)])
def test_prolongation(shape, nrhs):
    def run(S, vec):
        x = vec(0, 1)
        S.prolong_add(vec(1, 2), x)
        return [x]

    _compare(shape, nrhs, 3, torch.complex64, run, 1e-5)


# FP64 products with the coarsest inverses: plain launches from 2048 rows of the batch on (11 items of 192 rows)
@pytest.mark.parametrize("split", [(1, 1, 1), (2, 2, 1)])
def test_fp64_coarsest_products(split):
    def run(S, vec):
        b = vec(2, 3)
        x = torch.empty_like(b)
        S.coarse_solve(b, x)
        return [x]

    _compare((32, 32), 11, 3, torch.complex128, run, 1e-10, prec=ehs.EHS_C128, coarse_dd=split, coarse_dd_overlap=1)


# the complex64 operator: a plain launch above 1.5 M cells of the batch in 3D
@pytest.mark.parametrize("shape,nrhs", [((24, 16, 20), 197)])
def test_complex64_operator(shape, nrhs):
    def run(S, vec):
        x, b = vec(0, 1), vec(0, 2)
        y, r = torch.empty_like(x), torch.empty(S.level_shape(1), dtype=x.dtype, device=x.device)
        S.op_apply(x, y)
        S.residual_restrict(b, x, r)
        return [y, r]

    _compare(shape, nrhs, 3, torch.complex64, run, 1e-5)
