"""FP64 coarsest solves in any choice of units (k_dense.cu, k_invert.cu): the inverse must not lose digits where
displacements and pressures differ in scale, nor across a strong contrast of the medium."""
import numpy as np
import pytest
import torch

from oracle import multigrid as mg, operators as op
from paper_1806_11277_gb300 import ehs, synth

pytestmark = pytest.mark.gpu

ALPHA = 0.2


def _medium(units, shape):
    if len(shape) == 2:
        m = synth.random_2d(n=shape[0], nx=shape[1], sigma=0.25, seed=3, corr=4.0, abl=4)
    else:
        full = synth.layered_3d(n=max(shape), abl=2, corr=3.0)
        cut = tuple(slice(0, s) for s in shape)
        m = synth.Medium(full.lam[cut], full.mu[cut], full.rho[cut], full.omega, full.h, 2)
    lam, mu, rho, omega, h = m.lam, m.mu, m.rho, m.omega, m.h
    if units == "si":                     # km/s and g/cm^3 with h = 1 -> m/s and kg/m^3 with h = 10 m
        lam, mu, rho, omega, h = lam * 1e9, mu * 1e9, rho * 1e3, omega * 100.0, 10.0
    elif units == "unit square":
        h, omega = 1.0 / 512, omega * 512
    elif units == "contrast":             # stiff stripes, 1e4 in mu and lambda
        f = np.where(np.arange(shape[-1]) // 7 % 2 == 0, 1.0, 1e4)
        lam, mu = lam * f, mu * f
    elif units == "nearly incompressible":
        lam = lam * 1e3
    return synth.Medium(lam, mu, rho, omega, h, m.abl_cells)


class _Scaled:
    """Solves with a dense matrix equilibrated by its diagonal, one step of refinement in extended precision."""

    def __init__(self, K):
        self.d = 1.0 / np.sqrt(np.abs(K.diagonal()))
        self.A = (K.toarray() * self.d[:, None]) * self.d
        self.cond = np.linalg.cond(self.A)

    def solve(self, b):
        bs = b * self.d
        x = np.linalg.solve(self.A, bs)
        r = bs.astype(np.clongdouble) - self.A.astype(np.clongdouble) @ x.astype(np.clongdouble)
        return (x + np.linalg.solve(self.A, r.astype(np.complex128))) * self.d


def _overlap(med):
    return 2 if med.lam.ndim == 2 else 1      # half a core at most: 6 cells in 2D, 2 in 3D


def _hierarchy(med, split):
    parts = op.parts_for(med)
    H = mg.Hierarchy(op.assemble_mixed(parts, ALPHA), med.lam.shape, 3,
                     coarse_dd=(split, _overlap(med)) if split else None)
    if split:
        H.cdd.subs = [(c, idx, _Scaled(H.K[-1][idx][:, idx])) for c, idx, _ in H.cdd.subs]
    else:
        H.coarse = _Scaled(H.K[-1])
        H.coarse_solve = H.coarse.solve
    return H


# 12 x 14 coarsest cells: no component ends at a whole block of columns, with or without subdomains
@pytest.mark.parametrize("split", [None, (2, 2)])
@pytest.mark.parametrize("units", ["km", "si", "unit square", "contrast", "nearly incompressible"])
def test_coarsest_solve_and_cycle_in_any_units(units, split):
    _check(units, (48, 56), split)


@pytest.mark.parametrize("split", [None, (2, 2, 1)])
def test_coarsest_solve_and_cycle_in_si_units_3d(split):
    _check("si", (16, 24, 16), split)


def _check(units, shape, split):
    med = _medium(units, shape)
    H = _hierarchy(med, split)
    kw = dict(coarse_dd=tuple(split) + (1,) * (3 - len(split)), coarse_dd_overlap=_overlap(med)) if split else {}
    rng = np.random.default_rng(5)
    with ehs.solver_for(med, levels=3, alpha=ALPHA, w=[0.75, 0.5], prec=ehs.EHS_C128, **kw) as S:
        for level, run, ref in ((2, S.coarse_solve, H.coarse_solve), (0, S.vcycle, H.cycle)):
            K = H.K[level]
            d = 1.0 / np.sqrt(np.abs(K.diagonal()))         # both equations and both unknowns of size one
            b = (rng.standard_normal(K.shape[0]) + 1j * rng.standard_normal(K.shape[0])) / d
            bt = torch.from_numpy(op.dofs_to_slots(b, H.shapes[level])[None]).cuda()
            xt = torch.empty_like(bt)
            run(bt, xt)
            x, want = op.slots_to_dofs(xt[0].cpu().numpy(), H.shapes[level]) / d, ref(b) / d
            # an exact coarsest solve: the rounding errors of N steps, summed as a random walk, times the condition
            # of the equilibrated matrix (18 to 160 here); else the bar of one FP64 cycle
            tol = 4 * np.sqrt(K.shape[0]) * 2.0 ** -53 * H.coarse.cond if level and not split else 1e-10
            nu = sum(op.dof_sizes(H.shapes[level])[:-1])
            for part in (slice(0, nu), slice(nu, None)):
                err = np.abs(x - want)[part].max() / np.abs(want[part]).max()
                assert err <= tol, (level, err)


# the panel in global memory (N > 12800) and the 16-column panel with several matrices (N > 3200)
@pytest.mark.parametrize("cells,media", [((64, 67), 1), ((33, 33), 2)])
def test_large_coarsest_solve_inverts_the_coarsest_operator(cells, media):
    meds = [synth.random_2d(n=2 * cells[0], nx=2 * cells[1], sigma=0.25, seed=k, corr=4.0, abl=4)
            for k in range(media)]
    with ehs.solver_for(meds, levels=2, alpha=ALPHA, prec=ehs.EHS_C128) as S:
        gen = torch.Generator(device="cuda").manual_seed(1)
        b = torch.randn(S.level_shape(1), dtype=torch.complex128, device="cuda", generator=gen)
        b[:, 0, :, 0] = 0
        b[:, 1, 0, :] = 0
        x, r = torch.empty_like(b), torch.empty_like(b)
        S.coarse_solve(b, x)
        S.op_apply(x, r, level=1, shifted=True)
        # backward stable: |A x - b| <= c N u |A| |A^{-1}| |b|, |A| |A^{-1}| below 1e3 here
        n = 3 * cells[0] * cells[1]
        assert float(((r - b).abs().amax() / b.abs().amax()).cpu()) <= n * 2.0 ** -53 * 1e3


# finite media whose operator overflows FP64: setup reports the matrix, with or without subdomains
@pytest.mark.parametrize("split", [(1, 1, 1), (2, 2, 1)])
def test_a_coarsest_matrix_that_overflows_is_reported(split):
    m = synth.random_2d(n=48, nx=56, sigma=0.25, seed=3, corr=4.0, abl=4)
    f = 1e308 / m.mu.max()
    huge = synth.Medium(-0.5 * f * m.mu, f * m.mu, m.rho, m.omega, m.h, m.abl_cells)
    with pytest.raises(ehs.EhsError, match="singular") as e:
        ehs.solver_for(huge, levels=3, alpha=ALPHA, prec=ehs.EHS_C128, coarse_dd=split, coarse_dd_overlap=2).close()
    assert ehs.STATUS[e.value.status] == "ERR_ARG"
