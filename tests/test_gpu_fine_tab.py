"""Fine-level tables and the spread transfer kernels at ragged and smallest sizes, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import multigrid as mg, operators as op
from paper_1806_11277_gb300 import ehs, synth

pytestmark = pytest.mark.gpu


def _media(shape, n):
    if len(shape) == 2:
        return [synth.random_2d(n=shape[0], nx=shape[1], sigma=0.3, seed=k, corr=3.0, abl=2) for k in range(n)]
    m = synth.layered_3d(n=max(shape), abl=2, corr=3.0)
    cut = tuple(slice(0, s) for s in shape)
    return [synth.Medium(m.lam[cut], m.mu[cut], m.rho[cut], m.omega, m.h, 2)]


# the smallest grids, a block that ends inside a row, several items per medium and several media; 2D and 3D
@pytest.mark.parametrize("shape,media,nrhs", [((4, 4), 1, 1), ((12, 20), 2, 2), ((36, 28), 1, 1), ((4, 8, 4), 1, 2),
                                              ((12, 8, 20), 1, 1)])
def test_fine_level_and_transfers_match_the_oracle(shape, media, nrhs):
    meds = _media(shape, media)
    d = len(shape)
    with ehs.solver_for(meds, levels=2, alpha=0.3, nrhs=nrhs, w=[0.6]) as S:
        for dt, tol in ((torch.complex128, 1e-11), (torch.complex64, 2e-5)):   # the bars of a sweep
            gen = torch.Generator(device="cuda").manual_seed(3)
            vec = lambda l: torch.randn(S.level_shape(l), dtype=torch.complex128, device="cuda", generator=gen).to(dt)
            x, b, e = vec(0), vec(0), vec(1)
            for v in (x, b, e):
                for k in range(d):
                    v[:, k].select(d - k, 0).zero_()
            y, ys, sm, rc, pr = (torch.zeros_like(x) for _ in range(5))
            rc = torch.zeros_like(e)
            S.op_apply(x, y)
            S.op_apply(x, ys, shifted=True)
            sm.copy_(x)
            S.smooth(b, sm, nsweeps=2)
            S.residual_restrict(b, x, rc)
            pr.copy_(x)
            S.prolong_add(e, pr)
            for it in range(S.items):
                parts = op.parts_for(meds[it // nrhs])
                K, Ks = op.assemble_mixed(parts), op.assemble_mixed(parts, 0.3)
                H = mg.Hierarchy(Ks, shape, 2, w=[0.6])
                cs = tuple(s // 2 for s in shape)
                f = lambda v, sh: op.slots_to_dofs(v[it].cpu().numpy().astype(np.complex128), sh)
                xe, be, ee = f(x, shape), f(b, shape), f(e, cs)
                want = [(y, K @ xe, shape), (ys, Ks @ xe, shape), (sm, H.relax(0, be, H.relax(0, be, xe)), shape),
                        (rc, H.P[0].T @ (be - Ks @ xe), cs), (pr, xe + H.P[0] @ ee, shape)]
                for got, ref, sh in want:
                    g = f(got, sh)
                    assert np.abs(g - ref).max() / np.abs(ref).max() <= tol, (it, dt)
