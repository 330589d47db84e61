"""FP64 inverses of the coarsest matrices (k_invert.cu) at the edges of its blocks, tiles and storage rules."""
import numpy as np
import pytest
import torch

from paper_1806_11277_gb300 import ehs, synth

pytestmark = pytest.mark.gpu


# coarsest cells (n_y, n_x) -> N = 3 n_y n_x: below one block of 32 columns, one column over, whole blocks and
# update tiles, a ragged end, the first sizes of the 16-column panel (N > 3200) and of the panel in global
# memory (N > 6400); one and several matrices per launch
@pytest.mark.parametrize("cells,media", [((2, 2), 1), ((11, 1 + 2), 3), ((4, 8), 2), ((8, 8), 1), ((5, 13), 2),
                                          ((32, 34), 1), ((46, 47), 1)])
def test_exact_coarsest_solve_inverts_the_coarsest_operator(cells, media):
    ny, nx = 2 * cells[0], 2 * cells[1]
    meds = [synth.random_2d(n=ny, nx=nx, sigma=0.25 + 0.1 * k, seed=k, corr=4.0, abl=1) for k in range(media)]
    with ehs.solver_for(meds, levels=2, alpha=0.2, prec=ehs.EHS_C128) as S:
        gen = torch.Generator(device="cuda").manual_seed(1)
        b = torch.randn(S.level_shape(1), dtype=torch.complex128, device="cuda", generator=gen)
        b[:, 0, :, 0] = 0
        b[:, 1, 0, :] = 0
        x, r = torch.empty_like(b), torch.empty_like(b)
        S.coarse_solve(b, x)
        S.op_apply(x, r, level=1, shifted=True)
        # a backward stable inverse leaves |A x - b| <= c N u |A| |A^{-1}| |b|, |A| |A^{-1}| below 1e3 here
        n = 3 * cells[0] * cells[1]
        err = float(((r - b).abs().amax() / b.abs().amax()).cpu())
        assert err <= max(n, 32) * 2.0 ** -53 * 1e3, err
        assert bool(np.isfinite(err))
