"""pz_set_corrections sends the species-to-element map only when it changes: alternating maps,
and calls without abundances between them, give what a fresh context gives."""
import numpy as np
import pytest

import paper_2607_24141_gb300 as pz
from tiny import tiny_problem

pytestmark = pytest.mark.gpu


def test_alternating_element_maps():
    import torch
    prob = tiny_problem(n_lambda=300, n_depth=9, n_lines=60, W=80)
    ns = prob.atmos.n_species
    maps = [np.array([0, 1, 0], np.int32)[:ns], np.array([1, 0, 0], np.int32)[:ns], np.array([-1, 1, 1], np.int32)[:ns]]
    dab = np.array([0.4, -0.3], np.float32)

    def kappa(s):
        kl = torch.empty((prob.atmos.n_depth, prob.grid.n_lambda), dtype=torch.float32, device=s.device)
        pz.pz_line_opacity(s.ctx, kl)
        return kl.cpu().numpy()

    fresh = []
    for m in maps + [None]:
        s = pz.Synthesizer(prob)
        pz.pz_set_corrections(s.ctx, None, None, None if m is None else dab, m, 0 if m is None else 2)
        fresh.append(kappa(s))
        s.close()
    assert not np.allclose(fresh[0], fresh[1], rtol=1e-3) and not np.allclose(fresh[0], fresh[3], rtol=1e-3)
    s = pz.Synthesizer(prob)
    for k in (0, 0, 1, 3, 1, 2, 3, 3, 0, 2):
        m = None if k == 3 else maps[k]
        pz.pz_set_corrections(s.ctx, None, None, None if m is None else dab, m, 0 if m is None else 2)
        np.testing.assert_allclose(kappa(s), fresh[k], rtol=2e-6)
    s.close()
