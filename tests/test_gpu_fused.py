"""The fused persistent Adam kernel where it runs: blocks of 4 and 16 sites (four warps per block),
and larger small blocks below the nested elimination's temperature line (a CTA per block).

Five Adam updates against the oracle's (spectral route) from the same seeded start; tolerances of
the fused path's other tests: phi within 1e-10 (float64) and 1e-6 (float32 blocks)."""
import numpy as np
import pytest

import oracle
from paper_2311_04435_gb300 import api, inputs

pytestmark = pytest.mark.gpu


# one block, a ragged count, one per SM and more (teams that take several blocks); L = 2 has
# doubled bonds
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("L,nw,T", [(2, 1, 0.3), (2, 77, 0.1), (4, 1, 0.3), (4, 5, 0.05),
                                    (4, 76, 0.1), (4, 311, 0.02), (4, 3, 0.004), (6, 5, 0.006),
                                    (8, 80, 0.006), (12, 3, 0.006)])
def test_fused_steps_match_oracle(L, nw, T, prec):
    p = api.Params(L, nw, U=4.0, T=T, delta=0.6, mu=0.1, t=0.9, prec=prec, ionic="half")
    ee = inputs.random_phi(3, p.N, 0.4)
    with api.Context(p) as c:
        c.set_site_energy(ee)
        c.adam_init(api.AdamConfig(lr=0.01, seed=1))
        om, gm = c.adam_step(5)
        phi = c.phi()
    op = oracle.make_params(L, nw, U=4.0, T=T, delta=0.6, mu=0.1, t=0.9, ionic=1)
    start = oracle.seed_phi(1, p.N)
    phi4 = oracle.adam_run_spectral(op, start, lr=0.01, max_steps=4, eps_extra=ee)[0]
    phi5 = oracle.adam_run_spectral(op, start, lr=0.01, max_steps=5, eps_extra=ee)[0]
    o_om, o_g = oracle.omega_grad_spectral(op, phi4, ee)[:2]
    tol = 1e-10 if prec == "fp64" else 1e-6
    assert np.max(np.abs(phi - phi5)) < tol
    assert om == pytest.approx(o_om, rel=tol)
    assert gm == pytest.approx(np.abs(o_g).max(), rel=1e3 * tol, abs=tol)
