"""Site terms far above the rest, up to float32's range, in the default elimination of the reduced
precisions: the site decouples, the others are as they are without it."""
import numpy as np
import pytest

from paper_2311_04435_gb300 import api, inputs

pytestmark = pytest.mark.gpu


# T = 0.03: the first blocks in sums of three float32; a pivot of every kind of front holds the
# large term in turn (leaf, separators, root)
@pytest.mark.parametrize("prec", ["fp32", "bf16x3"])
@pytest.mark.parametrize("T", [0.03, 0.2, 0.7])
def test_large_site_terms(T, prec):
    """Against the float64 dense elimination of the same field; double-float's 2^-48 with the
    margin of the other tests of this elimination: 1e-10."""
    L = 14
    for site, big in ((0, 1e19), (3, -1e25), (17, 2e30), (45, 1e37), (100, -3e37), (150, 5e18)):
        phi = inputs.random_phi(site, L * L, 0.8)
        phi[site] = big
        ref = {}
        for q in ("fp64", prec):
            with api.Context(api.Params(L, 8, U=4.0, T=T, delta=0.3, mu=0.1, prec=q)) as c:
                if q == "fp64":
                    c.set_pivoting("partial")
                ref[q] = c.blocks(phi)
                if q == prec:
                    om, g = c.grad(phi)
                    assert np.isfinite(om) and np.all(np.isfinite(g))
        (ld, gd), (ld64, gd64) = ref[prec], ref["fp64"]
        assert np.max(np.abs(gd - gd64)) <= 1e-10, site
        assert np.max(np.abs(ld - ld64) / np.abs(ld64)) <= 1e-10, site


def test_large_energies_of_a_density_of_states():
    p = api.Params(12, 4, U=4.0, T=0.1, delta=0.3, prec="fp32")
    phi = inputs.random_phi(1, p.N, 0.8)
    w = np.array([0.0, 1e20, -3e30, 0.5])
    with api.Context(p) as c:
        rho = c.dos(phi, w, 0.2)
    with api.Context(p) as c:
        near = c.dos(phi, w[[0, 3]], 0.2)
    assert np.array_equal(rho[:, [0, 3]], near)
    assert np.all(np.abs(rho[:, 1:3]) <= 1e-35)  # eta / (pi w^2)
