"""The nested elimination (the path of a new context from 6 x 6 sites up) against the dense pivoted
elimination of the same context and the FP64 oracle.

Tolerances: float64 1e-11 (the oracle's dense LU and both GPU paths are good to a few hundred
2^-52 times |G| <= 1 / omega_0 here); double-float 2^-48 products through the same elimination,
1e-10 with the same margin; the dense reduced precisions keep the parity tests' 1e-7 and 2e-6.
"""
import numpy as np
import pytest

import oracle
from paper_2311_04435_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def _oparams(p):
    return oracle.make_params(p.L, p.n_omega, U=p.U, T=p.T, delta=p.delta, t=p.t, mu=p.mu,
                              ionic=0 if p.ionic == "paper" else 1)


# trees of every depth up to eight levels; fronts of one and several panels; leaves of 1 to 20
# sites, odd and even sides, in both forms (omega_0 and omega_1 below 4t, the others above)
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x3"])
@pytest.mark.parametrize("L", [6, 8, 10, 12, 14, 16, 18, 22, 24, 34])
def test_blocks_match_dense_elimination_and_oracle(L, prec):
    p = api.Params(L, 4, U=4.0, T=0.3, delta=0.9, mu=0.2, t=0.8, prec=prec, ionic="half")
    phi = inputs.random_phi(200 + L, p.N, 1.0)
    ee = inputs.random_phi(300 + L, p.N, 0.5)
    with api.Context(p) as c:
        c.set_site_energy(ee)
        ld, gd = c.blocks(phi)
        om, g = c.grad(phi)
        om_lu = c.potential(phi)
        again = c.blocks(phi)
        c.set_pivoting("partial")
        ld_d, gd_d = c.blocks(phi)
        c.set_pivoting("none")
        ld_n, gd_n = c.blocks(phi)
    tol = 1e-11 if prec == "fp64" else 1e-10
    assert np.array_equal(ld, again[0]) and np.array_equal(gd, again[1])
    assert np.array_equal(ld, ld_n) and np.array_equal(gd, gd_n)
    assert om_lu == om
    dense = dict(g=1e-10, ld=1e-10) if prec == "fp64" else dict(g=1e-7, ld=2e-6)
    assert np.max(np.abs(gd - gd_d)) <= dense["g"] and np.allclose(ld, ld_d, rtol=dense["ld"])
    o_om, o_g, o_ld, o_gd = oracle.omega_grad(_oparams(p), phi, eps_extra=ee, per_block=True)
    assert np.max(np.abs(gd - o_gd)) <= tol
    assert np.max(np.abs(ld - o_ld) / np.abs(o_ld)) <= tol
    assert om == pytest.approx(o_om, rel=tol) and np.max(np.abs(g - o_g)) <= 10 * tol


@pytest.mark.parametrize("prec", ["fp64", "3xtf32"])
def test_rule_on_the_smallest_frequency(prec):
    """Above the line the default differs from the dense elimination in the last bits, below it
    (pi T = 0.028) it is the dense elimination; the same for a density of states' eta."""
    w = np.linspace(-3.0, 3.0, 5)
    for T, nested in ((0.0105, True), (0.009, False)):
        p = api.Params(14, 3, U=4.0, T=T, delta=0.4, prec=prec)
        phi = inputs.random_phi(5, p.N, 1.0)
        with api.Context(p) as c:
            a, rho = c.blocks(phi)[1], c.dos(phi, w, T * np.pi)
            c.set_pivoting("partial")
            b, rho_d = c.blocks(phi)[1], c.dos(phi, w, T * np.pi)
        assert np.array_equal(a, b) != nested and np.array_equal(rho, rho_d) != nested
        assert np.max(np.abs(a - b)) <= (1e-10 if prec == "fp64" else 1e-6) * np.abs(b).max()
        assert np.max(np.abs(rho - rho_d)) <= (1e-10 if prec == "fp64" else 1e-4) * rho_d.max()


@pytest.mark.parametrize("L,prec", [(8, "fp32"), (14, "fp64"), (20, "bf16x3")])
def test_chunks_forward_backward_and_nan(L, prec, monkeypatch):
    torch = pytest.importorskip("torch")
    p = api.Params(L, 5, U=4.0, T=0.2, delta=0.4, prec=prec)
    phi = inputs.random_phi(L, p.N, 1.0)
    with api.Context(p) as c:
        om, g = c.grad(phi)
        x = torch.tensor(phi, dtype=torch.float64, device="cuda")
        om_t, g_t = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(x)
        c.forward_dev(x, om_t)
        c.backward_dev(x, g_t)
        torch.cuda.synchronize()
        assert float(om_t) == om and np.array_equal(g_t.cpu().numpy(), g)
        bad = phi.copy()
        bad[p.N // 2] = np.nan
        with pytest.raises(Exception, match="SCA_ENONFINITE"):
            c.grad(bad)
        assert np.array_equal(c.grad(phi)[1], g)
    monkeypatch.setenv("SCA_MAX_BLOCKS_RESIDENT", "3")
    with api.Context(p) as c:
        om3, g3 = c.grad(phi)
    assert om3 == om and np.array_equal(g3, g)


def test_profile_counts_the_nested_launches():
    """One launch eliminates and takes diag(G); a forward / backward pair takes two."""
    p = api.Params(20, 4, U=4.0, T=0.1, delta=0.4, prec="bf16x3")
    phi = inputs.seed_phi(1, p.N)
    with api.Context(p) as c:
        ref = c.grad(phi)
        c.profile(2)
        got = c.grad(phi)
        prof = c.profile_read()
    assert prof["nest_up"][1] == 1 and prof["nest_down"][1] == 0 and prof["update"][1] == 0
    assert prof["nest_up"][0] > 0.0 and got[0] == ref[0] and np.array_equal(got[1], ref[1])


def test_served_requests_on_both_sides_of_the_line():
    """Requests of one size bucket whose temperatures lie on both sides of the rule run in passes
    of their own kind and give what each gives alone."""
    reqs = [(api.Params(16, 3, U=4.0, T=T, delta=0.6, prec="bf16x3"),
             api.AdamConfig(lr=0.01, grad_tol=1e-9, max_steps=6, seed=40 + k))
            for k, T in enumerate((0.1, 0.005, 0.2, 0.006))]
    alone = [api.solve(p, a) for p, a in reqs]
    with api.Server(hbm_budget_bytes=8 << 30, max_slots=4, manual=True) as srv:
        ids = [srv.submit(p, a) for p, a in reqs]
        now = 0.0
        while any(srv.step(now)):
            now += 0.1
        mixed = [srv.poll(rid, 256) for rid in ids]
    for x, y in zip(alone, mixed):
        assert x.steps == y.steps and x.omega == y.omega and np.array_equal(x.phi, y.phi)


@pytest.mark.parametrize("L,prec,n_omega,t", [(6, "fp32", 77, 1.0), (8, "bf16x3", 110, 1.0),
                                              (8, "fp64", 80, 8.0), (20, "bf16x3", 100, 1.0)])
def test_more_blocks_than_sms(L, prec, n_omega, t):
    """A launch per level, the blocks in parts side by side (with t = 8 fewer than 64 of them have
    closed-form leaves): every block as the oracle has it, and to the bit what a pass of few
    blocks gives; the same for a density of states, where every block has dense leaves."""
    p = api.Params(L, n_omega, U=4.0, T=0.1, delta=0.9, t=t, prec=prec)
    phi = inputs.random_phi(400 + L, p.N, 1.0)
    w = np.linspace(-4.0, 4.0, 90)
    with api.Context(p) as c:
        ld, gd = c.blocks(phi)
        om = c.potential(phi)
        g = c.grad(phi)
        rho = c.dos(phi, w, 0.3)
    with api.Context(api.Params(L, 10, U=4.0, T=0.1, delta=0.9, t=t, prec=prec)) as c:
        few = c.blocks(phi)
        rho_few = np.concatenate([c.dos(phi, w[k:k + 10], 0.3) for k in range(0, 90, 10)], axis=1)
    assert np.array_equal(ld[:20], few[0]) and np.array_equal(gd[:20], few[1])
    assert np.array_equal(rho, rho_few) and om == g[0]
    o_om, o_g, o_ld, o_gd = oracle.omega_grad(_oparams(p), phi, per_block=True)
    tol = 1e-11 if prec == "fp64" else 1e-10
    assert np.max(np.abs(gd - o_gd)) <= tol
    assert np.max(np.abs(ld - o_ld) / np.abs(o_ld)) <= tol
    assert om == pytest.approx(o_om, rel=tol) and np.max(np.abs(g[1] - o_g)) <= 10 * tol
