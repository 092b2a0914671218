"""The dense elimination where the nested one is the default: asked for by partial pivoting (or below
the temperature line), at its full sizes, with its groups, SM partitions, resident inverses and
densities of states, each checked to be the path that ran; and the default beside it at the
tolerance of its own arithmetic.

Tolerances: dense as in the parity tests (float64 1e-10; the others 1e-7 of diag(G), 2e-6 of
ln|det|, 1e-5 of Omega; densities of states 2e-5 of the largest); the default 1e-10 in every
precision."""
import math

import numpy as np
import pytest

import oracle
from paper_2311_04435_gb300 import api, inputs

pytestmark = pytest.mark.gpu


def oparams(p):
    return oracle.make_params(p.L, p.n_omega, U=p.U, T=p.T, delta=p.delta, t=p.t, mu=p.mu,
                              ionic=0 if p.ionic == "paper" else 1)


def tol(prec, dense=True):
    if prec == "fp64" or not dense:
        return dict(om=1e-10, ld=1e-10, g=1e-10)
    return dict(om=1e-5, ld=2e-6, g=1e-7)


def ran(c, call):
    """The result of a call and the kinds of kernel that it launched."""
    c.profile(2)
    out = call()
    prof = c.profile_read()
    c.profile(False)
    return out, {k for k, (_, n) in prof.items() if n}


def check(res, ref, t):
    (ld, gd), (o_ld, o_gd) = res, ref
    assert np.allclose(ld, o_ld, rtol=t["ld"], atol=t["ld"])
    assert np.max(np.abs(gd - o_gd)) <= t["g"] * max(1.0, np.abs(o_gd).max())


@pytest.mark.parametrize("prec", ["3xtf32", "bf16x3"])
def test_40x40_sampled_blocks(prec):
    wl = inputs.WORKLOADS["ionic_40x40"]
    p = api.Params(wl.L, wl.n_omega, U=wl.U, T=wl.T, delta=wl.delta, t=wl.t, mu=wl.mu, prec=prec)
    phi = inputs.seed_phi(wl.seed, p.N)
    sample = [0, 1, 11, 12, 13, 128, 255]
    ref = oracle.blocks_sample(oparams(p), phi, sample)
    with api.Context(p) as c:
        (ld, gd), kinds = ran(c, lambda: c.blocks(phi))
        assert "nest_up" in kinds and "update" not in kinds
        check((ld[sample], gd[sample]), ref, tol(prec, dense=False))
        c.set_pivoting("partial")
        assert c.sm_partition()[0] > 0
        (ld, gd), kinds = ran(c, lambda: c.blocks(phi))
        assert {"panel", "update", "update_cross", "diag", "prep_piv", "refine"} <= kinds
        assert "nest_up" not in kinds
        check((ld[sample], gd[sample]), ref, tol(prec))


@pytest.mark.parametrize("prec", ["bf16x3", "fp32"])
def test_64x64_staggered_field_closed_form(prec):
    from test_oracle_pins import G_staggered, ld_staggered, sublattice
    wl = inputs.WORKLOADS["ionic_64x64"]
    p = api.Params(wl.L, wl.n_omega, U=wl.U, T=wl.T, delta=wl.delta, prec=prec)
    a, L, N = 0.8, wl.L, wl.L * wl.L
    s = sublattice(L)
    om_ref, g_a = N * a * a / wl.U, 2 * a / wl.U
    for n in range(wl.n_omega):
        w = (2 * n + 1) * math.pi * wl.T
        for sg in (1, -1):
            D = wl.delta + sg * a
            om_ref -= 2 * wl.T * ld_staggered(L, D, w)
            g_a -= 2 * wl.T * sg * G_staggered(L, D, w, -D).real
    with api.Context(p) as c:
        for mode in ("auto", "partial"):
            c.set_pivoting(mode)
            (om, g), kinds = ran(c, lambda: c.grad(a * s))
            assert ("nest_up" in kinds) == (mode == "auto") and ("panel" in kinds) == (mode == "partial")
            t = tol(prec, dense=mode == "partial")
            assert om == pytest.approx(om_ref, rel=t["om"])
            assert np.max(np.abs(g - g_a * s)) <= t["g"] * max(1.0, abs(g_a)) * 10


@pytest.mark.parametrize("mode", ["dominant", "both", "alternate"])
def test_sm_partition_leaves_results_unchanged(mode):
    p = api.Params(20, 8, U=6.0, T=0.1, delta=0.5, prec="bf16x3")
    phi = inputs.seed_phi(3, p.N)
    with api.Context(p) as c:
        c.set_pivoting("partial")
        (om0, g0), kinds = ran(c, lambda: c.grad(phi))
        assert "update" in kinds and "nest_up" not in kinds
        ps, ds = c.set_sm_partition(16, mode)
        assert ps >= 16 and ds > 0
        om1, g1 = c.grad(phi)
        assert c.set_sm_partition(0) == (0, 0)
        om2, g2 = c.grad(phi)
    assert om1 == om0 and om2 == om0
    assert np.array_equal(g1, g0) and np.array_equal(g2, g0)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "3xtf32", "bf16x3"])
@pytest.mark.parametrize("L", [12, 20])
def test_pivot_free_blocks_match_forced_pivoting(L, prec, monkeypatch):
    """6 pivoted and 14 dominant blocks; forcing the pivoted panel on all of them."""
    p = api.Params(L, 10, U=4.0, T=0.2, delta=0.6, prec=prec)
    assert api.pivoted_blocks(p) == 6
    phi = inputs.random_phi(33, p.N)
    ref = oracle.blocks_sample(oparams(p), phi, list(range(2 * p.n_omega)))
    with api.Context(p) as c:
        c.set_pivoting("partial")
        a, kinds = ran(c, lambda: c.blocks(phi))
        assert "nest_up" not in kinds and "panel" in kinds and "span_dominant" in kinds
    monkeypatch.setenv("SCA_PIVOT_ALL", "1")
    with api.Context(p) as c:
        b, kinds = ran(c, lambda: c.blocks(phi))
        assert "nest_up" not in kinds and "span_dominant" not in kinds
    check(a, ref, tol(prec))
    check(b, ref, tol(prec))
    check(a, b, tol(prec))


@pytest.mark.parametrize("L,prec", [(14, "fp64"), (14, "fp32"), (20, "3xtf32"), (20, "bf16x3")])
def test_resident_inverses(L, prec):
    """Forward and backward in two calls, the potential alone, and Adam steps."""
    torch = pytest.importorskip("torch")
    p = api.Params(L, 8, U=4.0, T=0.1, delta=0.4, prec=prec)
    phi = inputs.random_phi(L, p.N, 1.0)
    o_om, o_g, _, _ = oracle.omega_grad(oparams(p), phi, per_block=True)
    t = tol(prec)
    with api.Context(p) as c:
        c.set_pivoting("partial")
        (om, g), kinds = ran(c, lambda: c.grad(phi))
        assert "nest_up" not in kinds
        assert om == pytest.approx(o_om, rel=t["om"])
        assert np.max(np.abs(g - o_g)) <= t["g"] * max(1.0, np.abs(o_g).max()) * 10
        assert c.potential(phi) == pytest.approx(om, rel=t["om"])
        x = torch.tensor(phi, dtype=torch.float64, device="cuda")
        om_t, g_t = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(x)
        c.forward_dev(x, om_t)
        c.backward_dev(x, g_t)
        torch.cuda.synchronize()
        assert float(om_t) == om and np.allclose(g_t.cpu().numpy(), g, rtol=1e-12, atol=1e-14)
        c.adam_init(api.AdamConfig(lr=0.01), phi)
        c.adam_step(1)
        assert np.allclose(c.get_state()["m"], 0.1 * g, rtol=1e-9, atol=1e-12)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "3xtf32", "bf16x3"])
@pytest.mark.parametrize("L,eta", [(10, 0.2), (20, 0.15), (20, 4.5)])
def test_density_of_states(L, eta, prec):
    """Pivoted and, for eta > 4|t|, dominant resolvents; then the default's."""
    p = api.Params(L, 4, U=4.0, T=0.1, delta=0.6, mu=0.1, prec=prec)
    phi, ee = inputs.random_phi(30 + L, p.N, 1.2), inputs.random_phi(40 + L, p.N, 0.4)
    w = np.linspace(-5.5, 5.5, 7)
    op = oparams(p)
    ref = np.stack([oracle.dos(op, phi, s, w, eta, eps_extra=ee) for s in (1, -1)])
    with api.Context(p) as c:
        c.set_site_energy(ee)
        for mode in ("partial", "auto"):
            c.set_pivoting(mode)
            rho, kinds = ran(c, lambda: c.dos(phi, w, eta))
            assert ("nest_up" in kinds) == (mode == "auto")
            t = 1e-10 if prec == "fp64" or mode == "auto" else 2e-5
            assert np.max(np.abs(rho - ref)) <= t * np.abs(ref).max()


@pytest.mark.parametrize("L,prec", [(6, "fp32"), (8, "fp64"), (12, "3xtf32")])
def test_fused_kernel_matches_the_blocked_path(L, prec, monkeypatch):
    """Below the temperature line, where the fused kernel runs from 6 x 6 sites up."""
    p = api.Params(L, 6, U=4.0, T=0.008, delta=0.4, prec=prec)
    ad = api.AdamConfig(lr=0.01, seed=11)
    out = {}
    for fused in ("1", "0"):
        monkeypatch.setenv("SCA_FUSED", fused)
        with api.Context(p) as c:
            c.adam_init(ad)
            (om, gm), kinds = ran(c, lambda: c.adam_step(12))
            out[fused] = c.phi()
        assert ("fused" in kinds) == (fused == "1") and "nest_up" not in kinds
    t = 1e-10 if prec == "fp64" else 1e-6
    assert np.max(np.abs(out["1"] - out["0"])) < t


def test_dense_then_nested_then_dense_on_one_workspace():
    """The two share memory: alternating leaves each with its own bits."""
    for L, prec in ((8, "fp32"), (14, "fp64"), (20, "bf16x3")):
        p = api.Params(L, 5, U=4.0, T=0.1, delta=0.4, prec=prec)
        phi = inputs.random_phi(L, p.N, 1.0)
        with api.Context(p) as c:
            res = []
            for mode in ("partial", "auto", "partial", "none", "partial"):
                c.set_pivoting(mode)
                res.append(c.blocks(phi))
        for k in (2, 4):
            assert np.array_equal(res[0][0], res[k][0]) and np.array_equal(res[0][1], res[k][1])
        assert np.array_equal(res[1][1], res[3][1]) and not np.array_equal(res[0][1], res[1][1])
