"""Accuracy of the default elimination on clean and staggered lattices at small Im z, where parts
of the lattice cut out by separators have levels at the energy itself.

Exact values in closed form: with A = z + d S + t K (S the checkerboard signs, K the adjacency of
the torus, S K = -K S), A^{-1} = (z - d S - t K) / (z^2 - d^2 - t^2 K^2), so
G_ii = (z - d s_i) g, g the mean over k of 1 / (z^2 - d^2 - e_k^2), ln|det A| = 1/2 sum_k
ln|z^2 - d^2 - e_k^2|.

Tolerances: rounding grows like (|t| / Im z)^4 in units of the arithmetic that a block takes.
Float64 contexts: sums of three float32 (2^-70) below Im z = 0.5 |t|, (1 / 0.03)^4 2^-70 = 1e-15;
float64 above, 16 units of 2^-53; a few such sums: 1e-14 of the largest |G|.  The others: the same
below 0.3 (from 12 x 12 sites up 0.15), double-float above, (1 / 0.15)^4 2^-48 = 7e-12: 1e-11.
"""
import numpy as np
import pytest

from paper_2311_04435_gb300 import api, inputs

pytestmark = pytest.mark.gpu

ld = np.longdouble


def signs(L):
    x, y = np.meshgrid(np.arange(L), np.arange(L), indexing="ij")
    return np.where((x + y) % 2 == 0, 1.0, -1.0).reshape(-1)


def exact(L, z, d):
    """diag(G) and ln|det A| for t = 1, site terms z + d s_i."""
    k = 2 * ld(np.pi) * np.arange(L) / L
    e = (2 * (np.cos(k)[:, None] + np.cos(k)[None, :])).reshape(-1)
    den = np.clongdouble(z) ** 2 - ld(d) ** 2 - e ** 2
    return (z - d * signs(L)) * np.mean(1 / den), np.sum(np.log(np.abs(den))) / 2


# pi T on both sides of every line of the rule; Im z / |t| = 0.0301 to 0.6
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16x3"])
@pytest.mark.parametrize("L", [6, 8, 12, 14])
def test_weak_fields_at_small_frequencies(L, prec):
    tol = 1e-14 if prec == "fp64" else 1e-11
    for w0 in (0.0301, 0.05, 0.07, 0.11, 0.157, 0.25, 0.314, 0.6):
        for mu, d in ((0.0, 0.0), (0.01, 0.0), (0.2, 0.05)):
            p = api.Params(L, 2, U=4.0, T=w0 / np.pi, delta=0.0, mu=mu, prec=prec)
            with api.Context(p) as c:
                lds, gd = c.blocks(d * signs(L))
                om, g = c.grad(d * signs(L))
                assert c.potential(d * signs(L)) == om
            for b in range(4):
                sg = -1 if b & 1 else 1
                w = (2 * (b >> 1) + 1) * np.pi * p.T
                G, l0 = exact(L, mu + 1j * w, sg * d)
                scale = np.abs(G).max()
                assert np.max(np.abs(gd[b] - sg * G.real)) <= tol * scale, (w, mu, d)
                assert abs(lds[b] - l0) <= 1e2 * tol, (w, mu, d)


@pytest.mark.parametrize("L", [6, 8, 20])
def test_density_of_states_of_the_clean_lattice(L):
    """Float64, small broadening, energies on the pieces' levels (0, 1) and off them; batches of
    64 blocks, on the small lattices more than fit at once."""
    p = api.Params(L, 32, U=4.0, T=0.2, delta=0.0, prec="fp64")
    w = np.concatenate([[0.0, 1.0, 2.0], np.linspace(-4.2, 4.2, 41)])
    with api.Context(p) as c:
        for eta in (0.0301, 0.05, 0.2, 0.6):
            rho = c.dos(np.zeros(p.N), w, eta)
            ref = np.array([-float(np.mean(exact(L, x + 1j * eta, 0.0)[0]).imag) / np.pi for x in w])
            assert np.max(np.abs(rho - ref)) <= 2e-14 * ref.max(), eta


@pytest.mark.parametrize("L,prec,T", [(6, "fp64", 0.02), (8, "fp64", 0.012), (14, "fp64", 0.05),
                                      (8, "fp32", 0.0115), (20, "bf16x3", 0.015)])
def test_mixed_arithmetic_forward_backward_and_passes(L, prec, T, monkeypatch):
    """Blocks of two arithmetics in one evaluation: the split forward / backward, a
    repeat, and passes of one and three blocks give the gradient to the bit."""
    torch = pytest.importorskip("torch")
    p = api.Params(L, 9, U=4.0, T=T, delta=0.1, prec=prec)
    phi = inputs.random_phi(L, p.N, 0.3)
    with api.Context(p) as c:
        om, g = c.grad(phi)
        x = torch.tensor(phi, dtype=torch.float64, device="cuda")
        om_t, g_t = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(x)
        c.forward_dev(x, om_t)
        c.backward_dev(x, g_t)
        torch.cuda.synchronize()
        assert float(om_t) == om and np.array_equal(g_t.cpu().numpy(), g)
        again = c.grad(phi)
        assert again[0] == om and np.array_equal(again[1], g)
    for resident in ("1", "3"):
        monkeypatch.setenv("SCA_MAX_BLOCKS_RESIDENT", resident)
        with api.Context(p) as c:
            om3, g3 = c.grad(phi)
        assert om3 == om and np.array_equal(g3, g)


@pytest.mark.parametrize("prec", ["fp64", "bf16x3"])
def test_served_requests_in_mixed_arithmetic(prec):
    """Requests of one size bucket whose blocks take different arithmetics share passes and give
    what each gives alone."""
    reqs = [(api.Params(16, 5, U=4.0, T=T, delta=0.3, prec=prec),
             api.AdamConfig(lr=0.01, grad_tol=1e-9, max_steps=5, seed=60 + k))
            for k, T in enumerate((0.2, 0.012, 0.05, 0.03, 0.006))]
    alone = [api.solve(p, a) for p, a in reqs]
    with api.Server(hbm_budget_bytes=16 << 30, max_slots=5, manual=True) as srv:
        ids = [srv.submit(p, a) for p, a in reqs]
        now = 0.0
        while any(srv.step(now)):
            now += 0.1
        mixed = [srv.poll(rid, 256) for rid in ids]
    for x, y in zip(alone, mixed):
        assert x.steps == y.steps and x.omega == y.omega and np.array_equal(x.phi, y.phi)


def test_more_blocks_than_sms_with_wider_ones():
    """A launch per level for the float64 blocks beside the wider ones: the first blocks
    equal those of a small pass, all are near the closed form."""
    p = api.Params(10, 80, U=4.0, T=0.05, delta=0.0, prec="fp64")
    phi = 0.02 * signs(10)
    with api.Context(p) as c:
        lds, gd = c.blocks(phi)
    with api.Context(api.Params(10, 6, U=4.0, T=0.05, delta=0.0, prec="fp64")) as c:
        few = c.blocks(phi)
    assert np.array_equal(lds[:12], few[0]) and np.array_equal(gd[:12], few[1])
    for b in range(0, 160, 7):
        sg = -1 if b & 1 else 1
        G, l0 = exact(10, 1j * (2 * (b >> 1) + 1) * np.pi * p.T, sg * 0.02)
        assert np.max(np.abs(gd[b] - sg * G.real)) <= 1e-14 * np.abs(G).max()


@pytest.mark.parametrize("L", [6, 12])
def test_entries_beyond_float32(L):
    """A float64 context's wider blocks with a site term of 1e100 in one block of each pair: its
    site decouples (G = 1 / a), the rest is the lattice without it; the other spin's blocks too."""
    torch = pytest.importorskip("torch")
    p = api.Params(L, 3, U=4.0, T=0.02, delta=0.0, mu=0.1, prec="fp64")
    phi = inputs.random_phi(L, p.N, 0.4)
    phi[5] = 1e100
    with api.Context(p) as c:
        lds, gd = c.blocks(phi)
        om, g = c.grad(phi)
        x = torch.tensor(phi, dtype=torch.float64, device="cuda")
        om_t, g_t = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty_like(x)
        c.forward_dev(x, om_t)
        c.backward_dev(x, g_t)
        torch.cuda.synchronize()
        assert float(om_t) == om and np.array_equal(g_t.cpu().numpy(), g)
        c.set_pivoting("partial")
        lds_d, gd_d = c.blocks(phi)
    # the dense elimination loses nothing here: a few hundred 2^-53 of |G| <= 1 / omega_0
    assert np.max(np.abs(gd - gd_d)) <= 1e-12 and np.max(np.abs(lds - lds_d)) <= 1e-12 * 400
