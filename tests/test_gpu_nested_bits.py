"""The nested elimination's results are the same to the bit however its work is split: a CTA or a
cluster per block, or a launch per level; alone or beside other requests of a size bucket."""
import numpy as np
import pytest

from paper_2311_04435_gb300 import api, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("L", [6, 10, 16])
def test_blocks_do_not_depend_on_their_number(L, prec):
    """160 and 152 blocks (a launch per level, a CTA per block) against 80, 40, 12 and 2 (clusters
    of 1, 2, 8 and 8)."""
    phi = inputs.random_phi(500 + L, L * L, 0.5)
    res = {}
    for nw in (80, 76, 40, 20, 6, 1):
        p = api.Params(L, nw, U=4.0, T=0.2, delta=0.3, t=1.2, prec=prec)
        with api.Context(p) as c:
            res[nw] = c.blocks(phi)
    for nw in (76, 40, 20, 6, 1):
        assert np.array_equal(res[80][0][:2 * nw], res[nw][0]), nw
        assert np.array_equal(res[80][1][:2 * nw], res[nw][1]), nw


@pytest.mark.parametrize("prec", ["fp64", "3xtf32"])
def test_served_requests_equal_the_same_alone(prec):
    reqs = [(api.Params(16, nw, U=4.0, T=0.25, delta=0.3, prec=prec),
             api.AdamConfig(lr=0.01, grad_tol=1e-9, max_steps=5, seed=60 + k))
            for k, nw in enumerate((5, 12, 40, 3))]
    alone = [api.solve(p, a) for p, a in reqs]
    with api.Server(hbm_budget_bytes=16 << 30, max_slots=4, manual=True) as srv:
        ids = [srv.submit(p, a) for p, a in reqs]
        now = 0.0
        while any(srv.step(now)):
            now += 0.1
        mixed = [srv.poll(rid, 256) for rid in ids]
    for x, y in zip(alone, mixed):
        assert x.steps == y.steps and x.omega == y.omega and np.array_equal(x.phi, y.phi)


@pytest.mark.parametrize("L,nw,T,prec", [(14, 20, 0.05, "fp64"), (14, 100, 0.05, "fp64"),
                                         (8, 90, 0.03, "fp32"), (20, 30, 0.1, "bf16x3")])
def test_captured_gradient_replays_to_the_bit(L, nw, T, prec):
    """Blocks of one and two arithmetics, one launch or one per level: every stream that an
    evaluation uses forks from the caller's and joins it again."""
    torch = pytest.importorskip("torch")
    p = api.Params(L, nw, U=4.0, T=T, delta=0.3, prec=prec)
    fields = [inputs.random_phi(7 + k, p.N, 0.4) for k in range(2)]
    with api.Context(p) as c:
        want = [c.grad(f) for f in fields]
        x = torch.tensor(fields[0], dtype=torch.float64, device="cuda")
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            c.grad_dev(x)
            s.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                om, g = c.grad_dev(x)
            for f, (om_ref, g_ref) in zip(fields, want):
                x.copy_(torch.tensor(f, dtype=torch.float64))
                graph.replay()
                s.synchronize()
                assert float(om) == om_ref and np.array_equal(g.cpu().numpy(), g_ref)
