"""The calls that the framework's users make, at the sizes they make them, for timing.

Kinds of call (paper_2311_04435_gb300.api):
  adam        Context.adam_init from a start field, adam_step(steps), phi and moments read back
  grad        Context.grad: Omega and its gradient from a host field
  potential   Context.potential: Omega alone (elimination without the inverse)
  autograd    sca_potential(phi, ctx) on a CUDA tensor and .backward()
  dos         Context.dos: the density of states of both spins on a frequency grid
  metropolis  a Metropolis chain on exp(-Omega/T)
  serve       a batch of solve requests of mixed sizes through a Server

Sizes are those of inputs.WORKLOADS, of the serving trace (inputs.serving_trace) and of the GPU
tests; temperatures 0.05..0.6, U 2..8, Delta 0..2 as in the serving trace.
"""
import math

import numpy as np
import torch

from paper_2311_04435_gb300 import api, inputs


def _nw(T):
    """Frequencies of a served request at temperature T (cut-off omega = 20)."""
    return int(math.ceil(20.0 / (2.0 * math.pi * T)))


def _case(kind, L, n_omega, prec, U, T, delta, **kw):
    c = dict(kind=kind, L=L, n_omega=n_omega, prec=prec, U=U, T=T, delta=delta, mu=0.0,
             ionic="paper", disorder=0.0, steps=1, n_w=0, eta=0.0)
    c.update(kw)
    return c


def listed():
    return [
        # the paper-size Hubbard plaquette in float64, 20 of its 2000 Adam steps: latency
        _case("adam", 4, 64, "fp64", 6.0, 0.1, 0.0, steps=20, name="adam_4x4_fp64"),
        # the middle size of the small served requests, a batch of Adam steps in one call
        _case("adam", 12, 32, "bf16x3", 4.0, 0.1, 1.0, steps=8, name="adam_12x12_bf16x3"),
        # a small disordered lattice off half filling (Delta/2 convention), ragged 196-row blocks
        _case("grad", 14, 32, "fp32", 3.0, 0.1, 0.9, mu=0.2, ionic="half", disorder=0.5,
              name="grad_14x14_fp32_disorder"),
        # sampling the static field: Omega evaluations one after another, float64
        _case("metropolis", 10, 32, "fp64", 4.0, 0.2, 0.6, steps=8, name="metropolis_10x10_fp64"),
        # the 20x20 ionic workload (512 blocks), the paper's lattice, two Adam steps
        _case("adam", 20, 256, "bf16x3", 6.0, 0.1, 0.5, steps=2, name="adam_20x20_bf16x3"),
        # the same workload's gradient on the plain float64 path
        _case("grad", 20, 256, "fp64", 6.0, 0.1, 0.5, name="grad_20x20_fp64"),
        # spectral function of the 20x20 lattice: 64 energies, both spins, small broadening
        _case("dos", 20, 64, "3xtf32", 6.0, 0.1, 0.5, n_w=64, eta=0.05, name="dos_20x20_3xtf32"),
        # a differentiable Omega inside a PyTorch program, the largest served lattice
        _case("autograd", 32, 64, "3xtf32", 5.0, 0.05, 0.3, name="autograd_32x32_3xtf32"),
        # the benchmark: one SCA+Adam step of the 40x40 ionic workload (256 blocks)
        _case("adam", 40, 128, "bf16x3", 4.0, 0.1, 1.0, name="adam_40x40_bf16x3"),
        # Omega alone on that workload, as a line search or a comparison of minima takes it
        _case("potential", 40, 128, "bf16x3", 4.0, 0.1, 1.0, name="potential_40x40_bf16x3"),
        # serving: requests of every size of the trace at once, eight updates each
        _case("serve", 32, 0, "bf16x3", 0.0, 0.0, 0.0, steps=8, requests=12,
              sizes="8,12,16,20,24,32", name="serve_mix_bf16x3"),
        # the largest single instance: one step of the 64x64 workload (128 blocks)
        _case("adam", 64, 64, "bf16x3", 6.0, 0.2, 0.5, name="adam_64x64_bf16x3"),
    ]


def _even_log(rng, lo, hi):
    return max(lo, min(hi, 2 * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2))))


def draw(rng):
    kind = rng.choice(["adam", "adam", "grad", "grad", "potential", "autograd", "dos",
                       "metropolis", "serve"])
    prec = rng.choice(["fp64", "fp32", "3xtf32", "bf16x3", "bf16x3"])
    if kind == "metropolis":
        prec = "fp64"
    T = math.exp(rng.uniform(math.log(0.05), math.log(0.6)))
    if kind == "serve":
        sizes = sorted({_even_log(rng, 6, 32) for _ in range(4)})
        return _case("serve", sizes[-1], 0, "bf16x3", 0.0, 0.0, 0.0, steps=8,
                     requests=rng.randint(3, 12), sizes=",".join(str(s) for s in sizes))
    L = _even_log(rng, 4, {"fp64": 24, "fp32": 40, "3xtf32": 48, "bf16x3": 64}[prec])
    steps = rng.randint(1, 8) if kind in ("adam", "metropolis") else 1
    # dense multiply-adds a drawn case may stand for: below the largest listed case of its type
    cap = {"fp64": 2.5e11, "fp32": 4e12, "3xtf32": 1.5e13, "bf16x3": 4e13}[prec]
    per_block = 8.0 * (L * L) ** 3 * steps
    n_omega = max(1, min(int(rng.choice([1.0, 1.0, 2.0]) * _nw(T)) + rng.randint(0, 3),
                         int(cap / (2 * per_block))))
    if 2 * n_omega * per_block > cap:
        steps = 1
    c = _case(kind, L, n_omega, prec, rng.uniform(2.0, 8.0), T, rng.uniform(0.0, 2.0), steps=steps,
              mu=rng.choice([0.0, 0.0, rng.uniform(-0.5, 0.5)]),
              ionic=rng.choice(["paper", "paper", "half"]),
              disorder=rng.choice([0.0, 0.0, rng.uniform(0.1, 1.0)]))
    if kind == "dos":
        c["n_w"] = rng.randint(max(1, n_omega // 2), n_omega)
        c["eta"] = math.exp(rng.uniform(math.log(0.05), math.log(0.3)))
    return c


# ------------------------------------------------------------------ inputs

def _params(c):
    return api.Params(c["L"], c["n_omega"], U=c["U"], T=c["T"], delta=c["delta"], mu=c["mu"],
                      prec=c["prec"], ionic=c["ionic"])


def _start(c, seed):
    """The random start of an Adam run for training calls; a staggered order with noise, as late
    in a run, for single evaluations."""
    rng = np.random.default_rng([seed, 1])
    N = c["L"] ** 2
    if c["kind"] == "adam":
        return rng.uniform(-0.5, 0.5, N)
    return inputs.neel_phi(c["L"], rng.uniform(0.4, 1.6)) + rng.uniform(-0.3, 0.3, N)


def _disorder(c, seed):
    if not c["disorder"]:
        return None
    return np.random.default_rng([seed, 2]).uniform(-c["disorder"], c["disorder"], c["L"] ** 2)


def _grid(c, seed):
    half = np.random.default_rng([seed, 3]).uniform(4.0, 6.0)
    return np.linspace(-half, half, c["n_w"])


def _requests(c, seed):
    rng = np.random.default_rng([seed, 4])
    sizes = [int(s) for s in c["sizes"].split(",")]
    out = []
    for k in range(c["requests"]):
        T = float(rng.uniform(0.05, 0.6))
        out.append((api.Params(sizes[k % len(sizes)], _nw(T), U=float(rng.uniform(2.0, 8.0)), T=T,
                               delta=float(rng.uniform(0.0, 2.0)), prec=c["prec"]),
                    api.AdamConfig(lr=0.01, grad_tol=1e-6, max_steps=c["steps"],
                                   seed=int(rng.integers(1, 2 ** 31)))))
    return out


def prepare(case, seed):
    st = {"case": case}
    if case["kind"] == "serve":
        # the HBM budget and slots of the benchmark's serving sweep
        st["server"] = api.Server(hbm_budget_bytes=120 << 30, max_slots=64, manual=True)
        st["requests"] = _requests(case, seed)
        st["now"] = 0.0
        return st
    ctx = api.Context(_params(case))
    ee = _disorder(case, seed)
    if ee is not None:
        ctx.set_site_energy(ee)
    st["ctx"] = ctx
    st["phi"] = _start(case, seed)
    if case["kind"] == "autograd":
        st["phi"] = torch.tensor(st["phi"], dtype=torch.float64, device="cuda")
    if case["kind"] == "dos":
        st["w"] = _grid(case, seed)
    if case["kind"] == "metropolis":
        st["chain_seed"] = seed
    return st


def _kept(x, c):
    """Omega and the density of states in the precision that the path promises: 1e-5 relative in
    the reduced precisions, so float32 holds them; float64 on the float64 path."""
    return x if c["prec"] == "fp64" else x.float()


_CHAIN_DELTA = 0.02  # proposal width of the Metropolis chains


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "serve":
        srv = state["server"]
        ids = [(srv.submit(p, a), p.N) for p, a in state["requests"]]
        while True:
            state["now"] += 0.05
            in_flight, queued = srv.step(state["now"])
            if in_flight == 0 and queued == 0:
                break
        out = [srv.poll(rid, N) for rid, N in ids]
        return [{"phi": r.phi, "omega": r.omega, "steps": r.steps, "gmax": r.gmax} for r in out]
    ctx = state["ctx"]
    if kind == "adam":
        ctx.adam_init(api.AdamConfig(lr=0.01), state["phi"])
        omega, gmax = ctx.adam_step(c["steps"])
        s = ctx.get_state()
        return {"omega": omega, "gmax": gmax, "phi": s["phi"], "m": s["m"], "v": s["v"]}
    if kind == "grad":
        omega, g = ctx.grad(state["phi"])
        return {"omega": omega, "grad": g}
    if kind == "potential":
        return {"omega": ctx.potential(state["phi"])}
    if kind == "autograd":
        x = state["phi"].detach().requires_grad_(True)
        omega = api.sca_potential(x, ctx)
        omega.backward()
        return {"omega": _kept(omega.detach(), c), "grad": x.grad}
    if kind == "dos":
        rho = torch.from_numpy(ctx.dos(state["phi"], state["w"], c["eta"]))
        return {"rho": _kept(rho, c)}
    if kind == "metropolis":
        ctx.metropolis_init(_CHAIN_DELTA, seed=state["chain_seed"], phi0=state["phi"])
        trace, accepted, omega, total = ctx.metropolis_step(c["steps"])
        return {"trace": trace, "accepted": accepted, "omega": omega, "total": total,
                "phi": ctx.phi()}
    raise ValueError(kind)


# -------------------------------------------------------------------- work

def _resolvent_flops(L, gradient):
    """Real operations that one complex-symmetric L x L periodic lattice cannot do without: the
    last separator of a torus holds about 2L sites, whose dense symmetric factorisation takes
    (2L)^3/6 complex multiply-adds (8 operations each), its inverse three times that."""
    return 8.0 * (2.0 * L) ** 3 / (2.0 if gradient else 6.0)


def work(case):
    kind, L = case["kind"], case["L"]
    N = L * L
    if kind == "serve":  # fields out; omegas and norms are noise beside them
        flops = bytes_ = 0.0
        for p, a in _requests(case, 0):
            flops += 2 * p.n_omega * _resolvent_flops(p.L, True) * (a.max_steps + 1)
            bytes_ += 8.0 * p.N + 24.0
        return {"bytes": bytes_, "flops": flops}
    blocks = 2 * (case["n_w"] if kind == "dos" else case["n_omega"])
    evals = case["steps"] + (1 if kind == "metropolis" else 0)
    flops = blocks * evals * _resolvent_flops(L, kind not in ("potential", "metropolis"))
    vectors = {"adam": 4, "grad": 2, "potential": 1, "autograd": 2, "dos": 1, "metropolis": 2}[kind]
    bytes_ = 8.0 * (vectors * N + 3 * case["n_w"] + 2 * case["steps"])
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------- exact
# H_sigma is real symmetric, so one diagonalisation per spin gives every frequency:
# ln|det A_n| = 1/2 sum_a ln(w_n^2 + (mu - e_a)^2), Re G_n,ii = sum_a V_ia^2 (mu - e_a) /
# (w_n^2 + (mu - e_a)^2).

def _hopping(L):
    K = np.zeros((L * L, L * L))
    for x in range(L):
        for y in range(L):
            i = x * L + y
            for j in (((x + 1) % L) * L + y, x * L + (y + 1) % L):
                K[i, j] -= 1.0
                K[j, i] -= 1.0
    return K


def _site_signs(L):
    x, y = np.meshgrid(np.arange(L), np.arange(L), indexing="ij")
    return np.where((x + y) % 2 == 0, 1.0, -1.0).reshape(-1)


class _Exact:
    def __init__(self, L, n_omega, U, T, delta, mu=0.0, ionic="paper", ee=None):
        self.L, self.U, self.T, self.mu = L, U, T, mu
        self.w2 = ((2 * np.arange(n_omega) + 1) * math.pi * T) ** 2
        self.K = _hopping(L)
        self.eps = -_site_signs(L) * (0.5 * delta if ionic == "half" else delta)
        if ee is not None:
            self.eps = self.eps + ee

    def evaluate(self, phi, gradient=True):
        omega = float(np.sum(phi * phi)) / self.U
        g = 2.0 * phi / self.U
        for sg in (1, -1):
            H = self.K + np.diag(self.eps - sg * phi)
            if gradient:
                e, V = np.linalg.eigh(H)
            else:
                e, V = np.linalg.eigvalsh(H), None
            d = self.mu - e
            den = self.w2[:, None] + d[None, :] ** 2
            omega -= self.T * float(np.sum(np.log(den)))
            if gradient:
                g = g - 2.0 * self.T * sg * ((V * V) @ (d * np.sum(1.0 / den, axis=0)))
        return omega, g

    def adam(self, phi, lr, steps):
        phi = phi.copy()
        m, v = np.zeros_like(phi), np.zeros_like(phi)
        omega = gmax = 0.0
        for k in range(1, steps + 1):
            omega, g = self.evaluate(phi)
            gmax = float(np.max(np.abs(g)))
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            phi = phi - (lr / (1 - 0.9 ** k)) * m / (np.sqrt(v) / math.sqrt(1 - 0.999 ** k) + 1e-8)
        return omega, gmax, phi, m, v


def exact(case, seed):
    kind, L = case["kind"], case["L"]
    if kind == "metropolis":  # a chain of decisions
        return None
    if kind == "serve":
        out = []
        for p, a in _requests(case, seed):
            ex = _Exact(p.L, p.n_omega, p.U, p.T, p.delta)
            phi = ex.adam(inputs.seed_phi(a.seed, p.N), a.lr, a.max_steps)[2]
            omega, g = ex.evaluate(phi)
            out.append({"phi": phi, "omega": omega, "steps": None,
                        "gmax": float(np.max(np.abs(g)))})
        return out
    ex = _Exact(L, case["n_omega"], case["U"], case["T"], case["delta"], case["mu"],
                case["ionic"], _disorder(case, seed))
    phi = _start(case, seed)
    if kind == "adam":
        if case["steps"] * (L / 40.0) ** 6 > 40.0:  # over about 12 s of diagonalisations
            return None
        omega, gmax, phi, m, v = ex.adam(phi, 0.01, case["steps"])
        return {"omega": omega, "gmax": gmax, "phi": phi, "m": m, "v": v}
    if kind == "grad":
        omega, g = ex.evaluate(phi)
        return {"omega": omega, "grad": g}
    if kind == "potential":
        return {"omega": ex.evaluate(phi, gradient=False)[0]}
    if kind == "autograd":
        omega, g = ex.evaluate(phi)
        return {"omega": torch.tensor(omega, dtype=torch.float64, device="cuda"),
                "grad": torch.tensor(g, dtype=torch.float64, device="cuda")}
    if kind == "dos":
        w = _grid(case, seed)
        rho = []
        for sg in (1, -1):
            e = np.linalg.eigvalsh(ex.K + np.diag(ex.eps - sg * phi))
            d = w[:, None] + case["mu"] - e[None, :]
            rho.append(np.sum(case["eta"] / (d * d + case["eta"] ** 2), axis=1) / (math.pi * L * L))
        return {"rho": torch.from_numpy(np.stack(rho))}
    return None
