"""Performance cases of the OrderMoE library: what a user's program has it do, at the sizes of this
repository's workloads (synth.WORKLOADS), tests and benchmark, and odd sizes between them.

Six kinds of call:
  layer      one MoE layer over T tokens (router, selection, permutation, SwiGLU FFN, combine), by
             the steps of layer.MoELayer or by the one call ordermoe_layer_forward
  stack      L layers on the residual map (layer.LayerStack), eager or replayed as a CUDA graph
  select     routing and server-expert selection with the look-ahead horizon H
  plan       the whole offline plan (ordermoe_plan)
  calibrate  similarity, counts and transitions of a calibration set, the logits kept
  batches    a queue of batches from and to pinned host memory (ordermoe_layer_forward_batches)
"""
import math

import numpy as np
import torch

from paper_2607_17154_gb300 import binding as B
from paper_2607_17154_gb300 import synth
from paper_2607_17154_gb300.layer import LayerStack, MoELayer, build_tables

DEV = "cuda:0"

# layer shapes of synth.WORKLOADS (d, experts, routed, d_ff, servers, clusters, budget, homes)
TINY = dict(d=256, E=8, k=2, dff=512, M=4, K=2, qbar=0.05, home="uniform")
WIDE = dict(d=4096, E=8, k=2, dff=14336, M=4, K=4, qbar=0.05, home="uniform")
FINE = dict(d=2048, E=64, k=6, dff=1408, M=8, K=8, qbar=0.10, home="zipf1.1")


def listed():
    return [
        # the smallest layer: a few launches' latency
        dict(name="tiny_layer", kind="layer", T=64, call=True, **TINY),
        # a decode step of a batch of 128 on 8 wide experts, the default horizon, one graph a step
        dict(name="decode_wide", kind="stack", L=4, T=128, H=3, graph=True, **dict(WIDE, qbar=0.5)),
        # a small ragged decode batch on 64 narrow experts, launched from the host
        dict(name="decode_fine", kind="stack", L=4, T=33, H=1, graph=False, **dict(FINE, qbar=0.5)),
        # a chunk of a prompt on the wide layer (about 127 rows an expert)
        dict(name="chunk_wide", kind="layer", T=509, call=True, **WIDE),
        # a full prefill batch on the wide layer (the benchmark's default)
        dict(name="prefill_wide", kind="layer", T=4096, call=False, **WIDE),
        # a chunk of a prompt on the 64-expert layer (about 96 rows an expert)
        dict(name="chunk_fine", kind="layer", T=1021, call=True, **FINE),
        # a full prefill batch on the 64-expert layer
        dict(name="prefill_fine", kind="layer", T=8192, call=False, **FINE),
        # decisions of a prompt's tokens on the 64-expert layer with the default horizon
        dict(name="select_fine", kind="select", T=2048, d=2048, E=64, k=6, M=8, K=8, qbar=0.5, H=3,
             home="zipf1.1"),
        # the offline plan of 24 layers of 64 experts over the full calibration set
        dict(name="plan_full", kind="plan", L=24, E=64, d=2048, N=262144, k=6, M=8, K=8, ratio=2.0),
        # the plan of 32 layers of 8 experts over a small calibration set (a re-plan while serving)
        dict(name="plan_small", kind="plan", L=32, E=8, d=4096, N=4096, k=2, M=4, K=4, ratio=2.0),
        # offline statistics of 40-expert layers (not a power of two), transitions included
        dict(name="calibrate_odd", kind="calibrate", L=8, E=40, d=1024, N=32768, k=4, K=8),
        # a queue of requests served from and to host memory
        dict(name="batches_fine", kind="batches", nbatch=6, T=1536, **FINE),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["layer", "layer", "layer", "stack", "stack", "select", "plan", "plan",
                       "calibrate", "batches"])
    shape = dict(rng.choice([TINY, WIDE, FINE, FINE]))
    if kind == "layer":
        return dict(kind=kind, T=_log_int(rng, 1, 8192 if shape["E"] == 64 else 4096),
                    call=rng.random() < 0.6, **shape)
    if kind == "stack":
        shape["qbar"] = rng.choice([0.1, 0.5])
        H = rng.choice([1, 1, 2, 3]) if shape["E"] == 8 else rng.choice([1, 1, 2])
        return dict(kind=kind, L=rng.randint(2, 4), T=_log_int(rng, 1, 256), H=H,
                    graph=rng.random() < 0.5, **shape)
    if kind == "select":
        E, k, M, K, d = rng.choice([(8, 2, 4, 4, 4096), (16, 4, 6, 4, 1024), (64, 6, 8, 8, 2048)])
        return dict(kind=kind, T=_log_int(rng, 16, 2048 if E == 64 else 4096), d=d, E=E, k=k, M=M,
                    K=K, qbar=rng.choice([0.1, 0.5]), H=rng.choice([2, 3]),
                    home=rng.choice(["uniform", "zipf1.1"]))
    if kind == "plan":
        E, K, k, M = rng.choice([(8, 4, 2, 4), (16, 4, 2, 4), (32, 8, 4, 8), (64, 8, 6, 8)])
        return dict(kind=kind, L=rng.randint(4, 32 if E < 64 else 24), E=E,
                    d=rng.choice([1024, 2048]), N=_log_int(rng, 1000, 131072), k=k, M=M, K=K,
                    ratio=rng.choice([1.25, 1.5, 2.0]))
    if kind == "calibrate":
        E, K, k = rng.choice([(8, 4, 2), (12, 4, 3), (24, 8, 4), (40, 8, 4), (48, 8, 4), (64, 8, 6)])
        return dict(kind=kind, L=rng.randint(2, 16), E=E, d=rng.choice([512, 1024, 2048]),
                    N=_log_int(rng, 500, 32768), k=k, K=K)
    return dict(kind=kind, nbatch=rng.randint(2, 8), T=_log_int(rng, 64, 2048), **shape)


# ----------------------------------------------------------------- inputs
def _decisions(c, seed, L):
    """What the selection reads for L layers: similarities (the cosines of the router rows, which
    the similarity over N(0, 1) calibration tokens estimates), groups, a placement with one copy of
    every expert and replicas of about a third, and transitions."""
    E, M, K = c["E"], c["M"], c["K"]
    rng = np.random.default_rng(seed + 77)
    routers = [synth.router_weights(E, c["d"], K, seed + 101 + 1000 * l, device=DEV)
               for l in range(L)]
    sims = []
    for W in routers:
        W = W.double()
        W = W / W.norm(dim=1, keepdim=True)
        s = (W @ W.T).float().cpu().numpy()
        np.fill_diagonal(s, 1.0)
        sims.append(s)
    group = synth.cluster_of(E, K).astype(np.int32)
    place = []
    for _ in range(L):
        x = (rng.random((M, E)) < 0.33 / M).astype(np.uint8)
        x[rng.permutation(E) % M, np.arange(E)] = 1
        place.append(x)
    P = rng.gamma(1.0, size=(max(L - 1, 1), E, E)) + 0.01
    P = (P / P.sum(-1, keepdims=True)).astype(np.float32)
    return routers, sims, group, place, P


def _tables(c, seed, sims, group, place):
    sp = synth.server_params(c["M"], c["d"], c.get("dff", 1408), seed)
    stride = B.ordermoe_tables_bytes(c["E"], c["M"])
    buf = torch.zeros(len(sims) * stride, dtype=torch.uint8, device=DEV)
    for l, s in enumerate(sims):
        build_tables(s, group, place[l], 0.5, c["qbar"], sp, DEV, out=buf[l * stride:(l + 1) * stride])
    return buf, stride


def _ffn(c, seed, l):
    return synth.ffn_weights(c["E"], c["d"], c["dff"], seed + 202 + 1000 * l, device=DEV)


def _homes(c, seed, n=None):
    return torch.as_tensor(synth.homes(n or c["T"], c["M"], seed, c["home"])).to(DEV)


def _plan_inputs(c, seed):
    W = torch.stack([synth.router_weights(c["E"], c["d"], c["K"], seed + 101 + 1000 * l, device=DEV)
                     for l in range(c["L"])])
    return W, synth.calibration(c["N"], c["d"], seed, device=DEV)


def _new(*shape, dt=torch.float32):
    return torch.empty(*shape, dtype=dt, device=DEV)


def prepare(case, seed):
    c, s = case, {"case": case}
    kind = c["kind"]
    if kind in ("layer", "batches"):
        routers, sims, group, place, _ = _decisions(c, seed, 1)
        tables, _ = _tables(c, seed, sims, group, place)
        W1, W3, W2 = _ffn(c, seed, 0)
        if kind == "batches":
            n, T = c["nbatch"], c["T"]
            scratch = _new(B.ordermoe_layer_batches_scratch_bytes(T, c["E"], c["d"], c["dff"], c["k"]),
                           dt=torch.uint8)
            s["desc"] = B.make_layer_desc(T, routers[0], W1, W3, W2, tables, c["k"], scratch)
            s["X"] = synth.hidden(n * T, c["d"], seed, DEV).cpu().view(n, T, c["d"]).pin_memory()
            s["home"] = _homes(c, seed, n * T).cpu().view(n, T).pin_memory()
            s["y"] = torch.empty_like(s["X"]).pin_memory()
            return s
        T = c["T"]
        s["X"], s["home"] = synth.hidden(T, c["d"], seed, DEV), _homes(c, seed)
        s["y"] = _new(T, c["d"], dt=torch.bfloat16)
        if c["call"]:
            scratch = _new(B.ordermoe_layer_scratch_bytes(T, c["E"], c["d"], c["dff"], c["k"]),
                           dt=torch.uint8)
            s["desc"] = B.make_layer_desc(T, routers[0], W1, W3, W2, tables, c["k"], scratch)
            s["loc"], s["qhat"] = torch.empty_like(s["home"]), _new(T)
        else:
            s["layer"] = MoELayer(routers[0], W1, W3, W2, tables, c["k"], T)
        return s
    if kind == "stack":
        L, T, H = c["L"], c["T"], c["H"]
        routers, sims, group, place, P = _decisions(c, seed, L)
        tables, stride = _tables(c, seed, sims, group, place)
        layers = []
        for l in range(L):
            W1, W3, W2 = _ffn(c, seed, l)
            layers.append({"W_r": routers[l], "W1": W1, "W3": W3, "W2": W2})
        s["home"] = _homes(c, seed)
        s["loc"], s["qhat"] = s["home"].clone(), _new(T)
        s["hs"] = [synth.hidden(T, c["d"], seed, DEV)] + [_new(T, c["d"], dt=torch.bfloat16)
                                                        for _ in range(L)]
        s["xs"] = [_new(T, c["d"], dt=torch.bfloat16) for _ in range(L + 1)]
        s["stack"] = LayerStack(layers, tables, c["k"], T, DEV, H=H, stride=stride,
                                P=torch.as_tensor(P).to(DEV))
        s["graph"] = None
        if c["graph"]:
            s["graph"] = s["stack"].capture_residual(s["hs"], s["xs"], s["home"], s["loc"], s["qhat"],
                                                     prologue=lambda: _reset(s))
        return s
    if kind == "select":
        T, k = c["T"], c["k"]
        routers, sims, group, place, P = _decisions(c, seed, c["H"])
        s["tables"], s["stride"] = _tables(c, seed, sims, group, place)
        s["P"] = torch.as_tensor(P).to(DEV)
        s["W_r"], s["X"], s["home"] = routers[0], synth.hidden(T, c["d"], seed, DEV), _homes(c, seed)
        s["loc"], s["qhat"] = s["home"].clone(), _new(T)
        # tokens in the middle of a stack: some have moved, some have spent part of the budget
        rng = np.random.default_rng(seed + 5)
        moved = rng.random(T) < 0.4
        s["loc0"] = s["home"].clone()
        s["loc0"][torch.as_tensor(moved).to(DEV)] = torch.as_tensor(
            rng.integers(0, c["M"], int(moved.sum())).astype(np.uint8)).to(DEV)
        s["q0"] = torch.as_tensor((rng.random(T) * 0.6 * c["qbar"]).astype(np.float32)).to(DEV)
        s["out"] = [_new(T, k, dt=dt) for dt in (torch.int32, torch.float32, torch.int32, torch.uint8,
                                                 torch.uint8)]
        return s
    s["W"], s["X"] = _plan_inputs(c, seed)
    L, E, N = c["L"], c["E"], c["N"]
    s["sim"], s["counts"] = _new(L, E, E), _new(L, E, dt=torch.int32)
    if kind == "calibrate":
        s["ws"] = _new(B.ordermoe_similarity_workspace_bytes(L, E, N), dt=torch.uint8)
        s["tcount"], s["P"] = _new(L - 1, E, E, dt=torch.int32), _new(L - 1, E, E)
        return s
    M = c["M"]
    f64 = torch.float64
    s["ws"] = _new(B.ordermoe_plan_workspace_bytes(L, E, N), dt=torch.uint8)
    s["p"] = torch.ones(L, E, dtype=f64, device=DEV)
    s["C"] = torch.as_tensor(synth.capacities(M, L * E, c["ratio"], seed), dtype=f64).to(DEV)
    s["pi"] = torch.as_tensor(synth.token_shares(synth.homes(4096, M, seed, "zipf1.1"), M),
                              dtype=f64).to(DEV)
    i32, u8 = torch.int32, torch.uint8
    s.update(group=_new(L, E, dt=i32), n_groups=_new(L, dt=i32), theta=_new(L),
             importance=_new(L, E, dt=f64), placement=_new(L, M, E, dt=u8), used=_new(M, dt=f64),
             status=_new(1, dt=i32), replicas=_new(M, dt=i32), cover=_new(L, M, E, dt=u8),
             covered=_new(L, dt=i32))
    return s


# ------------------------------------------------------------------- runs
def _reset(s):
    s["loc"].copy_(s["home"])
    s["qhat"].zero_()


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "layer":
        if c["call"]:
            _reset(s)
            B.ordermoe_layer_forward(s["desc"], c["T"], s["X"], s["home"], s["loc"], s["qhat"], s["y"])
            return {"y": s["y"], "loc": s["loc"], "qhat": s["qhat"]}
        m = s["layer"]
        m.forward(s["X"], s["home"], None, None, s["y"])
        return {"y": s["y"], "topk_w": m.topk_w, "chosen": m.chosen, "server": m.server,
                "kind": m.kind}
    if kind == "stack":
        if s["graph"] is not None:
            s["graph"].replay()
        else:
            _reset(s)
            s["stack"].step_residual(s["hs"], s["xs"], s["home"], s["loc"], s["qhat"])
        return {"h": s["hs"][-1], "x": s["xs"][-1], "loc": s["loc"], "qhat": s["qhat"]}
    if kind == "select":
        s["loc"].copy_(s["loc0"])
        s["qhat"].copy_(s["q0"])
        B.ordermoe_route_select_lookahead(s["X"], s["W_r"], None, c["T"], c["E"], c["d"], c["k"], 1,
                                          s["tables"], s["stride"], c["H"], s["P"], s["home"],
                                          s["loc"], s["qhat"], None, *s["out"])
        return {"topk": s["out"][0], "topk_w": s["out"][1], "chosen": s["out"][2],
                "server": s["out"][3], "kind": s["out"][4], "loc": s["loc"], "qhat": s["qhat"]}
    if kind == "batches":
        B.ordermoe_layer_forward_batches(s["desc"], c["nbatch"], c["T"], s["X"], s["home"], s["y"])
        return {"y": s["y"]}
    if kind == "calibrate":
        L, E, N = c["L"], c["E"], c["N"]
        B.ordermoe_similarity(s["W"], s["X"], L, E, c["d"], N, c["k"], s["sim"], s["counts"], s["ws"])
        logits = s["ws"][:N * L * E * 4].view(torch.float32)
        B.ordermoe_transitions(logits, N, L, E, c["k"], s["tcount"], s["P"])
        return {"sim": s["sim"], "counts": s["counts"], "tcount": s["tcount"], "P": s["P"],
                "logits": logits.view(N, L, E)}
    B.ordermoe_plan(s["W"], s["X"], c["L"], c["E"], c["d"], c["N"], c["k"], c["M"], 0.5, 0.9, 0.5,
                    0.5, 0.5, 0.5, 0.5, s["p"], s["C"], s["pi"], s["sim"], s["counts"], s["group"],
                    s["n_groups"], s["theta"], s["importance"], s["placement"], s["used"],
                    s["status"], s["replicas"], s["cover"], s["covered"], s["ws"])
    return {n: s[n] for n in ("sim", "counts", "group", "n_groups", "theta", "importance",
                              "placement", "used", "status", "replicas", "cover", "covered")}


def work(case):
    """Each input read and each output written once; an expert's weights only when a token is
    expected to reach it (each token takes k distinct experts of E)."""
    c = case
    kind = c["kind"]
    if kind in ("plan", "calibrate"):
        C = c["L"] * c["E"]
        flops = 2.0 * c["N"] * C * c["d"] + 2.0 * c["N"] * C * c["E"]
        nbytes = 2.0 * c["N"] * c["d"] + 2.0 * C * c["d"] + 8.0 * C * c["E"]
        if kind == "calibrate":
            nbytes += 4.0 * c["N"] * C  # the logits are kept
        return {"bytes": nbytes, "flops": flops}
    T, d, E, k = c["T"], c["d"], c["E"], c["k"]
    route = 2.0 * T * d * E
    if kind == "select":
        return {"bytes": 2.0 * T * d + 2.0 * E * d + T * (14.0 * k + 12), "flops": route}
    hit = E * (1.0 - (1.0 - k / E) ** T)
    n = {"layer": 1, "stack": c.get("L"), "batches": c.get("nbatch")}[kind]
    weights = 2.0 * 3 * hit * d * c["dff"] * (1 if kind == "batches" else n)
    return {"bytes": weights + n * (2.0 * E * d + 4.0 * T * d),
            "flops": n * (6.0 * T * k * d * c["dff"] + route)}


def tolerance(case):
    """Outputs in bf16 of GEMMs with a bf16 intermediate: about 3e-3 off the 64-bit values, 2^-8 of
    a value at most where a rounding falls the other way; a stack repeats that over its layers.
    Similarities, gate weights and logits are fp32 sums. Whole numbers may differ for near ties."""
    kind = case["kind"]
    if kind in ("layer", "batches"):
        return {"rel": 1e-2, "max": 0.1, "differ": 1e-3}
    if kind == "stack":
        return {"rel": 2e-2, "max": 0.5, "differ": 5e-3}
    if kind == "select":
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    return {"rel": 2e-5, "max": 1e-3, "differ": 1e-3}


# ------------------------------------------------------- the same in 64 bits
class _Method:
    """The routing and FFN of the method on 64-bit tensors. Its decisions compare fp32 costs (the
    interface rounds each table entry once to fp32 and adds with one rounded operation), so the
    selection alone is stated in fp32."""

    def __init__(self, c, seed, L):
        self.c = c
        self.routers, sims, group, place, P = _decisions(c, seed, L)
        self.sp = synth.server_params(c["M"], c["d"], c.get("dff", 1408), seed)
        t = lambda a: torch.as_tensor(a).to(DEV)  # noqa: E731
        F, z = t(self.sp.F), self.sp.z
        comp = self.sp.c / F
        link = z / t(self.sp.B) + t(self.sp.tau)
        link.fill_diagonal_(0.0)
        dl = link + comp[None, :]
        self.A = (self.sp.omega_T * dl[None] / comp[:, None, None]).float()  # [home][from][to]
        self.P = t(P)
        self.Q, self.Cq, self.sub, self.on = [], [], [], []
        g = t(group)
        for l in range(L):
            sm = t(sims[l])
            q = 0.5 * (1.0 - sm.clamp(max=1.0))
            q.fill_diagonal_(0.0)
            self.Q.append(q)
            self.Cq.append((self.sp.omega_Q * q.double() / float(np.float32(c["qbar"]))).float())
            self.sub.append((g[:, None] == g[None]) & (sm >= 0.5)
                            & ~torch.eye(c["E"], dtype=torch.bool, device=DEV))
            self.on.append(t(place[l]).bool())  # [M][E]
        self.qbar = float(np.float32(c["qbar"]))
        self.subs = [[s[r].nonzero().flatten().tolist() for r in range(c["E"])] for s in self.sub]
        self.hosts = [[o[:, e].nonzero().flatten().tolist() for e in range(c["E"])] for o in self.on]

    def phi(self, D, l, a, m, kx, q):
        """The cheapest expected cost of the D layers after l, from server m after expert kx."""
        out = torch.zeros_like(q)
        if D == 0:
            return out
        for kt in range(self.c["E"]):
            p = self.P[l][kx, kt]
            best = torch.full_like(q, math.inf)
            for kk in [kt] + self.subs[l + 1][kt]:
                qk, cq = self.Q[l + 1][kt, kk], self.Cq[l + 1][kt, kk]
                fits = q + qk <= self.qbar if kk != kt else None
                for m2 in self.hosts[l + 1][kk]:
                    v = self.A[a, m, m2] + cq + self.phi(D - 1, l + 1, a, m2, kk, q + qk)
                    best = torch.minimum(best, v if fits is None else torch.where(fits, v, math.inf))
            out = out + p * best
        return out

    def route(self, l, X):
        lg = X.double() @ self.routers[l].double().T
        w, idx = torch.topk(torch.softmax(lg, 1), self.c["k"], dim=1)
        return idx, w / w.sum(1, keepdim=True)

    def select(self, l, idx, a, s, q, H):
        T, k = idx.shape
        E, M = self.c["E"], self.c["M"]
        taken = torch.zeros(T, E, dtype=torch.bool, device=DEV).scatter_(1, idx, True)
        chosen, server, first = torch.empty_like(idx), torch.empty_like(idx), s
        rows = torch.arange(T, device=DEV)
        for j in range(k):
            r = idx[:, j]
            qn = q[:, None] + self.Q[l][r]
            ok = self.sub[l][r] & ~taken & (qn <= self.qbar)
            ok[rows, r] = True
            cost = self.A[a, s][:, None, :] + self.Cq[l][r][:, :, None]  # [T][E][M]
            cost = torch.where(ok[:, :, None] & self.on[l].T[None], cost, math.inf)
            if H > 1:
                for e in range(E):
                    for m in self.hosts[l][e]:
                        t = cost[:, e, m].isfinite().nonzero().flatten()
                        if len(t):
                            cost[t, e, m] += self.phi(H - 1, l, a[t], m, e, qn[t, e])
            # ties: exact, the current server, the lower server, the lower expert
            key = cost.contiguous().view(torch.int32).long() << 32
            key |= (torch.arange(E, device=DEV)[None] != r[:, None]).long()[:, :, None] << 31
            key |= (torch.arange(M, device=DEV)[None] != s[:, None]).long()[:, None, :] << 30
            key |= torch.arange(M, device=DEV)[None, None, :] << 8
            key |= torch.arange(E, device=DEV)[None, :, None]
            best = key.view(T, -1).amin(1)
            e, m = best & 0xFF, (best >> 8) & 0xFF
            chosen[:, j], server[:, j] = e, m
            q = qn[rows, e]
            taken[rows, e] = True
            if j == 0:
                first = m
        return chosen, server, first, q

    def ffn(self, X, chosen, w, weights):
        W1, W3, W2 = weights
        y = torch.zeros(X.shape[0], self.c["d"], dtype=torch.float64, device=DEV)
        for e in range(self.c["E"]):
            t, j = (chosen == e).nonzero(as_tuple=True)
            if len(t):
                x = X[t].double()
                h = torch.nn.functional.silu(x @ W1[e].double().T) * (x @ W3[e].double().T)
                y.index_add_(0, t, (h @ W2[e].double().T) * w[t, j][:, None])
        return y


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("layer", "batches"):
        m = _Method(c, seed, 1)
        n = c["T"] * c.get("nbatch", 1)
        X = synth.hidden(n, c["d"], seed, DEV)
        home = _homes(c, seed, n).long()
        idx, w = m.route(0, X)
        chosen, server, first, q = m.select(0, idx, home, home, torch.zeros(n, device=DEV), 1)
        y = m.ffn(X, chosen, w, _ffn(c, seed, 0))
        if kind == "batches":
            return {"y": y.view(c["nbatch"], c["T"], c["d"])}
        if c["call"]:
            return {"y": y, "loc": None, "qhat": q}
        return {"y": y, "topk_w": w, "chosen": None, "server": None, "kind": None}
    if kind == "stack":
        if c["H"] > 2 and c["E"] > 8:
            return None
        m = _Method(c, seed, c["L"])
        norm = lambda v: v / (v.square().mean(1, keepdim=True) + 1e-6).sqrt()  # noqa: E731
        # the residual stream and the layers' inputs are bf16 tensors of the interface
        bf = lambda v: v.to(torch.bfloat16).double()  # noqa: E731
        h = synth.hidden(c["T"], c["d"], seed, DEV).double()
        home = _homes(c, seed).long()
        s, q = home, torch.zeros(c["T"], device=DEV)
        for l in range(c["L"]):
            x = bf(norm(h))
            idx, w = m.route(l, x)
            chosen, _, s, q = m.select(l, idx, home, s, q, min(c["H"], c["L"] - l))
            h = bf(h + m.ffn(x, chosen, w, _ffn(c, seed, l)))
        return {"h": h, "x": norm(h), "loc": None, "qhat": q}
    if kind == "select":
        m = _Method(c, seed, 1)
        _, w = m.route(0, synth.hidden(c["T"], c["d"], seed, DEV))
        return {"topk": None, "topk_w": w, "chosen": None, "server": None, "kind": None, "loc": None,
                "qhat": None}
    W, X = _plan_inputs(c, seed)
    L, E, N = c["L"], c["E"], c["N"]
    G = torch.zeros(L, E, E, dtype=torch.float64, device=DEV)
    n = torch.zeros(L, E, dtype=torch.float64, device=DEV)
    pairs = torch.zeros(L - 1, E, E, dtype=torch.float64, device=DEV)
    logits = []
    Wd = W.view(L * E, -1).double()
    for x in X.split(16384):
        lg = (x.double() @ Wd.T).view(-1, L, E).transpose(0, 1)  # [L][n][E]
        G += lg.transpose(1, 2) @ lg
        top = torch.zeros_like(lg).scatter_(2, torch.topk(lg, c["k"], dim=2).indices, 1.0)
        n += top.sum(1)
        if kind == "calibrate":
            pairs += top[:-1].transpose(1, 2) @ top[1:]
            logits.append(lg.transpose(0, 1).contiguous())
    nrm = G.diagonal(dim1=1, dim2=2).sqrt()
    sim = G / (nrm[:, :, None] * nrm[:, None, :])
    sim.diagonal(dim1=1, dim2=2).fill_(1.0)
    if kind == "calibrate":
        P = pairs / pairs.sum(2, keepdim=True).clamp(min=1.0)
        return {"sim": sim, "counts": None, "tcount": None, "P": P, "logits": torch.cat(logits)}
    theta = [0.5 + 0.4 * (L - 1 - l) / (L - 1) for l in range(L)]
    imp = np.zeros((L, E))
    S, cnt = sim.cpu().numpy(), n.cpu().numpy()
    for l in range(L):
        dom, grp = [], np.zeros(E, int)
        for j in sorted(range(E), key=lambda e: (-cnt[l, e], e)):
            best = max(range(len(dom)), key=lambda g: S[l, j, dom[g]]) if dom else -1
            if best < 0 or S[l, j, dom[best]] < theta[l]:
                grp[j] = len(dom)
                dom.append(j)
            else:
                grp[j] = best
        for j in range(E):
            imp[l, j] = 0.5 * cnt[l, j] / cnt[l].sum() + 0.5 * S[l, j, grp == grp[j]].mean()
    out = dict.fromkeys(("counts", "group", "n_groups", "placement", "used", "status", "replicas",
                         "cover", "covered"))
    return dict(out, sim=sim, theta=torch.tensor(theta, dtype=torch.float64),
                importance=torch.as_tensor(imp))
