"""GPU parity of the look-ahead selection (Eqs. 41-43): transition statistics
and the depth-H cost-to-go, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_17154_gb300 import binding as B
from paper_2607_17154_gb300 import synth
from paper_2607_17154_gb300.layer import build_tables

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.lib()
    yield
    code, detail = B.ordermoe_device_error()
    assert code == 0, (code, detail)


@pytest.mark.parametrize("N,L,E,kf", [(5000, 4, 8, 2), (3000, 3, 64, 6), (100, 2, 5, 5)])
def test_transitions_given_logits_bit_exact(N, L, E, kf):
    rng = np.random.default_rng(N + E)
    logits = rng.standard_normal((N, L, E)).astype(np.float32)
    logits[:7] = 0.25                                   # ties
    cnt = torch.empty(L - 1, E, E, dtype=torch.int32, device=DEV)
    P = torch.empty(L - 1, E, E, dtype=torch.float32, device=DEV)
    B.ordermoe_transitions(torch.as_tensor(logits).to(DEV), N, L, E, kf, cnt, P)
    rc, rP = oracle.transitions(logits, kf)
    np.testing.assert_array_equal(cnt.cpu().numpy(), rc)
    np.testing.assert_array_equal(P.cpu().numpy(), rP)


@pytest.mark.parametrize("N,L,E,kf", [
    (78500, 2, 12, 3),   # two tiles of tokens a block, the last one ragged
    (257, 9, 17, 1), (700, 3, 64, 8), (300, 3, 33, 9), (1, 2, 1, 1), (513, 4, 40, 5),
    (300, 2, 64, 64), (260, 3, 7, 7), (300, 2, 12, 12),  # every expert
    (300, 2, 63, 4), (520, 2, 33, 2), (300, 3, 5, 2)])   # rows that 16-byte loads do not fit
def test_topk_sets_with_ties_infinities_and_nan(N, L, E, kf):
    """The counts and transitions against the rule itself (kf passes, each
    taking the first unused maximum): equal logits across the boundary, -inf
    and +inf, and NaN logits, which are taken only where a pass starts on one."""
    rng = np.random.default_rng(N + E + kf)
    logits = np.round(rng.standard_normal((N, L, E)) * 2).astype(np.float32) / 2
    logits[rng.random((N, L, E)) < 0.02] = -np.inf
    logits[rng.random((N, L, E)) < 0.01] = np.inf
    logits[::7][rng.random(logits[::7].shape) < 0.03] = np.nan
    logits[0] = -np.inf
    sets = np.zeros((N, L, E), bool)
    n, l = np.ogrid[:N, :L]
    for _ in range(kf):
        best = np.full((N, L), -1)
        bv = np.zeros((N, L), np.float32)
        for e in range(E):
            with np.errstate(invalid="ignore"):
                take = ~sets[:, :, e] & ((best < 0) | (logits[:, :, e] > bv))
            best[take], bv[take] = e, logits[:, :, e][take]
        sets[n, l, best] = True
    s = sets.astype(np.float32)  # sums below 2^24
    want = np.stack([s[:, i].T @ s[:, i + 1] for i in range(L - 1)]).astype(np.int64)
    cnt = torch.empty(L - 1, E, E, dtype=torch.int32, device=DEV)
    P = torch.empty(L - 1, E, E, dtype=torch.float32, device=DEV)
    B.ordermoe_transitions(torch.as_tensor(logits).to(DEV), N, L, E, kf, cnt, P)
    np.testing.assert_array_equal(cnt.cpu().numpy(), want)
    row = want.sum(2, keepdims=True)
    np.testing.assert_array_equal(P.cpu().numpy(), (want / np.maximum(row, 1)).astype(np.float32))
    # unaligned rows, layer by layer: E + 1 floats apart
    wide = torch.zeros(L, N, E + 1, dtype=torch.float32, device=DEV)
    wide[:, :, :E] = torch.as_tensor(logits).to(DEV).transpose(0, 1)
    B.ordermoe_transitions_strided(wide, N, L, E, kf, E + 1, N * (E + 1), cnt, P)
    np.testing.assert_array_equal(cnt.cpu().numpy(), want)
    c = torch.empty(E, dtype=torch.int32, device=DEV)
    B.ordermoe_expert_counts(torch.as_tensor(logits[:, 0].copy()).to(DEV), N, E, kf, c)
    np.testing.assert_array_equal(c.cpu().numpy(), sets[:, 0].sum(0))


def stack_tables(rng, L, E, M, qbar, cheap_links):
    """L layers' tables, random groups/placements, as one device buffer plus the
    oracle's own copies."""
    stride = B.ordermoe_tables_bytes(E, M)
    buf = torch.zeros(L * stride, dtype=torch.uint8, device=DEV)
    otabs = []
    for l in range(L):
        Wt = rng.standard_normal((E, 6)); Wt[:, 0] += 3.0 * (np.arange(E) % 3)
        nrm = np.linalg.norm(Wt, axis=1, keepdims=True)
        sim = ((Wt / nrm) @ (Wt / nrm).T).astype(np.float32); np.fill_diagonal(sim, 1.0)
        group = (np.arange(E) % 3).astype(np.int32)
        x = (rng.random((M, E)) < 0.35).astype(np.uint8)
        for e in range(E):
            if not x[:, e].any():
                x[rng.integers(M), e] = 1
        sp = synth.server_params(M, 4096, 14336, seed=l)
        if cheap_links:
            sp.tau[:] *= 1e-3
        theta = 0.2
        build_tables(sim, group, x, theta, qbar, sp, DEV, out=buf[l * stride:(l + 1) * stride])
        otabs.append(oracle.tables(sim, group, x, theta, qbar, sp.F, sp.B, sp.tau, sp.z, sp.c,
                                   sp.omega_T, sp.omega_Q))
    return buf, stride, otabs


@pytest.mark.parametrize("E,M,k,H,cheap", [(8, 4, 2, 1, True), (8, 4, 2, 2, True), (8, 4, 2, 3, True),
                                           (16, 4, 3, 3, False), (6, 3, 2, 4, True), (32, 8, 2, 2, True),
                                           # H = 3 with 8 servers and dear links: many losses fall
                                           # between the two tabulated cases, their evaluations
                                           # listed and shared by the warps, which read the second
                                           # level's rows and list order
                                           (16, 8, 3, 3, False),
                                           # H = 4: three levels of tables, all checks passing (cheap
                                           # links) and failing or open ones (dear)
                                           (8, 4, 2, 4, False), (16, 4, 3, 4, True), (12, 5, 2, 4, False)])
def test_route_select_lookahead_given_logits_bit_exact(E, M, k, H, cheap):
    rng = np.random.default_rng(E * 10 + H)
    T = 300
    qbar = 0.2
    buf, stride, otabs = stack_tables(rng, H, E, M, qbar, cheap)
    P = rng.random((max(H - 1, 1), E, E)).astype(np.float32)
    P[P < 0.5] = 0
    P = (P / np.maximum(P.sum(axis=2, keepdims=True), 1e-9)).astype(np.float32)
    logits = rng.standard_normal((T, E)).astype(np.float32)
    home = rng.integers(0, M, T).astype(np.uint8)
    loc = np.where(rng.random(T) < 0.5, home, rng.integers(0, M, T)).astype(np.uint8)
    qhat = (rng.random(T) * 0.1).astype(np.float32)
    g = [torch.empty(T, k, dtype=dt, device=DEV)
         for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
    gl = torch.as_tensor(loc).to(DEV); gq = torch.as_tensor(qhat).to(DEV)
    B.ordermoe_route_select_lookahead(None, None, torch.as_tensor(logits).to(DEV), T, E, 0, k, 1, buf,
                                      stride, H, torch.as_tensor(P).to(DEV) if H > 1 else None,
                                      torch.as_tensor(home).to(DEV), gl, gq, None, *g)
    idx, _ = oracle.topk(logits, k)
    ref = oracle.select_lookahead(idx, otabs[:H], P[:H - 1], home, loc, qhat)
    for name, got, want in zip(("chosen", "server", "kind"), (g[2], g[3], g[4]), ref[:3]):
        np.testing.assert_array_equal(got.cpu().numpy(), want, err_msg=name)
    np.testing.assert_array_equal(gl.cpu().numpy(), ref[3])
    np.testing.assert_array_equal(gq.cpu().numpy(), ref[4])
    if H > 1:
        myo = oracle.select(idx, otabs[0], home, loc, qhat)
        print("decisions changed by the look-ahead:", int((myo[0] != ref[0]).sum() + (myo[1] != ref[1]).sum()))


@pytest.mark.parametrize("T,E,M,k,H,skew", [
    (5001, 8, 4, 2, 3, True),     # several tokens a warp, one home with most of them, a ragged last block
    (6, 64, 8, 6, 3, False),      # two experts a lane, every loss regime, prefix minima in the table
    (40, 64, 32, 2, 2, False),    # prefix minima too many for the table: the direct minimum
    (64, 64, 32, 2, 2, True),     # more open evaluations in a step than are listed
    (20, 24, 3, 4, 3, True),      # an evaluation by all warps, lanes past the targets
    (4, 33, 32, 3, 3, True), (60, 1, 1, 1, 4, False), (17, 13, 2, 8, 4, False)])
def test_lookahead_tokens_by_home_bit_exact(T, E, M, k, H, skew):
    """Losses spread over the whole budget, so that candidates fall on the
    tables with every check passing, on those with every check failing and
    between; homes uneven, some servers without tokens."""
    rng = np.random.default_rng(T + E + M)
    qbar = 0.3
    buf, stride, otabs = stack_tables(rng, H, E, M, qbar, True)
    P = rng.random((H - 1, E, E)).astype(np.float32)
    P[P < 0.3] = 0
    P = (P / np.maximum(P.sum(axis=2, keepdims=True), 1e-9)).astype(np.float32)
    logits = rng.standard_normal((T, E)).astype(np.float32)
    home = rng.integers(0, M, T).astype(np.uint8)
    if skew:
        home[rng.random(T) < 0.8] = M // 2
    loc = np.where(rng.random(T) < 0.5, home, rng.integers(0, M, T)).astype(np.uint8)
    qhat = (rng.random(T) * 1.1 * qbar).astype(np.float32)
    g = [torch.empty(T, k, dtype=dt, device=DEV)
         for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
    gl = torch.as_tensor(loc).to(DEV); gq = torch.as_tensor(qhat).to(DEV)
    cnt = torch.zeros(4, dtype=torch.int32, device=DEV)
    B.ordermoe_route_select_lookahead(None, None, torch.as_tensor(logits).to(DEV), T, E, 0, k, 1, buf,
                                      stride, H, torch.as_tensor(P).to(DEV),
                                      torch.as_tensor(home).to(DEV), gl, gq, None, *g, cnt)
    idx, _ = oracle.topk(logits, k)
    ref = oracle.select_lookahead(idx, otabs[:H], P, home, loc, qhat)
    for name, got, want in zip(("chosen", "server", "kind"), (g[2], g[3], g[4]), ref[:3]):
        np.testing.assert_array_equal(got.cpu().numpy(), want, err_msg=name)
    np.testing.assert_array_equal(gl.cpu().numpy(), ref[3])
    np.testing.assert_array_equal(gq.cpu().numpy(), ref[4])
    np.testing.assert_array_equal(cnt.cpu().numpy(), np.bincount(ref[2].ravel(), minlength=4))


@pytest.mark.parametrize("T,E,M,M_stride,k,H,groups", [
    (30, 64, 32, 32, 2, 4, 64),   # the most of everything: no class table, no rows; no substitutes
    (30, 64, 32, 32, 2, 4, 16),   # the same with substitutes: open evaluations by the whole block
    (40, 64, 8, 32, 2, 4, 32),    # a stride with room for more servers than the tables have
    (40, 64, 3, 32, 3, 3, 16), (40, 33, 8, 32, 2, 2, 8), (50, 8, 4, 32, 2, 4, 4),
    (40, 64, 16, 16, 2, 4, 32), (20, 64, 20, 25, 2, 3, 16)])
def test_lookahead_at_the_limits_of_shared_memory(T, E, M, M_stride, k, H, groups):
    """Every E <= 64, M <= 32 and H <= 4, and any stride that holds the tables:
    what does not fit in a block's shared memory is done without. Two servers
    an expert and three successors a transition row, so that the oracle's
    recursion stays small."""
    rng = np.random.default_rng(E + M + M_stride + H + groups)
    qbar = 0.25
    used = B.ordermoe_tables_bytes(E, M)
    stride = B.ordermoe_tables_bytes(E, M_stride)
    buf = torch.zeros(H * stride, dtype=torch.uint8, device=DEV)
    group = (np.arange(E) % groups).astype(np.int32)
    otabs = []
    for l in range(H):
        sim = (0.4 + 0.6 * rng.random((E, E))).astype(np.float32)
        np.fill_diagonal(sim, 1.0)
        x = np.zeros((M, E), np.uint8)
        x[rng.integers(0, M, E), np.arange(E)] = 1
        x[rng.integers(0, M, E), np.arange(E)] = 1
        sp = synth.server_params(M, 4096, 14336, seed=l)
        sp.tau[:] *= 1e-3
        build_tables(sim, group, x, 0.2, qbar, sp, DEV, out=buf[l * stride:l * stride + used])
        otabs.append(oracle.tables(sim, group, x, 0.2, qbar, sp.F, sp.B, sp.tau, sp.z, sp.c, sp.omega_T,
                                   sp.omega_Q))
    P = np.zeros((H - 1, E, E), np.float32)
    for h in range(H - 1):
        for e in range(E):
            P[h, e, rng.choice(E, 3, replace=False)] = (0.5, 0.25, 0.25)
    logits = rng.standard_normal((T, E)).astype(np.float32)
    home = rng.integers(0, M, T).astype(np.uint8)
    loc = np.where(rng.random(T) < 0.5, home, rng.integers(0, M, T)).astype(np.uint8)
    qhat = (rng.random(T) * qbar).astype(np.float32)
    g = [torch.empty(T, k, dtype=dt, device=DEV)
         for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
    gl = torch.as_tensor(loc).to(DEV); gq = torch.as_tensor(qhat).to(DEV)
    B.ordermoe_route_select_lookahead(None, None, torch.as_tensor(logits).to(DEV), T, E, 0, k, 1, buf,
                                      stride, H, torch.as_tensor(P).to(DEV),
                                      torch.as_tensor(home).to(DEV), gl, gq, None, *g)
    idx, _ = oracle.topk(logits, k)
    ref = oracle.select_lookahead(idx, otabs, P, home, loc, qhat)
    for name, got, want in zip(("chosen", "server", "kind"), (g[2], g[3], g[4]), ref[:3]):
        np.testing.assert_array_equal(got.cpu().numpy(), want, err_msg=name)
    np.testing.assert_array_equal(gl.cpu().numpy(), ref[3])
    np.testing.assert_array_equal(gq.cpu().numpy(), ref[4])


def test_lookahead_of_many_tokens_in_several_launches():
    """More tokens than one launch takes (131072): the last launch has 77, and
    reports the index of the token in the call."""
    rng = np.random.default_rng(11)
    T, E, M, k, H, qbar = 131072 + 77, 8, 4, 2, 2, 0.2
    buf, stride, otabs = stack_tables(rng, H, E, M, qbar, True)
    P = rng.random((H - 1, E, E)).astype(np.float32)
    P = (P / P.sum(axis=2, keepdims=True)).astype(np.float32)
    logits = rng.standard_normal((T, E)).astype(np.float32)
    home = rng.integers(0, M, T).astype(np.uint8)
    loc = rng.integers(0, M, T).astype(np.uint8)
    qhat = (rng.random(T) * qbar).astype(np.float32)
    g = [torch.empty(T, k, dtype=dt, device=DEV)
         for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
    idx, _ = oracle.topk(logits, k)
    ref = oracle.select_lookahead(idx, otabs, P, home, loc, qhat)
    for bad in (False, True):
        loc_in = loc.copy()
        if bad:
            loc_in[T - 3] = M
        gl = torch.as_tensor(loc_in).to(DEV); gq = torch.as_tensor(qhat).to(DEV)
        cnt = torch.zeros(4, dtype=torch.int32, device=DEV)
        B.ordermoe_route_select_lookahead(None, None, torch.as_tensor(logits).to(DEV), T, E, 0, k, 1, buf,
                                          stride, H, torch.as_tensor(P).to(DEV),
                                          torch.as_tensor(home).to(DEV), gl, gq, None, *g, cnt)
        assert B.ordermoe_device_error() == ((B.DEV_BAD_INDEX, T - 3) if bad else (0, 0))
        ok = np.arange(T) != (T - 3 if bad else -1)
        for name, got, want in zip(("chosen", "server", "kind"), (g[2], g[3], g[4]), ref[:3]):
            np.testing.assert_array_equal(got.cpu().numpy()[ok], want[ok], err_msg=name)
        np.testing.assert_array_equal(gl.cpu().numpy()[ok], ref[3][ok])
        np.testing.assert_array_equal(gq.cpu().numpy()[ok], ref[4][ok])
        np.testing.assert_array_equal(cnt.cpu().numpy(), np.bincount(ref[2][ok].ravel(), minlength=4))


def test_threads_with_calls_of_different_sizes():
    """Two host threads whose calls share a kernel and ask for different
    amounts of shared memory, each on its own stream: both succeed at every
    call and give what they give alone."""
    import threading

    def prepare(E, M, H, T, seed):
        rng = np.random.default_rng(seed)
        buf, stride, _ = stack_tables(rng, H, E, M, 0.2, True)
        P = rng.random((H - 1, E, E)).astype(np.float32)
        P = torch.as_tensor((P / P.sum(axis=2, keepdims=True)).astype(np.float32)).to(DEV)
        logits = torch.as_tensor(rng.standard_normal((T, E)).astype(np.float32)).to(DEV)
        home = torch.as_tensor(rng.integers(0, M, T).astype(np.uint8)).to(DEV)
        out = [torch.empty(T, 2, dtype=dt, device=DEV)
               for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
        stream = torch.cuda.Stream()

        def call():
            B.ordermoe_route_select_lookahead(None, None, logits, T, E, 0, 2, 1, buf, stride, H, P, home,
                                              None, None, None, *out, None, stream)
        return call, out

    # one instantiation each: the selection of 33-64 experts (H = 2) or of 9-16 (H = 4)
    for small, large in (((33, 2, 2), (64, 8, 2)), ((9, 2, 4), (16, 8, 4))):
        pairs = [prepare(*small, 4, 1), prepare(*large, 4, 2)]
        torch.cuda.synchronize()
        want = []
        for call, out in pairs:
            call()
            torch.cuda.synchronize()
            want.append([o.clone() for o in out])
        errors = []

        def loop(call):
            try:
                for _ in range(400):
                    call()
            except Exception as e:  # noqa: BLE001
                errors.append(e)

        ts = [threading.Thread(target=loop, args=(call,)) for call, _ in pairs]
        [t.start() for t in ts]
        [t.join() for t in ts]
        torch.cuda.synchronize()
        assert not errors, errors[0]
        for (_, out), w in zip(pairs, want):
            for a, b in zip(out, w):
                assert torch.equal(a, b)


def test_lookahead_horizon_one_equals_route_select():
    rng = np.random.default_rng(5)
    E, M, k, T = 8, 4, 2, 200
    buf, stride, otabs = stack_tables(rng, 1, E, M, 0.2, True)
    logits = torch.as_tensor(rng.standard_normal((T, E)).astype(np.float32)).to(DEV)
    home = torch.as_tensor(rng.integers(0, M, T).astype(np.uint8)).to(DEV)
    outs = []
    for fn in ("plain", "lookahead"):
        g = [torch.empty(T, k, dtype=dt, device=DEV)
             for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
        if fn == "plain":
            B.ordermoe_route_select(None, None, logits, T, E, 0, k, 1, buf, home, None, None, None, *g)
        else:
            B.ordermoe_route_select_lookahead(None, None, logits, T, E, 0, k, 1, buf, stride, 1, None,
                                              home, None, None, None, *g)
        outs.append([t.cpu() for t in g])
    for a, b in zip(*outs):
        assert torch.equal(a, b)


def test_decode_stack_with_lookahead_h3_follows_the_oracle():
    """32 Mixtral-shaped routers, batch 128, H = 3: each layer looks two layers
    ahead with the transition statistics of the calibration logits. The
    oracle follows every token through the 32 selections (fed the same fp32
    logits, so each decision is compared exactly)."""
    w = synth.workload("decode_stack")
    L, T, E, k, M = w.L, w.T, w.E, w.k, w.M
    H = 3
    rng = np.random.default_rng(21)
    buf, stride, otabs = stack_tables(rng, L, E, M, w.qbar, cheap_links=True)
    cal = rng.standard_normal((4096, L, E)).astype(np.float32)
    _, P = oracle.transitions(cal, k)
    gP = torch.as_tensor(P).to(DEV)
    logits = rng.standard_normal((L, T, E)).astype(np.float32)
    home = rng.integers(0, M, T).astype(np.uint8)
    gl = torch.as_tensor(home).to(DEV); gq = torch.zeros(T, device=DEV)
    gh = torch.as_tensor(home).to(DEV)
    gch = []
    for l in range(L):
        Hl = min(H, L - l)
        g = [torch.empty(T, k, dtype=dt, device=DEV)
             for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
        B.ordermoe_route_select_lookahead(None, None, torch.as_tensor(logits[l]).to(DEV), T, E, 0, k, 1,
                                          buf[l * stride:], stride, Hl,
                                          gP[l:l + Hl - 1].contiguous() if Hl > 1 else None,
                                          gh, gl, gq, None, *g)
        gch.append(g[2].cpu().numpy())
    loc = home.copy(); q = np.zeros(T, np.float32)
    for l in range(L):
        Hl = min(H, L - l)
        idx, _ = oracle.topk(logits[l], k)
        ch, sv, kd, loc, q = oracle.select_lookahead(idx, otabs[l:l + Hl], P[l:l + Hl - 1], home, loc, q)
        np.testing.assert_array_equal(gch[l], ch, err_msg="layer %d" % l)
    np.testing.assert_array_equal(gl.cpu().numpy(), loc)
    np.testing.assert_array_equal(gq.cpu().numpy(), q)
    assert (q <= np.float32(w.qbar)).all()


@pytest.mark.parametrize("E,M,k,H", [(8, 4, 2, 3), (16, 6, 4, 2), (64, 8, 6, 2)])
def test_router_path_lookahead_bit_exact(E, M, k, H):
    """Router GEMM on the tensor cores, then the warp-per-token look-ahead
    pass: the decisions follow the oracle given the logits the router wrote
    (T spans three 128-row router tiles with a ragged tail)."""
    rng = np.random.default_rng(E + 100 * H)
    T, d = 300, 256
    buf, stride, otabs = stack_tables(rng, H, E, M, 0.25, cheap_links=True)
    P = rng.random((H - 1, E, E)).astype(np.float32)
    P[P < 0.6] = 0
    P = (P / np.maximum(P.sum(axis=2, keepdims=True), 1e-9)).astype(np.float32)
    X = torch.randn(T, d, device=DEV).to(torch.bfloat16)
    W_r = (torch.randn(E, d, device=DEV) * 0.2).to(torch.bfloat16)
    home = rng.integers(0, M, T).astype(np.uint8)
    loc = np.where(rng.random(T) < 0.5, home, rng.integers(0, M, T)).astype(np.uint8)
    qhat = (rng.random(T) * 0.1).astype(np.float32)
    g = [torch.empty(T, k, dtype=dt, device=DEV)
         for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
    lg = torch.empty(T, E, device=DEV)
    cnt = torch.zeros(4, dtype=torch.int32, device=DEV)
    gl = torch.as_tensor(loc).to(DEV); gq = torch.as_tensor(qhat).to(DEV)
    B.ordermoe_route_select_lookahead(X, W_r, None, T, E, d, k, 1, buf, stride, H,
                                      torch.as_tensor(P).to(DEV), torch.as_tensor(home).to(DEV),
                                      gl, gq, lg, *g, counters=cnt)
    logits = lg.cpu().numpy()
    idx, _ = oracle.topk(logits, k)
    np.testing.assert_array_equal(g[0].cpu().numpy(), idx)
    ch, sv, kd, rl, rq = oracle.select_lookahead(idx, otabs, P, home, loc, qhat)
    np.testing.assert_array_equal(g[2].cpu().numpy(), ch)
    np.testing.assert_array_equal(g[3].cpu().numpy(), sv)
    np.testing.assert_array_equal(g[4].cpu().numpy(), kd)
    np.testing.assert_array_equal(gl.cpu().numpy(), rl)
    np.testing.assert_array_equal(gq.cpu().numpy(), rq)
    np.testing.assert_array_equal(cnt.cpu().numpy(), np.bincount(kd.ravel(), minlength=4))


def test_lookahead_skips_a_nan_token_and_reports_it():
    rng = np.random.default_rng(9)
    E, M, k, T, H = 8, 4, 2, 70, 2
    buf, stride, otabs = stack_tables(rng, H, E, M, 0.2, cheap_links=True)
    P = np.full((1, E, E), 1.0 / E, np.float32)
    logits = rng.standard_normal((T, E)).astype(np.float32)
    bad = logits.copy(); bad[3, 5] = np.nan
    home = rng.integers(0, M, T).astype(np.uint8)
    g = [torch.empty(T, k, dtype=dt, device=DEV)
         for dt in (torch.int32, torch.float32, torch.int32, torch.uint8, torch.uint8)]
    gl = torch.as_tensor(home).to(DEV); gq = torch.zeros(T, device=DEV)
    B.ordermoe_route_select_lookahead(None, None, torch.as_tensor(bad).to(DEV), T, E, 0, k, 1, buf,
                                      stride, H, torch.as_tensor(P).to(DEV),
                                      torch.as_tensor(home).to(DEV), gl, gq, None, *g)
    code, detail = B.ordermoe_device_error()
    assert code == B.DEV_NAN_LOGIT and detail == 3
    idx, _ = oracle.topk(logits, k)
    ch, sv, kd, rl, rq = oracle.select_lookahead(idx, otabs, P, home, home.copy(),
                                                 np.zeros(T, np.float32))
    keep = np.arange(T) != 3
    np.testing.assert_array_equal(g[2].cpu().numpy()[keep], ch[keep])
    np.testing.assert_array_equal(g[3].cpu().numpy()[keep], sv[keep])
    np.testing.assert_array_equal(gl.cpu().numpy()[keep], rl[keep])
    assert gl[3].item() == home[3] and gq[3].item() == 0.0       # state of the NaN token kept
    assert (g[0][3] == -1).all().item()


def test_layer_stack_lookahead_through_layer_forward():
    """Six small layers through ordermoe_layer_forward with H = 3 (router on the
    tensor cores, tables of all layers in one stack, transition matrices
    between them): the carried location and loss follow the oracle's
    look-ahead selection on the oracle's own router logits, for every token
    whose top-k has no near tie at any layer."""
    from paper_2607_17154_gb300.layer import LayerStack
    rng = np.random.default_rng(44)
    L, T, E, k, M, d, dff, H = 6, 300, 8, 2, 4, 256, 512, 3
    buf, stride, otabs = stack_tables(rng, L, E, M, 0.3, cheap_links=True)
    P = rng.random((L - 1, E, E)).astype(np.float32)
    P[P < 0.5] = 0
    P = (P / np.maximum(P.sum(axis=2, keepdims=True), 1e-9)).astype(np.float32)
    layers, Wrb = [], []
    for l in range(L):
        Wr = synth.router_weights(E, d, 2, seed=70 + l, device=DEV)
        W1, W3, W2 = synth.ffn_weights(E, d, dff, seed=80 + l, device=DEV)
        layers.append({"W_r": Wr, "W1": W1, "W3": W3, "W2": W2})
        Wrb.append(synth.bits(Wr))
    stack = LayerStack(layers, buf, k, T, DEV, H=H, stride=stride, P=torch.as_tensor(P).to(DEV))
    Xs = [synth.hidden(T, d, 90 + l, device=DEV) for l in range(L)]
    ys = [torch.empty(T, d, dtype=torch.bfloat16, device=DEV) for _ in range(L)]
    home_np = rng.integers(0, M, T).astype(np.uint8)
    home = torch.as_tensor(home_np).to(DEV)
    loc, qhat = home.clone(), torch.zeros(T, device=DEV)
    counters = torch.zeros(4, dtype=torch.int32, device=DEV)
    stack.step(Xs, home, loc, qhat, ys, counters)
    torch.cuda.synchronize()
    assert counters.sum().item() == L * T * k
    o_loc, o_q = home_np.copy(), np.zeros(T, np.float32)
    clear = np.ones(T, bool)
    for l in range(L):
        logits = oracle.router_logits(synth.bits(Xs[l]), Wrb[l])
        srt = -np.sort(-logits.astype(np.float64), axis=1)
        clear &= np.abs(np.diff(srt[:, :k + 1], axis=1)).min(axis=1) > 1e-3
        idx, _ = oracle.topk(logits, k)
        Hl = min(H, L - l)
        _, _, _, o_loc, o_q = oracle.select_lookahead(idx, otabs[l:l + Hl], P[l:l + Hl - 1], home_np,
                                                      o_loc, o_q)
    assert clear.mean() > 0.6
    np.testing.assert_array_equal(loc.cpu().numpy()[clear], o_loc[clear])
    np.testing.assert_array_equal(qhat.cpu().numpy()[clear], o_q[clear])
    assert torch.isfinite(ys[-1].float()).all()


def test_layer_stack_graph_replay_equals_eager_step():
    """A step captured as one CUDA graph and replayed gives the eager step's
    outputs bit for bit (location, loss, every layer's y), with look-ahead."""
    from paper_2607_17154_gb300.layer import LayerStack
    rng = np.random.default_rng(45)
    L, T, E, k, M, d, dff, H = 4, 128, 8, 2, 4, 256, 512, 3
    buf, stride, _ = stack_tables(rng, L, E, M, 0.3, cheap_links=True)
    P = rng.random((L - 1, E, E)).astype(np.float32)
    P = (P / P.sum(axis=2, keepdims=True)).astype(np.float32)
    layers = []
    for l in range(L):
        W1, W3, W2 = synth.ffn_weights(E, d, dff, seed=180 + l, device=DEV)
        layers.append({"W_r": synth.router_weights(E, d, 2, seed=170 + l, device=DEV),
                       "W1": W1, "W3": W3, "W2": W2})
    stack = LayerStack(layers, buf, k, T, DEV, H=H, stride=stride, P=torch.as_tensor(P).to(DEV))
    Xs = [synth.hidden(T, d, 190 + l, device=DEV) for l in range(L)]
    home = torch.as_tensor(rng.integers(0, M, T).astype(np.uint8)).to(DEV)
    outs = []
    for mode in ("eager", "graph"):
        ys = [torch.zeros(T, d, dtype=torch.bfloat16, device=DEV) for _ in range(L)]
        loc, qhat = home.clone(), torch.zeros(T, device=DEV)

        def reset():
            loc.copy_(home)
            qhat.zero_()
        if mode == "eager":
            reset()
            stack.step(Xs, home, loc, qhat, ys)
        else:
            g = stack.capture(Xs, home, loc, qhat, ys, prologue=reset)
            for y in ys:
                y.zero_()
            loc.fill_(0)
            g.replay()
        torch.cuda.synchronize()
        outs.append([loc.clone(), qhat.clone()] + [y.clone() for y in ys])
    for a, b in zip(*outs):
        assert torch.equal(a, b)


def test_residual_stack_lookahead_teacher_forced():
    """Six small layers on the residual map (each layer reads RMSNorm of the
    residual stream) through ordermoe_layer_forward_residual with H = 3: with
    the oracle fed each layer's recorded router logits (teacher forcing), the
    look-ahead selection carries the same location and accumulated loss for
    every token, bit for bit, near ties included; the recorded logits match
    the oracle's on the GPU's layer inputs; a CUDA-graph replay of the step
    gives the eager step's results bit for bit."""
    from paper_2607_17154_gb300.layer import LayerStack
    rng = np.random.default_rng(46)
    L, T, E, k, M, d, dff, H = 6, 300, 8, 2, 4, 256, 512, 3
    buf, stride, otabs = stack_tables(rng, L, E, M, 0.3, cheap_links=True)
    P = rng.random((L - 1, E, E)).astype(np.float32)
    P[P < 0.5] = 0
    P = (P / np.maximum(P.sum(axis=2, keepdims=True), 1e-9)).astype(np.float32)
    layers, Wrb = [], []
    for l in range(L):
        Wr = synth.router_weights(E, d, 2, seed=270 + l, device=DEV)
        W1, W3, W2 = synth.ffn_weights(E, d, dff, seed=280 + l, device=DEV)
        layers.append({"W_r": Wr, "W1": W1, "W3": W3, "W2": W2})
        Wrb.append(synth.bits(Wr))
    stack = LayerStack(layers, buf, k, T, DEV, H=H, stride=stride, P=torch.as_tensor(P).to(DEV))
    home_np = rng.integers(0, M, T).astype(np.uint8)
    home = torch.as_tensor(home_np).to(DEV)
    h0 = synth.hidden(T, d, 290, device=DEV)
    outs = []
    for mode in ("eager", "graph"):
        hs = [h0] + [torch.zeros_like(h0) for _ in range(L)]
        xs = [torch.zeros_like(h0) for _ in range(L + 1)]
        loc, qhat = home.clone(), torch.zeros(T, device=DEV)
        logits = torch.zeros(L, T, E, device=DEV)

        def reset():
            loc.copy_(home)
            qhat.zero_()
        if mode == "eager":
            counters = torch.zeros(4, dtype=torch.int32, device=DEV)
            reset()
            stack.step_residual(hs, xs, home, loc, qhat, counters=counters, logits=logits)
            torch.cuda.synchronize()
            assert counters.sum().item() == L * T * k
            lg = logits.cpu().numpy()
            o_loc, o_q = home_np.copy(), np.zeros(T, np.float32)
            for l in range(L):
                np.testing.assert_allclose(lg[l], oracle.router_logits(synth.bits(xs[l]), Wrb[l]),
                                           rtol=1e-3, atol=2e-3)
                idx, _ = oracle.topk(lg[l], k)
                Hl = min(H, L - l)
                _, _, _, o_loc, o_q = oracle.select_lookahead(idx, otabs[l:l + Hl], P[l:l + Hl - 1],
                                                              home_np, o_loc, o_q)
            np.testing.assert_array_equal(loc.cpu().numpy(), o_loc)
            np.testing.assert_array_equal(qhat.cpu().numpy().view(np.uint32), o_q.view(np.uint32))
            assert torch.isfinite(hs[-1].float()).all()
        else:
            g = stack.capture_residual(hs, xs, home, loc, qhat, prologue=reset)
            for t in hs[1:] + xs:
                t.zero_()
            loc.fill_(0)
            g.replay()
            torch.cuda.synchronize()
        outs.append([loc.clone(), qhat.clone()] + [t.clone() for t in hs[1:] + xs])
    for a, b in zip(*outs):
        assert torch.equal(a, b)
