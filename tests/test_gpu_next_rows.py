"""Parity of the draft-management entry points (through the C ABI) with the CPU oracle.

Integer results (tokens, trees, paths, indices) are bit-exact.  Where an fp32 probability decides an
integer (pruning, soft matching, sampling), the probabilities are compared within a tolerance, the decisions
are compared wherever the oracle's fp64 value is not within rounding of the threshold, and everything that
follows from the decisions the device took is checked bit-exactly by handing those decisions to the oracle."""
import ctypes as C

import numpy as np
import pytest

import launch_info
from paper_2402_11131_b200 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROB_RTOL = 2e-5       # fp32 log-sum-exp over <= 51200 logits against the fp64 oracle
MARGIN = 1e-4          # decisions within this relative distance of their threshold may fall on either side


@pytest.fixture(scope="module")
def cuda():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2402_11131_b200 import api, build
    build.build()
    api.lib()
    return api


def _desc_fields(d, n_max=64):
    return (d.n_nodes, d.max_depth, list(d.parent[:n_max]), list(d.depth[:n_max]), [int(x) for x in d.anc_mask[:n_max]])


def _i32(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()


# ---- next draft ------------------------------------------------------------------------------------
@pytest.mark.parametrize("B,gamma,V,k,max_nodes,ties", [(1, 4, 32000, 2, 64, False), (3, 3, 51200, 4, 64, False),
                                                         (2, 4, 4097, 8, 64, True), (2, 2, 37, 3, 9, True),
                                                         (1, 4, 32000, 1, 64, False), (16, 4, 32000, 2, 31, False)])
def test_next_draft_is_bit_exact(cuda, oracle, B, gamma, V, k, max_nodes, ties):
    api = cuda
    rng = np.random.default_rng(1000 + V + k)
    n_rows = 5
    lg = rng.standard_normal((B, n_rows, gamma, V)).astype(np.float32)
    if ties:
        lg = np.round(lg * 2) / 2                                        # heavy ties: lowest indices must win
    rows = rng.integers(0, n_rows, B).astype(np.int32)
    bonus = rng.integers(0, V, B).astype(np.int32)
    d_tokens = torch.full((B, max_nodes), -7, dtype=torch.int32, device="cuda")
    d_trees = api.empty_trees(B)
    ws = api.workspace(api.ss_next_draft_workspace_bytes(B, gamma, V))
    for rep in range(2):                                                 # the workspace is left ready for reuse
        api.ss_next_draft(torch.from_numpy(lg).cuda(), _i32(rows), _i32(bonus), k, max_nodes, d_tokens, d_trees, ws)
        assert api.ss_status(ws) == 0
        toks = d_tokens.cpu().numpy()
        descs = api.trees_from_device(d_trees)
        for b in range(B):
            want_tok, want_par = oracle.next_draft(lg[b, rows[b]], k, int(bonus[b]), max_nodes)
            n = len(want_tok)
            assert descs[b].n_nodes == n and descs[b].gamma == gamma
            np.testing.assert_array_equal(toks[b, :n], want_tok)
            assert (toks[b, n:] == -1).all()
            host = api.ss_tree_build(want_par, gamma)                    # the descriptor the host builder gives
            assert _desc_fields(descs[b]) == _desc_fields(host)


# clusters of 12 and 16 CTAs, and the sizes next to them; the CTAs of a sequence are the grid's first dimension
@pytest.mark.parametrize("B,gamma,V,k,ties,ctas", [(1, 3, 32768, 8, True, 6), (1, 3, 32769, 8, True, 12), (1, 3, 32773, 8, True, 12), (6, 3, 50257, 8, True, 12),
                                                   (6, 4, 51201, 8, True, 16), (7, 4, 51201, 8, True, 8), (2, 2, 131100, 8, True, 16),
                                                   (1, 4, 32768, 8, False, 8), (1, 4, 32766, 8, False, 16), (1, 1, 131100, 8, True, 8)])
def test_next_draft_with_clusters_beyond_eight_ctas(cuda, oracle, B, gamma, V, k, ties, ctas):
    api = cuda
    ws, lg = api.workspace(api.ss_next_draft_workspace_bytes(B, gamma, V)), torch.zeros((B, 1, gamma, V), device="cuda")
    trees, tokens, bonus = api.empty_trees(B), _i32(np.zeros((B, 64))), _i32(np.zeros(B))
    launched = launch_info.kernels(lambda: api.ss_next_draft(lg, None, bonus, k, 64, tokens, trees, ws))
    assert [x["grid"] for x in launched] == [(ctas, B, 1)]
    test_next_draft_is_bit_exact(cuda, oracle, B, gamma, V, k, 64, ties)


@pytest.mark.parametrize("call", ["draft", "sampled"])
def test_selection_keeps_no_logits_in_local_memory(cuda, call):
    """The batch of logits that a thread scans stays in registers (with an index into it, it would be 128 bytes of stack)."""
    api = cuda
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
    B, T, V, g = 2, 8, 20000, 2
    trees = api.trees_to_device([api.ss_tree_build([-1] + [0] * (T - 1), g)] * B)
    if call == "draft":
        ws = api.workspace(api.ss_next_draft_workspace_bytes(B, g, V))
        lg = torch.randn((B, 1, g, V), device="cuda")
        run = lambda: api.ss_next_draft(lg, None, i32(B), 2, T, i32(B, T), trees, ws)  # noqa: E731
    else:
        ws = api.workspace(api.ss_tree_verify_sampled_workspace_bytes(B, T, V))
        lg, u = torch.randn((B, T, V), device="cuda"), torch.rand((B, T), device="cuda")
        run = lambda: api.ss_tree_verify_sampled(lg, i32(B, T), trees, u, 4, i32(B), i32(B, api.SS_PATH_STRIDE), i32(B), i32(B), i32(B, T), ws)  # noqa: E731
    mine = [k for k in launch_info.kernels(run) if "next_draft" in k["name"] or "sampled_verify" in k["name"]]
    assert len(mine) == 1 and mine[0]["local_bytes"] <= 16


def test_next_draft_special_values_follow_the_order_of_the_verification(cuda, oracle):
    api = cuda
    V = 300
    lg = np.zeros((1, 1, 3, V), dtype=np.float32)
    lg[0, 0, 0, :] = np.nan; lg[0, 0, 0, [17, 5]] = [1.0, 1.0]            # NaNs rank below everything; ties by index
    lg[0, 0, 1, :] = -np.inf; lg[0, 0, 1, 250] = -3e38                    # -inf is an ordinary (lowest) value
    lg[0, 0, 2, :] = -0.0; lg[0, 0, 2, 9] = 0.0; lg[0, 0, 2, 100] = 1e-45   # -0 == +0; a subnormal is larger
    d_tokens = torch.zeros((1, 64), dtype=torch.int32, device="cuda")
    d_trees = api.empty_trees(1)
    ws = api.workspace(api.ss_next_draft_workspace_bytes(1, 3, V))
    api.ss_next_draft(torch.from_numpy(lg).cuda(), None, _i32([4]), 3, 64, d_tokens, d_trees, ws)
    want_tok, _ = oracle.next_draft(lg[0, 0], 3, 4, 64)
    np.testing.assert_array_equal(d_tokens.cpu().numpy()[0, :len(want_tok)], want_tok)
    assert list(want_tok[1:4]) == [5, 17, 0] and list(want_tok[4:7]) == [250, 0, 1] and list(want_tok[13:16]) == [100, 0, 1]


@pytest.mark.parametrize("V,k", [(4095, 8), (4097, 4), (16383, 3), (32771, 8)])       # 1, 2, 4 and 8 CTAs per row, odd rows unaligned
def test_next_draft_of_rows_with_more_ties_than_the_candidate_list(cuda, oracle, V, k):
    """A row's candidates are listed against a bound; rows of equal entries (one value, -inf, NaN) outgrow the list and
    are selected by passes over the row instead."""
    api = cuda
    lg = np.random.default_rng(V).standard_normal((2, 1, 4, V)).astype(np.float32)
    lg[0, 0, 1], lg[0, 0, 2], lg[0, 0, 3] = 0.5, -np.inf, np.nan
    lg[1, 0, 0], lg[1, 0, 0, V - 1] = 0.5, 0.75
    d_tokens = torch.zeros((2, 64), dtype=torch.int32, device="cuda")
    ws = api.workspace(api.ss_next_draft_workspace_bytes(2, 4, V))
    api.ss_next_draft(torch.from_numpy(lg).cuda(), None, _i32([4, 5]), k, 64, d_tokens, api.empty_trees(2), ws)
    assert api.ss_status(ws) == 0
    for b in range(2):
        want, _ = oracle.next_draft(lg[b, 0], k, 4 + b, 64)
        np.testing.assert_array_equal(d_tokens.cpu().numpy()[b, :len(want)], want)


# ---- pruning -----------------------------------------------------------------------------------------
@pytest.mark.parametrize("name", ["1.3b", "7b", "7b_ragged16"])
def test_tree_prune_matches_the_oracle(cuda, oracle, name):
    api = cuda
    st = W.make_step(W.CONFIGS[name])
    c = st.cfg
    B, T, V = c.batch, c.n_nodes, c.vocab
    lg = st.logits()                                                     # stands in for the early-exit logits
    tok = st.draft_tokens.astype(np.int32)
    descs = [api.ss_tree_build(st.parent[b][:st.nodes(b)], c.gamma) for b in range(B)]
    trees = api.trees_to_device(descs)
    # a threshold in the middle of the observed transition probabilities, so that both outcomes occur
    probs0 = oracle.tree_prune(lg[0], tok[0], st.parent[0], 0.0)["edge_prob"]
    tau = float(np.sort(probs0[1:])[len(probs0) // 2] * 1.5)
    out = dict(edge_prob=torch.zeros((B, T), device="cuda"), new_index=torch.zeros((B, T), dtype=torch.int32, device="cuda"),
               kept_nodes=torch.zeros((B, T), dtype=torch.int32, device="cuda"),
               kept_tokens=torch.zeros((B, T), dtype=torch.int32, device="cuda"))
    pruned = api.empty_trees(B)
    ws = api.workspace(api.ss_tree_prune_workspace_bytes(B, T, V))
    for rep in range(2):
        api.ss_tree_prune(torch.from_numpy(lg).cuda(), _i32(tok), trees, tau, out["edge_prob"], out["new_index"],
                          out["kept_nodes"], out["kept_tokens"], pruned, ws)
        assert api.ss_status(ws) == 0
        got = {k: v.cpu().numpy() for k, v in out.items()}
        pdesc = api.trees_from_device(pruned)
        n_dropped = 0
        for b in range(B):
            ref = oracle.tree_prune(lg[b], tok[b], st.parent[b], tau)
            np.testing.assert_allclose(got["edge_prob"][b], ref["edge_prob"], rtol=PROB_RTOL, atol=1e-30)
            dev_keep_edge = got["edge_prob"][b] >= np.float32(tau)      # the decision the device took, per edge
            clear = np.abs(ref["edge_prob"] - tau) > MARGIN * tau
            np.testing.assert_array_equal(dev_keep_edge[clear], (ref["edge_prob"] >= tau)[clear])
            follow = oracle.tree_prune(lg[b], tok[b], st.parent[b], tau, decide=dev_keep_edge.astype(np.uint8))
            n = len(follow["kept_nodes"])
            n_dropped += T - n
            np.testing.assert_array_equal(got["new_index"][b], follow["new_index"])
            np.testing.assert_array_equal(got["kept_nodes"][b, :n], follow["kept_nodes"])
            assert (got["kept_nodes"][b, n:] == -1).all()
            np.testing.assert_array_equal(got["kept_tokens"][b, :n], tok[b][follow["kept_nodes"]])
            assert _desc_fields(pdesc[b]) == _desc_fields(api.ss_tree_build(follow["new_parent"], c.gamma))
        assert 0 < n_dropped < B * T


@pytest.mark.parametrize("soft", [False, True])
@pytest.mark.parametrize("V", [1, 2, 33, 1023, 8191, 8193, 20001])       # one vector, unaligned rows, a batch of loads and one logit more
def test_row_statistics_at_the_edges_of_a_scan(cuda, V, soft):
    """Edge probabilities (and entropies) of short, unaligned and peaked rows with -inf and NaN among the logits, against fp64.  Rows 6
    and 7 have their mass away from the maximum: one logit above all others by 8, and one in 256 above the others by 5.25 (with
    others of its thread).  A term is off by at most 2 ulp of the exponential and a row's sum by the roundings of its longest chain of
    additions (20001 logits over 256 threads and 4 partial sums, then 10 merges: 30 roundings), SUM = 34 * 2^-24 = 2e-6 in all.  A
    probability's exponent child - (m + log Z) is rounded at the size of its terms, each by half an ulp, log Z by one; the entropy
    log Z - W / Z has SUM for log Z and twice that for the quotient.  (An exponential without the correction of its argument's rounding is off by
    3e-7 of such a row's sum, which no bound on fp32 results tells from their own roundings.)"""
    api = cuda
    B, T = 2, 9
    SUM, ULP = 34 * 2.0 ** -24, 2.0 ** -23
    rng = np.random.default_rng(77 + V)
    scale = np.array([1.0, 1.0, 4.0, 30.0, 1.0, 1.0, 0.0, 0.0, 1.0])[None, :, None]
    lg = (rng.standard_normal((B, T, V)) * scale + np.array([0.0, 300.0, 0.0, 0.0, -80.0, 5.0, -8.0, -5.25, 0.0])[None, :, None]).astype(np.float32)
    lg[:, 6, V // 2] = 0.0
    lg[:, 7, ::256] = 0.0
    tok = rng.integers(0, V, (B, T)).astype(np.int32)
    if V > 8:                                                            # (not at the children's tokens)
        for t, bad in ((0, np.nan), (4, -np.inf), (5, np.nan)):
            at = np.setdiff1d(rng.integers(0, V, V // 3), tok)
            lg[:, t, at] = bad
    parent = list(range(-1, T - 1))
    trees = api.trees_to_device([api.ss_tree_build(parent, 2)] * B)
    edge = torch.zeros((B, T), device="cuda")
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
    ws = api.workspace(api.ss_tree_prune_workspace_bytes(B, T, V))
    x = np.where(np.isnan(lg), -np.inf, lg.astype(np.float64))
    m = x.max(-1, keepdims=True)
    e = np.exp(x - m)
    z = e.sum(-1)
    log_z, lse = np.log(z), m[..., 0] + np.log(z)
    if soft:
        ent = torch.zeros((B, T), device="cuda")
        api.ss_tree_verify_soft(torch.from_numpy(lg).cuda(), _i32(tok), trees, 0.09, 0.3, i32(B), i32(B, api.SS_PATH_STRIDE), i32(B), i32(B), edge, ent, ws)
        w = -(np.where(e > 0, x - m, 0.0) * e).sum(-1) / z
        err = np.abs(ent.cpu().numpy() - (log_z + w))
        assert (err <= SUM + 2 * SUM * w + ULP * (log_z + w)).all(), err
    else:
        api.ss_tree_prune(torch.from_numpy(lg).cuda(), _i32(tok), trees, 0.1, edge, i32(B, T), i32(B, T), i32(B, T), api.empty_trees(B), ws)
    assert api.ss_status(ws) == 0
    child = np.take_along_axis(x[:, :-1], tok[:, 1:, None].astype(np.int64), -1)[..., 0]
    log_z, lse, z = log_z[:, :-1], lse[:, :-1], z[:, :-1]
    want = np.exp(child - m[:, :-1, 0]) / z
    rel = SUM + 2 * ULP + ULP * log_z + ULP / 2 * (np.abs(lse) + np.abs(child - lse))
    got = edge.cpu().numpy()
    assert (got[:, 0] == 1.0).all()
    err = np.abs(got[:, 1:] - want)
    assert (err <= rel * want + 1e-30).all(), err / want


@pytest.mark.parametrize("call", ["greedy", "soft", "prune"])
def test_rows_that_no_node_owns_cost_no_traffic(cuda, call):
    """Trees of one node in buffers for 64: of 131 MB of logits (more than L2 holds) only a 64th is needed.  A call that touches the
    others' 8000 logits, a batch each, takes about as long as with full trees; one that does not is launches and little else."""
    api = cuda
    B, N, V = 64, 64, 8000
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
    f32 = lambda *shape: torch.zeros(shape, dtype=torch.float32, device="cuda")  # noqa: E731
    lg, tok = torch.randn((B, N, V), device="cuda"), i32(B, N)
    out = (i32(B), i32(B, api.SS_PATH_STRIDE), i32(B), i32(B))
    ws = api.workspace((api.ss_tree_verify_workspace_bytes if call == "greedy" else api.ss_tree_prune_workspace_bytes)(B, N, V))
    edge, ent, node, pruned = f32(B, N), f32(B, N), (i32(B, N), i32(B, N), i32(B, N)), api.empty_trees(B)

    def run(trees):
        if call == "greedy":
            api.ss_tree_verify(lg, tok, trees, *out, node[0], ws)
        elif call == "soft":
            api.ss_tree_verify_soft(lg, tok, trees, 0.09, 0.3, *out, edge, ent, ws)
        else:
            api.ss_tree_prune(lg, tok, trees, 0.1, edge, *node, pruned, ws)

    def us(n_nodes):
        trees = api.trees_to_device([api.ss_tree_build([-1] + [0] * (n_nodes - 1), 1)] * B)
        run(trees)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(20):
                run(trees)
        best = 1e9
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(); g.replay(); b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 50)
        return best

    small, full = us(1), us(64)
    assert small < 0.42 * full, (small, full)             # (8 / 23 to 10 / 36 us; 14 / 21 to 16 / 35 with a batch of every row loaded)


# ---- attention directly behind the calls that write its trees ---------------------------------------------
@pytest.mark.parametrize("batch,heads", [(1, 8), (6, 30)])               # both kernels that read the trees before their wait
@pytest.mark.parametrize("writer", ["draft", "prune"])
def test_attention_sees_the_trees_that_the_call_before_it_wrote(cuda, writer, batch, heads):
    """compaction -> next draft (or pruning) -> attention on the new trees, which promises a stable prefix and so reads the
    descriptors before it waits for the kernel before it.  The trees alternate between two sizes, nothing
    synchronises; every output has to be that of its own tree."""
    api = cuda
    from paper_2402_11131_b200.step import DeviceStep
    T, g, V = 31, 4, 20000
    cfg = W.custom_config("order", batch=batch, n_layers=1, n_msa_layers=1, prefix_len=200, n_nodes=T, gamma=g, max_depth=4, vocab=V,
                          n_heads=heads, head_dim=128, tree_kind="topk_growth", config_id=990)
    st = W.make_step(cfg)
    dev = DeviceStep(st)
    dev.run_verify()
    dev.accept_len.fill_(1)                                              # (a path of the root alone moves nothing)
    full = dev.trees.clone()
    rng = np.random.default_rng(991)
    logits = torch.from_numpy(rng.standard_normal((batch, 1, g, V)).astype(np.float32)).cuda()
    exits = torch.from_numpy(rng.standard_normal((batch, T, V)).astype(np.float32)).cuda()
    new_tokens, index, kept, kept_tokens = (torch.zeros((batch, T), dtype=torch.int32, device="cuda") for _ in range(4))
    prob = torch.zeros((batch, T), device="cuda")
    ws = api.workspace(max(api.ss_next_draft_workspace_bytes(batch, g, V), api.ss_tree_prune_workspace_bytes(batch, T, V)))

    def write(kind):
        if writer == "draft":                                            # 31 nodes, or a chain of 5
            api.ss_next_draft(logits, None, dev.bonus_token, 2 - kind, T, new_tokens, dev.trees, ws)
        else:                                                            # all nodes, or the root alone
            api.ss_tree_prune(exits, dev.tokens, full, (0.0, 2.0)[kind], prob, index, kept, kept_tokens, dev.trees, ws)

    def outputs():
        return dev.o_main[0].clone(), dev.o_spec[0].clone()

    want = []
    for kind in (0, 1):
        write(kind)
        torch.cuda.synchronize()
        dev.o_main[0].fill_(7.0), dev.o_spec[0].fill_(7.0)
        dev.run_attention()
        torch.cuda.synchronize()
        want.append(outputs())
    assert not torch.equal(want[0][0], want[1][0])
    got = []
    for i in range(40):
        dev.o_main[0].fill_(7.0), dev.o_spec[0].fill_(7.0)
        dev.run_compact()
        write(i & 1)
        dev.run_attention()
        got.append(outputs())
    assert api.ss_status(dev.attn_ws) == 0 and api.ss_status(ws) == 0
    for i, out in enumerate(got):
        assert all(torch.equal(x, y) for x, y in zip(out, want[i & 1])), i


# ---- soft and sampled verification ----------------------------------------------------------------------
def _verify_outputs(B):
    return dict(accept_len=torch.full((B,), -7, dtype=torch.int32, device="cuda"),
                accept_path=torch.full((B, 64), -7, dtype=torch.int32, device="cuda"),
                last_node=torch.full((B,), -7, dtype=torch.int32, device="cuda"),
                bonus_token=torch.full((B,), -7, dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("name", ["tiny", "2.7b", "7b_ragged16"])
def test_soft_verification_matches_the_oracle(cuda, oracle, name):
    api = cuda
    st = W.make_step(W.CONFIGS[name])
    c = st.cfg
    B, T, V = c.batch, c.n_nodes, c.vocab
    lg = (st.logits() * 0.5).astype(np.float32)                          # flatter rows: the thresholds bite on some edges
    tok = st.draft_tokens.astype(np.int32)
    trees = api.trees_to_device([api.ss_tree_build(st.parent[b][:st.nodes(b)], c.gamma) for b in range(B)])
    eps, delta = 0.05, 0.3
    o = _verify_outputs(B)
    prob = torch.zeros((B, T), device="cuda")
    ent = torch.zeros((B, T), device="cuda")
    ws = api.workspace(api.ss_tree_prune_workspace_bytes(B, T, V))
    for rep in range(2):
        api.ss_tree_verify_soft(torch.from_numpy(lg).cuda(), _i32(tok), trees, eps, delta, o["accept_len"], o["accept_path"],
                                o["last_node"], o["bonus_token"], prob, ent, ws)
        assert api.ss_status(ws) == 0
        gp, ge = prob.cpu().numpy(), ent.cpu().numpy()
        lens = o["accept_len"].cpu().numpy()
        for b in range(B):
            ref = oracle.tree_verify_soft(lg[b], tok[b], st.parent[b], eps, delta, path_cap=64)
            np.testing.assert_allclose(gp[b], ref["edge_prob"], rtol=PROB_RTOL, atol=1e-30)
            np.testing.assert_allclose(ge[b], ref["node_entropy"], rtol=2e-5, atol=2e-5)
            par = st.parent[b]
            bar32 = np.minimum(np.float32(eps), np.float32(delta) * np.exp(-ge[b][np.maximum(par, 0)]).astype(np.float32))
            dev_ok = gp[b] >= bar32
            dev_ok[0] = True
            bar64 = np.minimum(eps, delta * np.exp(-ref["node_entropy"][np.maximum(par, 0)]))
            clear = np.abs(ref["edge_prob"] - bar64) > 10 * MARGIN * bar64
            clear[0] = False
            np.testing.assert_array_equal(dev_ok[clear], (ref["edge_prob"] >= bar64)[clear])
            follow = oracle.tree_verify_soft(lg[b], tok[b], par, eps, delta, decide=dev_ok.astype(np.uint8), path_cap=64)
            if clear[1:].all():
                assert int(lens[b]) == follow["accept_len"]
                np.testing.assert_array_equal(o["accept_path"][b].cpu().numpy(), follow["path"])
                assert int(o["last_node"][b]) == follow["last_node"]
                assert int(o["bonus_token"][b]) == follow["bonus_token"]
        assert lens.min() >= 1


@pytest.mark.parametrize("name,k", [("tiny", 3), ("1.3b", 8), ("7b", 4), ("7b_ragged16", 2)])
def test_sampled_verification_matches_the_oracle(cuda, oracle, name, k):
    api = cuda
    st = W.make_step(W.CONFIGS[name])
    c = st.cfg
    B, T, V = c.batch, c.n_nodes, c.vocab
    lg = st.logits()
    rng = np.random.default_rng(77 + k)
    u = rng.random((B, T)).astype(np.float32)
    # half of the children carry the token the oracle draws at their parent, so that paths get accepted
    tok = st.draft_tokens.astype(np.int32).copy()
    drawn_ref = np.zeros((B, T), dtype=np.int32)
    for b in range(B):
        drawn_ref[b] = oracle.tree_verify_sampled(lg[b], tok[b], st.parent[b], k, u[b], path_cap=64)["node_token"]
        for ch in range(1, T):
            if rng.random() < 0.5:
                tok[b, ch] = drawn_ref[b, st.parent[b][ch]]
    trees = api.trees_to_device([api.ss_tree_build(st.parent[b][:st.nodes(b)], c.gamma) for b in range(B)])
    o = _verify_outputs(B)
    node_token = torch.zeros((B, T), dtype=torch.int32, device="cuda")
    ws = api.workspace(api.ss_tree_verify_sampled_workspace_bytes(B, T, V))
    for rep in range(2):
        api.ss_tree_verify_sampled(torch.from_numpy(lg).cuda(), _i32(tok), trees, torch.from_numpy(u).cuda(), k,
                                   o["accept_len"], o["accept_path"], o["last_node"], o["bonus_token"], node_token, ws)
        assert api.ss_status(ws) == 0
        got_tok = node_token.cpu().numpy()
        n_same = 0
        for b in range(B):
            # the draw itself: equal to the oracle's unless u lies within rounding of a step of the distribution
            for t in range(T):
                idx = np.argsort(-lg[b, t], kind="stable")[:k]
                p = np.exp(lg[b, t, idx].astype(np.float64) - float(lg[b, t, idx[0]]))
                cdf = np.cumsum(p / p.sum())
                assert got_tok[b, t] in idx
                if np.min(np.abs(cdf - float(u[b, t]))) > 1e-5:
                    assert got_tok[b, t] == drawn_ref[b, t]
                    n_same += 1
            follow = oracle.tree_verify_sampled(lg[b], tok[b], st.parent[b], k, u[b], drawn=got_tok[b], path_cap=64)
            assert int(o["accept_len"][b]) == follow["accept_len"]
            np.testing.assert_array_equal(o["accept_path"][b].cpu().numpy(), follow["path"])
            assert int(o["last_node"][b]) == follow["last_node"]
            assert int(o["bonus_token"][b]) == follow["bonus_token"]
        assert n_same > 0.99 * B * T
        assert int(o["accept_len"].max()) >= 2


def test_verification_and_pruning_need_no_ancestor_words(cuda):
    """Descriptors that carry parents and depths only give what complete ones give: the ancestor words are the
    attention's."""
    api = cuda
    st = W.make_step(W.custom_config("noanc", batch=3, n_layers=1, prefix_len=4, n_nodes=40, gamma=2, max_depth=5, vocab=500, p_accept=0.8,
                                     tree_kind="topk_growth", config_id=992))
    B, T, V = 3, 40, 500
    logits, tok = torch.from_numpy(st.logits()).cuda(), _i32(st.draft_tokens)
    u = torch.rand((B, T), generator=torch.Generator().manual_seed(5)).cuda()
    ws = api.workspace(max(api.ss_tree_verify_workspace_bytes(B, T, V), api.ss_tree_prune_workspace_bytes(B, T, V),
                           api.ss_tree_verify_sampled_workspace_bytes(B, T, V)))
    results = []
    for with_words in (True, False):
        descs = [api.ss_tree_build(st.parent[b], 2) for b in range(B)]
        if not with_words:
            for d in descs:
                C.memset(C.addressof(d) + api.TreeDesc.anc_mask.offset, 0, 8 * 64)
        trees = api.trees_to_device(descs)
        for call in ("greedy", "soft", "sampled", "prune"):
            o = list(_verify_outputs(B).values())
            node = torch.zeros((B, T), dtype=torch.int32, device="cuda")
            prob, ent = torch.zeros((B, T), device="cuda"), torch.zeros((B, T), device="cuda")
            extra = [torch.zeros((B, T), dtype=torch.int32, device="cuda") for _ in range(3)]
            pruned = api.empty_trees(B)
            if call == "greedy":
                api.ss_tree_verify(logits, tok, trees, *o, node, ws)
            elif call == "soft":
                api.ss_tree_verify_soft(logits, tok, trees, 0.05, 0.3, *o, prob, ent, ws)
            elif call == "sampled":
                api.ss_tree_verify_sampled(logits, tok, trees, u, 2, *o, node, ws)
            else:
                api.ss_tree_prune(logits, tok, trees, 0.05, prob, *extra, pruned, ws)
            assert api.ss_status(ws) == 0
            results.append([t.cpu().clone() for t in (*o, node, prob, ent, *extra, pruned)])
    assert int(results[0][0].max()) >= 3                                 # (accept_len: there is a path to get wrong)
    for full, bare in zip(results[:4], results[4:]):
        assert all(torch.equal(x, y) for x, y in zip(full, bare))


# ---- stream insertion and value rotation ------------------------------------------------------------------
@pytest.mark.parametrize("rows,gamma,hidden", [(64, 4, 4096), (1, 1, 8), (37, 3, 2560), (1024, 4, 4096), (0, 2, 64)])
def test_stream_insert_is_bit_exact(cuda, oracle, rows, gamma, hidden):
    api = cuda
    rng = np.random.default_rng(rows + hidden)
    m = W.f32_to_bf16_bits(rng.standard_normal((rows, hidden)).astype(np.float32) * 2)
    p = W.f32_to_bf16_bits(rng.standard_normal((gamma, hidden)).astype(np.float32) * 0.02)
    out = torch.zeros((rows, gamma, hidden), dtype=torch.bfloat16, device="cuda")
    api.ss_stream_insert(api.bf16_to_device(m) if rows else torch.zeros((0, hidden), dtype=torch.bfloat16, device="cuda"),
                         api.bf16_to_device(p), out)
    torch.cuda.synchronize()
    if rows:
        np.testing.assert_array_equal(api.bf16_to_host_bits(out), oracle.stream_insert(m, p))


@pytest.mark.parametrize("width", [8, 24, 80, 512, 520, 1016, 1024, 1032])
def test_streams_of_narrow_widths_with_odd_numbers_of_rows(cuda, oracle, width):
    """Widths below 8 x 128 put several rows in a CTA: rows that fill no CTA, and one more than a CTA takes at a time."""
    api = cuda
    per_cta = 2 * max(256 // (width // 8), 1)
    for rows in (1, per_cta - 1, per_cta + 1, 7 * per_cta + 3):
        rng = np.random.default_rng(rows + width)
        m = W.f32_to_bf16_bits(rng.standard_normal((rows, width)).astype(np.float32))
        p = W.f32_to_bf16_bits(rng.standard_normal((3, width)).astype(np.float32))
        out = torch.full((rows + 1, 3, width), 7.0, dtype=torch.bfloat16, device="cuda")
        rot = out.clone()
        api.ss_stream_insert(api.bf16_to_device(m), api.bf16_to_device(p), out)
        api.ss_value_rotate(api.bf16_to_device(m), rot, 0.25)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(api.bf16_to_host_bits(out)[:rows], oracle.stream_insert(m, p))
        np.testing.assert_array_equal(api.bf16_to_host_bits(rot)[:rows], oracle.value_rotate(m, 3, 0.25))
        assert bool((out[rows] == 7.0).all()) and bool((rot[rows] == 7.0).all())


@pytest.mark.parametrize("rows,gamma,width,eps", [(64 * 32, 4, 128, 0.01), (5, 1, 8, 0.3), (2048, 3, 80, 1.0 / 4100)])
def test_value_rotation_is_bit_exact(cuda, oracle, rows, gamma, width, eps):
    api = cuda
    rng = np.random.default_rng(rows + width)
    v = W.f32_to_bf16_bits(rng.standard_normal((rows, width)).astype(np.float32))
    out = torch.zeros((rows, gamma, width), dtype=torch.bfloat16, device="cuda")
    api.ss_value_rotate(api.bf16_to_device(v), out, eps)
    torch.cuda.synchronize()
    eps32 = float(np.float32(eps))                                       # the C ABI takes epsilon as fp32
    np.testing.assert_array_equal(api.bf16_to_host_bits(out), oracle.value_rotate(v, gamma, eps32))


def test_next_rows_reject_bad_arguments_before_launching(cuda):
    api = cuda
    lib, a = api.lib(), C.c_void_p(0x10000)
    assert lib.ss_next_draft(a, 1, None, a, 1, 5, 100, 2, 64, a, a, a, 1 << 20, None) == api.SS_ERR_UNSUPPORTED
    assert lib.ss_next_draft(a, 1, None, a, 1, 4, 100, 9, 64, a, a, a, 1 << 20, None) == api.SS_ERR_UNSUPPORTED
    assert lib.ss_next_draft(a, 1, None, a, 1, 4, 100, 2, 64, a, a, a, 16, None) == api.SS_ERR_WORKSPACE
    assert lib.ss_next_draft(None, 1, None, a, 1, 4, 100, 2, 64, a, a, a, 1 << 20, None) == api.SS_ERR_INVALID_ARG
    assert lib.ss_tree_prune(a, a, a, 1, 65, 100, 0.1, a, a, a, a, a, a, 1 << 20, None) == api.SS_ERR_UNSUPPORTED
    assert lib.ss_tree_verify_sampled(a, a, a, a, 1, 8, 100, 0, a, a, a, a, None, a, 1 << 20, None) == api.SS_ERR_INVALID_ARG
    assert lib.ss_stream_insert(a, a, a, 4, 2, 12, None) == api.SS_ERR_UNSUPPORTED
    assert lib.ss_value_rotate(a, a, 4, 5, 64, 0.1, None) == api.SS_ERR_UNSUPPORTED
