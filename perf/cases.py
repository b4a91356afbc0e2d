"""The workloads whose speed counts: what a decode loop asks of this library, over the sizes it meets.

Every case goes through the public entry points of ``paper_2402_11131_b200.api`` as a serving program calls them:
buffers, tree descriptors, attention parameters and workspaces are made once and live on the GPU; a pass is the
calls of one decode step, launched one by one on the current stream.

Kinds
  step     one decode step: every layer's tree attention (plain layers, then the multi-stream layers), verification
           of the draft (greedy, soft or sampled), compaction of the accepted path's K/V, next draft
  verify   one verification call alone (the step of a program that owns its attention)
  prune    pruning of a draft by early-exit probabilities
  draft    the next draft from the stream logits of the last accepted node
  streams  stream initialisation and value rotation of one multi-stream layer's inputs
"""
import numpy as np
import torch

from paper_2402_11131_b200 import api
from paper_2402_11131_b200.workloads import draw_tree


def _step(name, batch, layers, msa_layers, heads, head_dim, prefix, nodes, depth, gamma, vocab, p, verify="greedy",
          lse=False):
    return dict(name=name, kind="step", batch=batch, layers=layers, msa_layers=msa_layers, heads=heads,
                head_dim=head_dim, prefix_lo=prefix[0], prefix_hi=prefix[1], nodes=nodes, depth=depth, gamma=gamma,
                vocab=vocab, p_lo=p[0], p_hi=p[1], verify=verify, top_k=4, lse=lse)


def _rows(name, kind, batch, nodes, vocab, mode="", gamma=4, top_k=4):
    return dict(name=name, kind=kind, mode=mode, batch=batch, nodes=nodes, depth=4, gamma=gamma, vocab=vocab, top_k=top_k)


def listed():
    return [
        # the smallest step: one small layer, launch latency and little else
        _step("step tiny", 1, 1, 1, 2, 64, (64, 64), 6, 2, 3, 512, (0.6, 0.6)),
        # one user decoding with a 1.3B-class model: short prefix, 16-node tree
        _step("step 1.3b", 1, 24, 4, 32, 64, (512, 512), 16, 3, 3, 51200, (0.7, 0.7)),
        # one user, 2.7B-class model: head_dim 80, 32-node tree
        _step("step 2.7b", 1, 32, 4, 32, 80, (1024, 1024), 32, 4, 3, 51200, (0.7, 0.7)),
        # one user, 7B-class model: the headline workload of bench.py
        _step("step 7b", 1, 32, 4, 32, 128, (2048, 2048), 64, 4, 4, 32000, (0.6, 0.6)),
        # sixteen users at once, each at another length: the largest step
        _step("step 7b ragged x16", 16, 32, 4, 32, 128, (512, 4096), 64, 4, 4, 32000, (0.4, 0.8)),
        # a few users on a small model with sizes that fit no tile: odd tree, odd head count, vocabulary not a
        # multiple of four, sampled verification, log-sum-exps wanted
        _step("step odd x5", 5, 8, 2, 13, 64, (37, 1301), 27, 4, 2, 50257, (0.5, 0.8), "sampled", True),
        # verification alone: the three criteria, one user and a batch
        _rows("verify greedy 7b x16", "verify", 16, 64, 32000, "greedy"),
        _rows("verify soft 2.7b", "verify", 1, 32, 51200, "soft"),
        _rows("verify sampled 7b", "verify", 1, 64, 32000, "sampled"),
        # early-exit pruning of a batch of drafts
        _rows("prune 7b x16", "prune", 16, 64, 32000),
        # the next draft of a batch: four streams, top 4
        _rows("draft 7b x16", "draft", 16, 64, 32000),
        # inputs of the first multi-stream layer of a batch: 16 trees of 64 nodes, hidden size 4096
        dict(name="streams 7b x16", kind="streams", rows=1024, gamma=4, hidden=4096),
    ]


def _log(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["verify", "verify", "prune", "draft", "streams"])
    if kind == "step":
        top = work(listed()[4])
        while True:
            layers = _log(rng, 1, 32)
            lo = _log(rng, 16, 4096)
            case = _step("", rng.choice([1, 1, 2, 4, 8, 16]), layers, rng.randint(0, min(layers, 8)), _log(rng, 2, 40),
                         rng.choice([64, 80, 128]), (lo, min(4096, lo * rng.choice([1, 2, 8]))), rng.randint(1, 64),
                         rng.randint(3, 6), rng.randint(1, 4), rng.choice([_log(rng, 512, 51200), 32000, 51200]),
                         (0.4, 0.8), rng.choice(["greedy", "greedy", "soft", "sampled"]), rng.random() < 0.25)
            del case["name"]
            w = work(case)
            if w["bytes"] <= top["bytes"] and w["flops"] <= top["flops"]:
                return case
    if kind == "streams":
        return dict(kind=kind, rows=_log(rng, 1, 1024), gamma=rng.randint(1, 4), hidden=8 * _log(rng, 16, 640))
    case = _rows("", kind, _log(rng, 1, 16), rng.randint(2, 64), rng.choice([_log(rng, 512, 51200), 32000, 51200]),
                 rng.choice(["greedy", "soft", "sampled"]) if kind == "verify" else "", rng.randint(1, 4), rng.randint(1, 8))
    del case["name"]
    return case


def _trees(rng, case):
    """One random draft per sequence: parent arrays and their descriptors on the device."""
    kind = "uniform_parent" if case["nodes"] < 8 else "topk_growth"
    parents = [draw_tree(rng, case["nodes"], case["depth"], kind) for _ in range(case["batch"])]
    return parents, api.trees_to_device([api.ss_tree_build(p, case["gamma"]) for p in parents])


def _verify_inputs(rng, gen, case, parents, p_accept):
    """Draft tokens and main-stream logits in which a parent agrees with one of its children with probability p."""
    B, T, V = case["batch"], case["nodes"], case["vocab"]
    tokens = rng.integers(0, V, size=(B, T)).astype(np.int32)
    logits = torch.randn((B, T, V), generator=gen, device="cuda", dtype=torch.float32)
    at = []
    for b in range(B):
        taken = set()
        hit = rng.random(T) < p_accept[b]
        for c in range(1, T):
            u = int(parents[b][c])
            if hit[c] and u not in taken:
                taken.add(u)
                at.append((b, u, int(tokens[b, c])))
    if at:
        i = torch.tensor(at, device="cuda").t()
        logits[i[0], i[1], i[2]] = 16.0
    return torch.from_numpy(tokens).cuda(), logits


def _verify_state(case, mode):
    B, T, V = case["batch"], case["nodes"], case["vocab"]
    size = {"greedy": api.ss_tree_verify_workspace_bytes, "soft": api.ss_tree_prune_workspace_bytes,
            "sampled": api.ss_tree_verify_sampled_workspace_bytes}[mode]
    i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
    f32 = lambda *shape: torch.zeros(shape, dtype=torch.float32, device="cuda")  # noqa: E731
    return dict(mode=mode, top_k=case["top_k"], verify_ws=api.workspace(size(B, T, V)), accept_len=i32(B),
                accept_path=i32(B, api.SS_PATH_STRIDE), last_node=i32(B), bonus_token=i32(B), node_token=i32(B, T),
                edge_prob=f32(B, T), entropy=f32(B, T))


def _draft_state(gen, case, n_rows):
    B, V, g = case["batch"], case["vocab"], case["gamma"]
    return dict(draft_k=case["top_k"], draft_nodes=case["nodes"],
                stream_logits=torch.randn((B, n_rows, g, V), generator=gen, device="cuda", dtype=torch.float32),
                new_tokens=torch.zeros((B, case["nodes"]), dtype=torch.int32, device="cuda"), new_trees=api.empty_trees(B),
                draft_ws=api.workspace(api.ss_next_draft_workspace_bytes(B, g, V)))


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(rng.integers(1 << 62)))
    kind = case["kind"]
    if kind == "streams":
        bf = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)  # noqa: E731
        rows, g, h = case["rows"], case["gamma"], case["hidden"]
        return dict(kind=kind, hidden=3 * bf(rows, h), emb=0.01 * bf(g, h), value=bf(rows, h), epsilon=0.05,
                    streams=torch.zeros((rows, g, h), dtype=torch.bfloat16, device="cuda"),
                    values=torch.zeros((rows, g, h), dtype=torch.bfloat16, device="cuda"))
    B, T = case["batch"], case["nodes"]
    if kind == "draft":
        st = dict(kind=kind, **_draft_state(gen, case, T))
        st["last_node"] = torch.from_numpy(rng.integers(0, T, size=B).astype(np.int32)).cuda()
        st["bonus_token"] = torch.from_numpy(rng.integers(0, case["vocab"], size=B).astype(np.int32)).cuda()
        return st
    parents, trees = _trees(rng, case)
    p_accept = rng.uniform(case.get("p_lo", 0.6), case.get("p_hi", 0.6), size=B)
    tokens, logits = _verify_inputs(rng, gen, case, parents, p_accept)
    st = dict(kind=kind, trees=trees, tokens=tokens, logits=logits)
    if kind == "prune":
        i32 = lambda *shape: torch.zeros(shape, dtype=torch.int32, device="cuda")  # noqa: E731
        st.update(threshold=0.05, edge_prob=torch.zeros((B, T), dtype=torch.float32, device="cuda"), new_index=i32(B, T),
                  kept_nodes=i32(B, T), kept_tokens=i32(B, T), pruned=api.empty_trees(B),
                  prune_ws=api.workspace(api.ss_tree_prune_workspace_bytes(B, T, case["vocab"])))
        return st
    mode = case["mode"] if kind == "verify" else case["verify"]
    st.update(_verify_state(case, mode))
    st["uniforms"] = torch.rand((B, T), generator=gen, device="cuda", dtype=torch.float32)
    if kind == "step":
        st.update(_draft_state(gen, case, T))
        _attention_state(rng, gen, case, st)
    return st


def _attention_state(rng, gen, case, st):
    """The KV cache of all layers (slot-major, ragged sequences one after another), this step's queries and stream
    K/V, the outputs, one workspace for all layers and each layer's call parameters."""
    B, T, H, d, g = case["batch"], case["nodes"], case["heads"], case["head_dim"], case["gamma"]
    n, n_msa = case["layers"], case["msa_layers"]
    # a ragged batch: lengths spread evenly over the range, in an order of the seed's (so a cache has one size per case)
    length = rng.permutation((case["prefix_lo"] + (case["prefix_hi"] - case["prefix_lo"]) * (np.arange(B) + 0.5) / B).astype(np.int64))
    cap = (length + T + 63) // 64 * 64
    start = np.concatenate([[0], np.cumsum(cap)[:-1]])
    dev = lambda a, t: torch.from_numpy(np.asarray(a)).to(t).cuda()  # noqa: E731
    kv_start, kv_len, kv_capacity = dev(start, torch.int64), dev(length, torch.int32), dev(cap, torch.int32)

    def bf(*shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)

    def zeros(*shape, dtype=torch.bfloat16):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    # unit-variance scores: queries ~ N(0, 1), scaled by 1 / sqrt(d) in the call
    k_all, v_all = bf(n, int(cap.sum()), H, d), bf(n, int(cap.sum()), H, d)
    q_main, o_main = bf(n, B, T, H, d), zeros(n, B, T, H, d)
    q_spec, k_spec, v_spec = (bf(n_msa, B, T, g, H, d) for _ in range(3))
    o_spec = zeros(n_msa, B, T, g, H, d)
    lse_main = zeros(n, B, T, H, dtype=torch.float32) if case["lse"] else None
    lse_spec = zeros(n_msa, B, T, g, H, dtype=torch.float32) if case["lse"] else None

    def params(i, ws):
        m = i - (n - n_msa)                     # >= 0: the m-th multi-stream layer
        spec = {} if m < 0 else dict(q_spec=q_spec[m], k_spec=k_spec[m], v_spec=v_spec[m], o_spec=o_spec[m],
                                     lse_spec=lse_spec[m] if case["lse"] else None)
        # nothing that runs before an attention call of the step writes a cached prefix, a length or a tree
        return api.make_attn_params(q_main=q_main[i], o_main=o_main[i], k_cache=k_all[i], v_cache=v_all[i],
                                    kv_start=kv_start, kv_len=kv_len, kv_capacity=kv_capacity, trees=st["trees"],
                                    gamma=g if m >= 0 else 0, sm_scale=d ** -0.5,
                                    lse_main=lse_main[i] if case["lse"] else None, workspace=ws, prefix_stable=True, **spec)

    ws = api.workspace(max(api.ss_msa_attention_workspace_bytes(params(i, None)) for i in range(n)))
    st.update(k_all=k_all, v_all=v_all, layout=api.make_cache_layout(k_all), kv_start=kv_start, kv_len=kv_len,
              kv_len_out=torch.zeros_like(kv_len), layers=[params(i, ws) for i in range(n)],
              attention=[t for t in (o_main, o_spec, lse_main, lse_spec) if t is not None],
              keep=(q_main, q_spec, k_spec, v_spec, kv_capacity, ws))


def _verify(s):
    if s["mode"] == "greedy":
        api.ss_tree_verify(s["logits"], s["tokens"], s["trees"], s["accept_len"], s["accept_path"], s["last_node"],
                           s["bonus_token"], s["node_token"], s["verify_ws"])
    elif s["mode"] == "soft":
        api.ss_tree_verify_soft(s["logits"], s["tokens"], s["trees"], 0.09, 0.3, s["accept_len"], s["accept_path"],
                                s["last_node"], s["bonus_token"], s["edge_prob"], s["entropy"], s["verify_ws"])
    else:
        api.ss_tree_verify_sampled(s["logits"], s["tokens"], s["trees"], s["uniforms"], s["top_k"], s["accept_len"],
                                   s["accept_path"], s["last_node"], s["bonus_token"], s["node_token"], s["verify_ws"])
    out = [s["accept_len"], s["accept_path"], s["last_node"], s["bonus_token"]]
    return out + ([s["edge_prob"], s["entropy"]] if s["mode"] == "soft" else [s["node_token"]])


def _draft(s):
    api.ss_next_draft(s["stream_logits"], s["last_node"], s["bonus_token"], s["draft_k"], s["draft_nodes"],
                      s["new_tokens"], s["new_trees"], s["draft_ws"])
    return [s["new_tokens"], s["new_trees"]]


def run(s):
    if s["kind"] == "step":
        for p in s["layers"]:
            api.ss_msa_attention(p)
        out = _verify(s)
        # the compaction is in place: a second pass on the same state sees the tree slots it has moved
        api.ss_kv_compact(s["k_all"], s["v_all"], s["layout"], s["kv_start"], s["kv_len"], s["accept_len"],
                          s["accept_path"], s["kv_len_out"])
        return s["attention"] + out + [s["k_all"], s["v_all"], s["kv_len_out"]] + _draft(s)
    if s["kind"] == "verify":
        return _verify(s)
    if s["kind"] == "prune":
        api.ss_tree_prune(s["logits"], s["tokens"], s["trees"], s["threshold"], s["edge_prob"], s["new_index"],
                          s["kept_nodes"], s["kept_tokens"], s["pruned"], s["prune_ws"])
        return [s["edge_prob"], s["new_index"], s["kept_nodes"], s["kept_tokens"], s["pruned"]]
    if s["kind"] == "draft":
        return _draft(s)
    api.ss_stream_insert(s["hidden"], s["emb"], s["streams"])
    api.ss_value_rotate(s["value"], s["values"], s["epsilon"])
    return [s["streams"], s["values"]]


def work(case):
    """Each input read once, each output written once (integers and the few moved K/V rows left out); prefixes of a
    ragged batch at their mean length, each node's root path at half the tree's depth."""
    kind = case["kind"]
    if kind == "streams":
        rows, g, h = case["rows"], case["gamma"], case["hidden"]
        return {"bytes": 2 * (2 * rows * h + g * h + 2 * rows * g * h), "flops": 4 * rows * g * h}
    B, T, V, g = case["batch"], case["nodes"], case["vocab"], case["gamma"]
    if kind == "draft":
        return {"bytes": 4 * B * g * V, "flops": B * g * V}
    total = {"bytes": 4 * B * T * V, "flops": B * T * V}
    if kind == "step":
        total["bytes"] += 4 * B * g * V
        H, d = case["heads"], case["head_dim"]
        L, path = (case["prefix_lo"] + case["prefix_hi"]) / 2, 1 + case["depth"] / 2
        for n, streams in ((case["layers"] - case["msa_layers"], 0), (case["msa_layers"], g)):
            rows = T * (1 + streams)
            total["bytes"] += n * B * 4 * H * d * (L + T + T * streams + rows)
            total["flops"] += n * B * 4 * H * d * (rows * (L + path) + T * streams * (streams + 1) / 2)
    return total


def tolerance(case):
    if case["kind"] == "step":
        # probabilities and outputs are rounded to bf16, everything between is fp32; integers and cache bytes are exact
        return {"rel": 5e-3, "max": 5e-2}
    if case["kind"] == "prune" or case.get("mode") == "soft":
        return {"rel": 1e-5, "max": 1e-4}      # fp32 sums over the vocabulary
    return "exact"
