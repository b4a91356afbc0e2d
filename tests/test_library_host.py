"""Host-side checks of the C-ABI library that need no GPU: it loads, exports every symbol the
header declares, builds tree descriptors, and rejects bad arguments before launching anything."""
import ctypes as C
import os
import re
import subprocess

import numpy as np
import pytest

from paper_2402_11131_b200 import api, build

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GOLDEN = os.path.join(os.path.dirname(__file__), "golden")


@pytest.fixture(scope="module")
def lib():
    build.build()
    return api.lib()


def test_every_declared_symbol_is_exported(lib):
    header = open(os.path.join(ROOT, "include", "ss_msa.h")).read()
    header = re.sub(r"/\*.*?\*/", "", header, flags=re.S)
    declared = set(re.findall(r"\b(ss_[a-z_]+)\s*\(", header))
    assert declared == set(api.EXPORTS)
    for name in declared:
        assert getattr(lib, name) is not None
    assert lib.ss_version() >= 100


def test_struct_sizes_match_the_header(lib):
    assert C.sizeof(api.TreeDesc) == 16 + 4 * 64 + 4 * 64 + 8 * 64
    assert C.sizeof(api.CacheLayout) == 40
    assert C.sizeof(api.AttnParams) == 24 + 8 * 8 + 3 * 8 + 8 * 8 + 8      # ... + flags (padded to 8)


def test_tree_build_paper_mask_example(lib):
    """Ancestor words of the App. A mask example: 'early' sees parameter, efficient and itself."""
    parent, vis = None, {}
    for line in open(os.path.join(GOLDEN, "mask_example.txt")):
        line = line.strip()
        if not line or line.startswith("#"):
            continue
        k, v = line.split(":")
        if k == "parent":
            parent = [int(x) for x in v.split()]
        else:
            vis[int(k)] = {int(x) for x in v.split()}
    d = api.ss_tree_build(parent, 2)
    assert d.n_nodes == 5 and d.max_depth == 2 and d.gamma == 2
    for t in range(5):
        assert {a for a in range(64) if (d.anc_mask[t] >> a) & 1} == vis[t]
    assert list(d.depth[:5]) == [0, 1, 1, 2, 2]
    assert list(d.parent[:6]) == parent + [-1]


def test_tree_build_matches_oracle_on_random_trees(lib, oracle):
    from paper_2402_11131_b200 import workloads as W
    rng = np.random.default_rng(1)
    for _ in range(50):
        T = int(rng.integers(1, 65))
        parent = W.draw_tree(rng, T, 6, "uniform_parent")
        d = api.ss_tree_build(parent, 0)
        depth, anc, md = oracle.tree_build(parent)
        assert d.max_depth == md and list(d.depth[:T]) == list(depth)
        for t in range(T):
            assert d.anc_mask[t] == sum(1 << a for a in range(T) if anc[t, a])


def test_tree_build_errors(lib):
    for bad, code in (([0, 0], api.SS_ERR_BAD_TREE), ([-1, 1], api.SS_ERR_BAD_TREE), ([-1, 0, 2], api.SS_ERR_BAD_TREE),
                      ([-1, -1], api.SS_ERR_BAD_TREE), ([], api.SS_ERR_BAD_TREE),
                      ([-1] + [0] * 64, api.SS_ERR_UNSUPPORTED)):
        with pytest.raises(api.SsError) as e:
            api.ss_tree_build(bad, 0)
        assert e.value.status == code
    with pytest.raises(api.SsError) as e:
        api.ss_tree_build([-1], api.SS_MAX_GAMMA + 1)
    assert e.value.status == api.SS_ERR_UNSUPPORTED
    out = api.TreeDesc()
    assert lib.ss_tree_build(None, 1, 0, C.byref(out)) == api.SS_ERR_INVALID_ARG


def _fake_params(**kw):
    """ss_attn_params with plausible, 16-byte aligned but never dereferenced pointers."""
    p = api.AttnParams()
    p.batch, p.n_heads, p.head_dim, p.gamma, p.max_nodes, p.sm_scale = 1, 2, 64, 3, 6, 1.0
    for f in ("q_main", "o_main", "q_spec", "k_spec", "v_spec", "o_spec", "k_cache", "v_cache", "kv_start",
              "kv_len", "trees", "workspace"):
        setattr(p, f, 0x10000)
    p.kv_slot_stride, p.kv_head_stride, p.kv_total_slots = 128, 64, 128
    p.workspace_bytes = 1 << 40
    for k, v in kw.items():
        setattr(p, k, v)
    return p


def test_attention_rejects_bad_arguments_before_any_launch(lib):
    ok_ws = lib.ss_msa_attention_workspace_bytes(C.byref(_fake_params()))
    assert ok_ws > 0
    cases = [
        (dict(head_dim=96), api.SS_ERR_UNSUPPORTED),
        (dict(max_nodes=65), api.SS_ERR_UNSUPPORTED),
        (dict(gamma=5), api.SS_ERR_UNSUPPORTED),
        (dict(batch=0), api.SS_ERR_INVALID_ARG),
        (dict(q_main=None), api.SS_ERR_INVALID_ARG),
        (dict(q_spec=None), api.SS_ERR_INVALID_ARG),
        (dict(k_cache=0x10008), api.SS_ERR_INVALID_ARG),      # misaligned
        (dict(kv_slot_stride=100), api.SS_ERR_INVALID_ARG),   # not a multiple of 8 elements
        (dict(kv_slot_stride=32), api.SS_ERR_INVALID_ARG),    # rows would overlap
        (dict(sm_scale=float("nan")), api.SS_ERR_INVALID_ARG),
        (dict(workspace_bytes=ok_ws - 1), api.SS_ERR_WORKSPACE),
        (dict(workspace=None), api.SS_ERR_INVALID_ARG),
    ]
    for kw, code in cases:
        assert lib.ss_msa_attention(C.byref(_fake_params(**kw)), None) == code, kw
    assert lib.ss_msa_attention(None, None) == api.SS_ERR_INVALID_ARG


@pytest.mark.parametrize("head_dim", [64, 80, 128])
def test_attention_workspace_follows_from_the_shapes_not_from_the_slab(lib, head_dim):
    """One answer for every slab a cache may grow to, also while there is none yet."""
    for T, gamma in ((1, 0), (12, 0), (12, 1), (16, 3), (33, 0), (64, 0), (40, 2), (64, 4)):
        for batch, heads in ((1, 2), (1, 32), (5, 13), (3, 32), (16, 32)):
            answers = {lib.ss_msa_attention_workspace_bytes(C.byref(_fake_params(
                batch=batch, n_heads=heads, head_dim=head_dim, gamma=gamma, max_nodes=T, kv_total_slots=slots)))
                for slots in (0, 1, 100, 512, 1024, 2048, 4096, 1 << 20, 1 << 30)}
            assert len(answers) == 1 and min(answers) >= 256, (T, gamma, batch, heads, answers)


def test_verify_and_compact_reject_bad_arguments_before_any_launch(lib):
    need = lib.ss_tree_verify_workspace_bytes(2, 6, 512)
    assert need >= 256 + 2 * 6 * 8
    a = 0x10000
    assert lib.ss_tree_verify(a, a, a, 2, 6, 512, a, a, a, a, None, a, need - 1, None) == api.SS_ERR_WORKSPACE
    assert lib.ss_tree_verify(None, a, a, 2, 6, 512, a, a, a, a, None, a, need, None) == api.SS_ERR_INVALID_ARG
    assert lib.ss_tree_verify(a, a, a, 2, 65, 512, a, a, a, a, None, a, 1 << 30, None) == api.SS_ERR_UNSUPPORTED
    assert lib.ss_tree_verify(a, a, a, 0, 6, 512, a, a, a, a, None, a, need, None) == api.SS_ERR_INVALID_ARG
    lo = api.CacheLayout()
    lo.n_layers, lo.n_heads, lo.head_dim, lo.layer_stride, lo.slot_stride, lo.head_stride = 2, 2, 64, 8192, 128, 64
    assert lib.ss_kv_compact(None, a, C.byref(lo), 1, a, a, a, a, a, None) == api.SS_ERR_INVALID_ARG
    lo.head_dim = 4
    assert lib.ss_kv_compact(a, a, C.byref(lo), 1, a, a, a, a, a, None) == api.SS_ERR_UNSUPPORTED
    lo.head_dim = 64
    assert lib.ss_kv_compact(a + 8, a, C.byref(lo), 1, a, a, a, a, a, None) == api.SS_ERR_INVALID_ARG


def test_error_strings(lib):
    assert lib.ss_error_string(0) == b"ok"
    assert b"workspace" in lib.ss_error_string(api.SS_ERR_WORKSPACE)


@pytest.mark.parametrize("kernel", ["small", "few", "half"])
def test_waits_of_heads_of_at_most_64_rows_keep_the_bound_of_the_workspace_header(kernel):
    """Read from the source, since no run can make a barrier's wait last: every wait of the kernels that such heads take
    goes by the bound in the control block, which is loaded from word 1 of the workspace."""
    src = open(os.path.join(ROOT, "paper_2402_11131_b200", "csrc", "ss_attention_%s.cuh" % kernel)).read()
    waits = re.findall(r"\b(mbar_wait\w*)\((.*?status)\)", src)
    assert len(waits) > 0
    for name, args in waits:
        assert name not in ("mbar_wait", "mbar_wait_warp", "mbar_wait_slow"), args       # these have the default bound
        assert "abort" not in args or "wait_limit" in args, (name, args)
    assert '"l"(a.status + 1)' in src and "c.wait_limit) = lim" in src


class _Stream:
    cuda_stream = 0                          # stands for a torch.cuda.Stream where there is no GPU


def test_binding_refuses_what_is_not_the_call_s_structure(lib):
    """As ctypes does: another structure is an ArgumentError, what is no ctypes object a TypeError; nothing is read."""
    class Derived(api.AttnParams):
        pass

    for call, own in ((lambda p: api.ss_msa_attention(p, _Stream()), api.AttnParams),
                      (lambda p: api.ss_kv_compact(None, None, p, torch.zeros(1), None, None, None, None, _Stream()), api.CacheLayout)):
        for other in (api.TreeDesc(), api.CacheLayout() if own is api.AttnParams else api.AttnParams(), C.c_int32(), C.pointer(own())):
            with pytest.raises(C.ArgumentError):
                call(other)
        for other in (None, b"\0" * 512, bytearray(512), np.zeros(64), 0):
            with pytest.raises(TypeError):
                call(other)
        with pytest.raises(api.SsError) as e:                # an empty structure reaches the library
            call(own())
        assert e.value.status == api.SS_ERR_INVALID_ARG
    with pytest.raises(api.SsError):
        api.ss_msa_attention(Derived(), _Stream())


def test_per_step_calls_go_to_the_library_that_was_loaded(lib, tmp_path):
    """A library under another path (a tracing build, say) gets every call, those that the binding's native part makes too."""
    names = [n for n in api.EXPORTS if n != "ss_error_string"]
    src = "".join("int %s() { return -77; }\n" % n for n in names) + 'const char* ss_error_string() { return "other"; }\n'
    (tmp_path / "other.c").write_text(src)
    other = str(tmp_path / "libother.so")
    subprocess.check_call(["gcc", "-w", "-shared", "-fPIC", "-o", other, str(tmp_path / "other.c")])
    with pytest.raises(api.SsError) as e:                    # (the native part is set up with the library as it is)
        api.ss_msa_attention(api.AttnParams(), _Stream())
    assert e.value.status == api.SS_ERR_INVALID_ARG
    x, own = torch.zeros((1, 1, 1, 1)), api._lib
    try:
        api._LIB_PATH, api._lib, api._native, path = other, None, None, api._LIB_PATH
        for call in (lambda: api.ss_msa_attention(api.AttnParams(), _Stream()),
                     lambda: api.ss_tree_verify(x[0], x, x, x, x, x, x, x, x, _Stream()),
                     lambda: api.ss_tree_verify_soft(x[0], x, x, 0.1, 0.1, x, x, x, x, x, x, x, _Stream()),
                     lambda: api.ss_tree_verify_sampled(x[0], x, x, x, 1, x, x, x, x, x, x, _Stream()),
                     lambda: api.ss_tree_prune(x[0], x, x, 0.1, x, x, x, x, x, x, _Stream()),
                     lambda: api.ss_next_draft(x, x, x, 1, 1, x, x, x, _Stream()),
                     lambda: api.ss_kv_compact(x, x, api.CacheLayout(), x, x, x, x, x, _Stream()),
                     lambda: api.ss_stream_insert(x[0, 0], x, x, _Stream()), lambda: api.ss_value_rotate(x[0, 0], x, 0.1, _Stream()),
                     lambda: api.ss_tree_build([-1], 0)):
            with pytest.raises(api.SsError) as e:
                call()
            assert e.value.status == -77
    finally:
        api._LIB_PATH, api._lib, api._native = path, own, None
    with pytest.raises(api.SsError) as e:
        api.ss_msa_attention(api.AttnParams(), _Stream())
    assert e.value.status == api.SS_ERR_INVALID_ARG


def _draft_plan(tmp_path, body):
    """The output of a program that includes the next draft's host rules."""
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text('#include <cstdio>\n#include "ss_draft_plan.h"\nint main() {\n%s\nreturn 0; }\n' % body)
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", build.CSRC, str(src), "-o", str(exe)])
    return subprocess.check_output([str(exe)], text=True).split()


def test_next_draft_cluster_sizes(tmp_path):
    """More than 8 CTAs where a segment of 8 spans more than one batch of 16384 words (rows of a vocabulary that is no multiple of four begin up
    to three words after an aligned address), for at most six sequences of at least two rows."""
    cases = [((1, 4, 32000), 8), ((1, 4, 32768), 8), ((1, 4, 32769), 16), ((1, 4, 32766), 16), ((1, 4, 32764), 8), ((6, 4, 51201), 16),
             ((7, 4, 51201), 8), ((1, 3, 32768), 6), ((1, 3, 32769), 12), ((1, 3, 50257), 12), ((6, 3, 51200), 12), ((16, 3, 51200), 6),
             ((1, 2, 65536), 8), ((1, 2, 65540), 16), ((1, 1, 131072), 8), ((1, 1, 131100), 8), ((1, 1, 262144), 8), ((1, 4, 4095), 4), ((1, 1, 37), 1)]
    got = _draft_plan(tmp_path, "\n".join('printf("%%d\\n", %d * ss::draft_ctas(%d, %d, %d, ss::kMaxClusterCtas));' % (c[1], *c) for c, _ in cases))
    assert [int(x) for x in got] == [want for _, want in cases]


def test_next_draft_falls_back_to_clusters_that_can_be_placed(tmp_path):
    """Where the device says that 12 CTAs do not fit, or the launch does, 6 take the sequence; an error of these is an error."""
    body = """
    const auto run = [](int vocab, bool fits, int limit) {          // a device that says `fits` and launches up to `limit` CTAs
        int asked = 0;
        const int err = ss::launch_draft(1, 3, vocab, [&](int ctas) { asked = ctas; return fits; },
                                         [&](int n) { std::printf("launch:%d ", 3 * n); return 3 * n <= limit ? 0 : 7; });
        std::printf("asked:%d error:%d\\n", asked, err);
    };
    run(51200, true, 16); run(51200, false, 16); run(51200, true, 8); run(51200, true, 0); run(32000, false, 16); run(32000, true, 0);"""
    assert _draft_plan(tmp_path, body) == ["launch:12", "asked:12", "error:0", "launch:6", "asked:12", "error:0", "launch:12", "launch:6", "asked:12",
                                           "error:0", "launch:12", "launch:6", "asked:12", "error:7", "launch:6", "asked:0", "error:0", "launch:6",
                                           "asked:0", "error:7"]
