"""Instruction-suffix prefill on the GPU (as2d_prefill, App. A.1): the tiny
workload's 150 retained "audio" positions plus 50 instruction tokens
prefilled by the library, against the oracle; chunking invariance; the
first verification block after it; argument errors."""
import ctypes

import numpy as np
import pytest

import oracle
from synth import workloads as W
from tests.helpers import MARGIN_SURE, Pair, bf16_bits, compare_block, run_gpu_block

pytestmark = pytest.mark.gpu

L0, N_INSTR, CAP = 150, 50, 256


@pytest.fixture(scope="module")
def pair():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return Pair(W.TINY, seed=0)


def _bf16_f32(bits):
    return (bits.astype(np.uint32) << 16).view(np.float32)


def _prefill_gpu(pair, tokens, chunks=None):
    import torch
    st = pair.state([L0], CAP, [0])
    first = torch.full((1,), -7, dtype=torch.int32, device="cuda")
    tok_d = torch.tensor(tokens, dtype=torch.int32, device="cuda")
    if chunks is None:
        st.prefill(tok_d, first)
    else:
        s0 = 0
        for c in chunks:
            st.prefill(tok_d[s0:s0 + c], first)
            s0 += c
    torch.cuda.synchronize()
    return st, int(first.item())


def test_prefill_matches_oracle(pair):
    cfg = pair.cfg
    instr = [int(t) for t in W.instruction_tokens(cfg, N_INSTR, 0)]
    oc = pair.oracle_cache(L0, CAP)
    ofirst, margin, _ = oracle.prefill(pair.oracle, oc, L0, instr)
    st, first = _prefill_gpu(pair, instr)
    ln, rt = st.read_state()
    assert ln == [L0 + N_INSTR] and rt == [first]
    if margin > MARGIN_SURE:
        assert first == ofirst
    for l in range(cfg.n_layers):
        for gpu, ref in ((st.kc, oc.k), (st.vc, oc.v)):
            g = _bf16_f32(bf16_bits(gpu[l, 0])[:, L0:L0 + N_INSTR])
            o = _bf16_f32(ref[l][:, L0:L0 + N_INSTR])
            assert np.max(np.abs(g - o)) < 3e-2, f"layer {l}"
    st.check()

    # the first verification block after the prefill, against the oracle
    cont, _ = oracle.greedy_continuation(pair.oracle, oc, L0 + N_INSTR, ofirst, 4)
    cand = W.replace_at(cont, 2, np.random.default_rng(0), cfg.vocab)
    if first == ofirst:
        ores = pair.oracle.verify_block(oc, L0 + N_INSTR, ofirst, cand)
        n, corr, greedy, logits = run_gpu_block(st, cfg, [cand])
        compare_block(ores, logits[:5], greedy[:5], n[0], corr[0], 4)
    st.close()


@pytest.mark.parametrize("chunks", [[1] * 100, [17, 83], [64, 36], [5, 90, 5], [99, 1]])
def test_prefill_is_chunking_invariant(pair, chunks):
    """Any split of the suffix into prefill calls gives bitwise the same cache
    and first token as one call of 100 tokens (one pass):
    pathwise equivalence and batch invariance."""
    cfg = pair.cfg
    instr = [int(t) for t in W.instruction_tokens(cfg, 100, 1)]
    ref, first_ref = _prefill_gpu(pair, instr)
    st, first = _prefill_gpu(pair, instr, chunks)
    assert first == first_ref
    for l in range(cfg.n_layers):
        assert np.array_equal(bf16_bits(st.kc[l, 0])[:, :L0 + 100], bf16_bits(ref.kc[l, 0])[:, :L0 + 100])
        assert np.array_equal(bf16_bits(st.vc[l, 0])[:, :L0 + 100], bf16_bits(ref.vc[l, 0])[:, :L0 + 100])
    assert st.read_state() == ref.read_state()
    st.close()
    ref.close()


@pytest.mark.parametrize("n,chunks", [(256, [64, 64, 128]), (257, [64, 193]), (300, [129, 171]), (320, [257, 63]), (321, [321]),
                                      (513, [200, 313])])
def test_prefill_wide_passes(pair, n, chunks):
    """Passes of up to 256 rows; 1, 44 and 64 rows past a pass (two halves) and
    65; and calls that outgrow the working state of the call before them (64 ->
    128 -> 256 rows): bitwise the cache and first token of one call."""
    cfg, cap = pair.cfg, L0 + n + 4
    instr = torch_tokens(cfg, n)

    def prefill(parts):
        import torch
        st = pair.state([L0], cap, [0])
        first = torch.full((1,), -7, dtype=torch.int32, device="cuda")
        at = 0
        for c in parts:
            st.prefill(instr[at:at + c], first)
            at += c
        torch.cuda.synchronize()
        st.check()
        return st, int(first.item())

    ref, first_ref = prefill([1] * 3 + [60] * ((n - 3) // 60) + ([(n - 3) % 60] if (n - 3) % 60 else []))
    for parts in ([n], chunks):
        st, first = prefill(parts)
        assert first == first_ref and st.read_state() == ref.read_state() == ([L0 + n], [first])
        for l in range(cfg.n_layers):
            for a, b in ((st.kc, ref.kc), (st.vc, ref.vc)):
                assert np.array_equal(bf16_bits(a[l, 0])[:, :L0 + n], bf16_bits(b[l, 0])[:, :L0 + n])
        st.close()
    ref.close()


def test_prefill_graph_outlives_growth(pair):
    """A prefill captured into a graph replays after a longer call has made a
    larger working state, and a long call under capture takes the passes of
    the state there is."""
    import torch
    cfg, n = pair.cfg, 200
    instr = torch_tokens(cfg, n + 8)
    ref = pair.state([L0], L0 + 512, [0])
    first_ref = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref.prefill(instr[:8], first_ref)
    ref.prefill(instr[8:8 + n], first_ref)

    st = pair.state([L0], L0 + 512, [0])
    first = torch.zeros(1, dtype=torch.int32, device="cuda")
    st.prefill(instr[:8], first)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        st.prefill(instr[8:8 + n], first, stream=side.cuda_stream)
    torch.cuda.synchronize()
    st.rollback([L0], [0])
    st.prefill(instr[:n], first)  # eager: makes the larger state
    st.rollback([L0 + 8], [0])
    graph.replay()
    torch.cuda.synchronize()
    st.check()
    assert int(first.item()) == int(first_ref.item())
    assert st.read_state() == ref.read_state()
    for l in range(cfg.n_layers):
        for a, b in ((st.kc, ref.kc), (st.vc, ref.vc)):
            assert np.array_equal(bf16_bits(a[l, 0])[:, :L0 + 8 + n], bf16_bits(b[l, 0])[:, :L0 + 8 + n])
    st.close()
    ref.close()


@pytest.mark.parametrize("mode", ["relaxed", "thread_local", "global"])
def test_first_prefill_under_capture(pair, mode):
    """The first prefill of a state, captured: the graph holds kernels alone, so
    the working state does not wait for a replay to be cleared, and calls before
    the first replay, replays and calls after it give bitwise what a fresh state
    gives."""
    import torch
    cfg, n = pair.cfg, 100
    instr = torch_tokens(cfg, n)
    ref = pair.state([L0], L0 + 256, [0])
    first_ref = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref.prefill(instr, first_ref)
    torch.cuda.synchronize()

    st = pair.state([L0], L0 + 256, [0])
    first = torch.zeros(1, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=side, capture_error_mode=mode):
        st.prefill(instr, first, stream=side.cuda_stream)
    assert set(graph_node_types(graph.raw_cuda_graph())) == {0}  # cudaGraphNodeTypeKernel

    def check():
        torch.cuda.synchronize()
        st.check()
        assert int(first.item()) == int(first_ref.item())
        assert st.read_state() == ref.read_state()
        for l in range(cfg.n_layers):
            for a, b in ((st.kc, ref.kc), (st.vc, ref.vc)):
                assert np.array_equal(bf16_bits(a[l, 0])[:, :L0 + n], bf16_bits(b[l, 0])[:, :L0 + n])
        first.fill_(-7)
        st.rollback([L0], [0])

    st.rollback([L0], [0])  # (the captured call raised the host's bound of the length)
    st.prefill(instr[:64], first)  # the state that the captured call made, before any replay
    st.prefill(instr[64:], first)
    check()
    graph.replay()
    check()
    st.prefill(instr, first)
    check()
    st.close()
    ref.close()


# passes of 150 + 150 and of 256 + 256 + 88 rows
@pytest.mark.parametrize("n,bad,kept", [(300, [299], [(0, 150)]), (300, [0], [(150, 300)]), (300, [3, 200], []),
                                        (600, [512], [(0, 512)]), (600, [256, 520], [(0, 256)]),
                                        (600, [255, 599], [(256, 512)]), (600, [10, 500], [(512, 600)])])
def test_prefill_root_after_flagged_pass(pair, n, bad, kept):
    """Bad token ids flag their passes: the state is the one after the rows of
    the other passes alone, its root the greedy token after the last of them."""
    import torch
    import paper_2609_37617_gb300 as lib
    instr = torch_tokens(pair.cfg, n)
    broken = instr.clone()
    broken[bad] = torch.tensor([pair.cfg.vocab, -1][:len(bad)], dtype=torch.int32, device="cuda")
    first = torch.zeros(1, dtype=torch.int32, device="cuda")
    ref = pair.state([L0], L0 + 700, [7])
    for a, b in kept:
        ref.prefill(instr[a:b], first)
    for warm in (False, True):  # the second time after a call that kept every pass
        st = pair.state([L0], L0 + 700, [7])
        if warm:
            st.prefill(instr, first)
            st.rollback([L0], [7])
        st.prefill(broken, first)
        torch.cuda.synchronize()
        with pytest.raises(lib.AS2DError):
            st.check()
        assert st.read_state() == ref.read_state()
        assert (int(first.item()) == -1) == (max(bad) >= {300: 150, 600: 512}[n])
        st.close()
    ref.close()


@pytest.mark.parametrize("n", [40, 100, 300])
def test_prefill_recovers_from_expired_waits(pair, n):
    """A prefill whose kernels' waits run out reports it; the next one, from
    the restored prefix, gives the bits of one before."""
    import torch
    import paper_2609_37617_gb300 as lib
    instr = torch_tokens(pair.cfg, n)
    st = pair.state([L0], L0 + 512, [0])
    first = torch.zeros(1, dtype=torch.int32, device="cuda")

    def prefill():
        st.prefill(instr, first)
        torch.cuda.synchronize()
        got = (int(first.item()), bf16_bits(st.kc)[:, 0, :, :L0 + n], bf16_bits(st.vc)[:, 0, :, :L0 + n])
        st.rollback([L0], [0])
        return got

    want = prefill()
    st.check()
    for limit in (0, 2000, 8000, 16000, 24000):
        st.set_wait_limit(limit)
        for _ in range(3):
            prefill()
        try:
            st.check()
            assert limit > 0, "a limit of 0 runs out"
        except lib.AS2DError as e:
            assert e.status == lib.AS2D_ERR_DEVICE and "timed out" in str(e)
        st.set_wait_limit(2_000_000_000)
        for a, b in zip(prefill(), want):
            assert np.array_equal(a, b), limit
        st.check()
    st.close()


def graph_node_types(graph):
    """cudaGraphNodeType of every node of a cudaGraph_t."""
    rt = ctypes.CDLL("libcudart.so.13")
    n = ctypes.c_size_t(0)
    assert rt.cudaGraphGetNodes(ctypes.c_void_p(graph), None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert rt.cudaGraphGetNodes(ctypes.c_void_p(graph), nodes, ctypes.byref(n)) == 0
    kind, kinds = ctypes.c_int(), []
    for node in nodes:
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    return kinds


def torch_tokens(cfg, n):
    import torch
    return torch.tensor([int(t) for t in W.instruction_tokens(cfg, n, 2)], dtype=torch.int32, device="cuda")


def test_prefill_argument_errors(pair):
    import torch
    import paper_2609_37617_gb300 as lib
    tok = torch.zeros(4, dtype=torch.int32, device="cuda")
    st = pair.state([L0], L0 + 3, [0])
    with pytest.raises(lib.AS2DError) as e:
        st.prefill(tok)                      # L0 + 4 > capacity
    assert e.value.status == lib.AS2D_ERR_CAPACITY
    assert lib._lib.as2d_prefill(st.handle, tok.data_ptr(), 0, None, None) == lib.AS2D_ERR_INVALID_ARG
    st.close()
    st2 = pair.state([L0, L0], CAP, [0, 0])
    with pytest.raises(lib.AS2DError) as e:
        st2.prefill(tok)
    assert e.value.status == lib.AS2D_ERR_UNSUPPORTED
    st2.close()
    bad = torch.full((3,), cfg_vocab(pair) + 5, dtype=torch.int32, device="cuda")
    st3 = pair.state([L0], CAP, [0])
    st3.prefill(bad)
    with pytest.raises(lib.AS2DError) as e:
        st3.check()
    assert e.value.status == lib.AS2D_ERR_DEVICE
    st3.close()


def cfg_vocab(pair):
    return pair.cfg.vocab
