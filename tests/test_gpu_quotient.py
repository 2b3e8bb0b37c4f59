"""The epilogues' quotients (csrc/quotient.cuh) against the division, and a
SwiGLU whose gates lie on both sides of the fast path's range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from synth import device as D
from synth import workloads as W
from tests.helpers import LOGIT_TOL, Pair, run_gpu_block

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
PAIRS = 1 << 32


def _lib_build():
    import importlib.util
    path = os.path.join(os.path.dirname(HERE), "paper_2609_37617_gb300", "build.py")
    spec = importlib.util.spec_from_file_location("_as2d_build", path)
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_against_the_division(tmp_path):
    """silu_mid: every float that it takes, bit for bit.  quotient: a correctly
    rounded reciprocal and one correction leave at most one unit in the last
    place."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    b = _lib_build()
    so = tmp_path / "quotient_check.so"
    subprocess.run([b.NVCC, *b.ARCH, *b.CFLAGS, "-shared", "-o", str(so), os.path.join(HERE, "quotient_check.cu")],
                   check=True, capture_output=True)
    out = (ctypes.c_uint64 * 5)()
    assert ctypes.CDLL(str(so)).quotient_check(ctypes.c_uint64(PAIRS), out) == 0
    taken, differ, most, q_differ, q_most = out
    print(f"silu: {differ} of {taken} differ, by at most {most}; quotient: {q_differ} of {PAIRS}, by at most {q_most}")
    bits = lambda x: int(np.float32(x).view(np.uint32))
    assert taken == bits(1e30) + bits(80.0)  # 0 .. 1e30 and -0 .. -80, both ends outside
    assert differ == 0
    assert q_most <= 1


def _scales(ffn):
    """Powers of two of the gate rows: of 16 rows alike (a warp's features) in
    the first half, one by one in the second.  Gates of N(0, 0.3) become ones
    about 80, well beyond it and past 1e30, beside unscaled ones."""
    e = np.array([0, 8, 14, 105])
    i = np.arange(ffn)
    return np.where(i < ffn // 2, e[(i // 16) % 4], e[i % 4])


@pytest.mark.parametrize("rows", [[9], [17] * 4, [16] * 16], ids=lambda r: f"{sum(r)}rows")
def test_swiglu_gates_of_every_range(rows):
    """Gate rows scaled up and the columns that read them scaled down by powers
    of two: exact in bf16, so the oracle sees the same weights."""
    import torch
    import paper_2609_37617_gb300 as lib
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    cfg, cap = W.ModelConfig("gates", 2, 256, 4, 2, 64, 448, 1032), 256
    e = _scales(cfg.ffn)
    host, dev = W.host_weights(cfg, 0), D.device_weights(cfg, 0)
    for l in range(cfg.n_layers):
        for name, f in ((f"w_gate.{l}", np.exp2(e)[:, None]), (f"w_down.{l}", np.exp2(-e)[None, :])):
            v = (host[name].astype(np.uint32) << 16).view(np.float32) * f.astype(np.float32)
            host[name] = (v.view(np.uint32) >> 16).astype(np.uint16)
            dev[name] = torch.from_numpy(v).cuda().bfloat16()
            assert np.array_equal(dev[name].view(torch.int16).cpu().numpy().view(np.uint16), host[name])
    torch.cuda.synchronize()
    pair = Pair(cfg, host_weights=host)
    pair.model = lib.Model(cfg, D.weight_pointers(cfg, dev))
    rng = np.random.default_rng(0)
    lens = [int(x) for x in rng.integers(1, cap - 20, size=len(rows))]
    roots = [int(x) for x in rng.integers(0, cfg.vocab, size=len(rows))]
    cands = [[int(t) for t in rng.integers(0, cfg.vocab, size=r - 1)] for r in rows]
    st = pair.state(lens, cap, roots)
    logits = run_gpu_block(st, cfg, cands)[3]
    st.check()
    st.close()
    at = 0
    for b in range(len(rows)):
        want = pair.oracle.verify_block(pair.oracle_cache(lens[b], cap, req=b), lens[b], roots[b], cands[b])
        assert np.max(np.abs(want["logits"] - logits[at:at + rows[b]])) <= LOGIT_TOL
        at += rows[b]
