"""GPU checks at the sizes where a kernel variant or a branch of a dispatch can go wrong, against the fp64 oracle.

Tolerances are those of the parity tests: O max abs 1e-2 / mean abs 1e-3, LSE 1e-3, gradients 2e-2 relative.
"""
import numpy as np
import pytest

from oracle import attention_ref as A
from paper_2602_21788_b200 import build, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

f64 = synth.bf16_bits_to_f64


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    torch.cuda.set_device(0)


def _wl(lens, degs, hq, hkv, D, seed=0):
    return synth.Workload(name="case", seed=seed, seqlens=np.asarray(lens, np.int32),
                          cp_degrees=np.asarray(degs, np.int32), hq=hq, hkv=hkv, head_dim=D)


def _rel(got, ref):
    return np.linalg.norm(np.asarray(got, np.float64) - ref) / max(np.linalg.norm(ref), 1e-30)


def _check(w, **kw):
    from paper_2602_21788_b200.runner import run_fwd_bwd
    q, k, v, do = w.tensors()
    res = run_fwd_bwd(w, q, k, v, do, fused=True, **kw)
    o_ref, lse_ref = A.attention_fwd_packed(f64(q), f64(k), f64(v), w.cu_seqlens)
    e = np.abs(res["o_f32"] - o_ref)
    assert e.max() <= 1e-2 and e.mean() <= 1e-3 and np.abs(res["lse"] - lse_ref).max() <= 1e-3
    for name, ref in zip(("dq", "dk", "dv"), A.attention_bwd_packed(f64(q), f64(k), f64(v), f64(do), w.cu_seqlens)):
        assert _rel(res[name], ref) <= 2e-2, name


@pytest.mark.parametrize("lens,hq,hkv,kv_pass", [
    ([127, 130, 1, 383], 4, 2, None),     # sequences that start inside a block of 128 packed rows; last block of 1 row
    ([128, 256], 2, 1, None),             # no partial last block
    ([200, 55], 6, 3, 2),                 # last block of 127 rows; passes of 2 + 1 KV heads
    ([640, 65], 12, 4, 1),
])
def test_backward_d64_blocked_dq_accumulator(lens, hq, hkv, kv_pass):
    _check(_wl(lens, [1] * len(lens), hq, hkv, 64, seed=11), kv_heads_per_bwd_pass=kv_pass)
