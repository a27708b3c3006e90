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


def _fused(plan, q, k, v, hq, stream):
    from paper_2602_21788_b200 import fcp
    o = torch.empty_like(q)
    lse = torch.empty(q.shape[:2], dtype=torch.float32, device="cuda")
    fcp.fcp_attn_fwd_fused(plan, q, k, v, o, lse, stream=stream.cuda_stream)
    return o, lse


@pytest.mark.parametrize("threads", [1, 3])
def test_plan_blocks_are_handed_on_only_after_the_work_that_reads_them(threads):
    """Plans that are dropped right after their calls were queued, with the next plan (of another batch) uploaded at
    once: from one thread over two streams, and from several threads with a stream each."""
    import threading
    from paper_2602_21788_b200 import fcp
    hq, hkv, D = 8, 2, 128
    batches = [[3000, 1000, 96], [128] * 32, [4096], [700, 650, 1300, 1446]]
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn((4096, h, D), dtype=torch.bfloat16, device="cuda", generator=g) for h in (hq, hkv, hkv))
    main = torch.cuda.current_stream()
    want = {}
    for i, lens in enumerate(batches):
        plan = fcp.Plan(lens, [1] * len(lens), hq, hkv, D).upload()
        want[i] = _fused(plan, q, k, v, hq, main)
    torch.cuda.synchronize()
    got, failed = [], []

    def work(t):
        try:
            streams = [torch.cuda.Stream(), torch.cuda.Stream()]
            busy = torch.zeros(1 << 27, device="cuda")
            torch.cuda.synchronize()
            for r in range(12):
                i, st = (r + t) % len(batches), streams[r & 1]
                with torch.cuda.stream(st):
                    busy.add_(1.0)                      # keeps the stream busy: the calls below stay queued for a while
                    plan = fcp.Plan(batches[i], [1] * len(batches[i]), hq, hkv, D).upload(st.cuda_stream)
                    got.append((i, _fused(plan, q, k, v, hq, st)))
                del plan
        except Exception as e:                          # a thread's failure must reach the test
            failed.append(e)

    ts = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    assert len(got) == 12 * threads
    for i, (o, lse) in got:
        assert torch.equal(o, want[i][0]) and torch.equal(lse, want[i][1]), i
    fcp.fcp_release_cached()
    plan = fcp.Plan(batches[0], [1, 1, 1], hq, hkv, D).upload()
    o, lse = _fused(plan, q, k, v, hq, main)
    torch.cuda.synchronize()
    assert torch.equal(o, want[0][0]) and torch.equal(lse, want[0][1])


@pytest.mark.parametrize("lens,hq,hkv,D", [
    ([900, 130], 2, 1, 128),                        # a single slice
    ([12000, 7000, 1001], 6, 3, 64),                # odd number of KV heads: one pass each, two kernel lanes
    ([5000, 9000, 6000, 4000], 8, 1, 128),          # one KV head: runs of sequences only
    ([11000, 8000, 1500, 6000], 20, 10, 128),       # passes of two KV heads and runs
    ([19100, 300, 129], 8, 4, 128),                 # long enough for its copies to be cut by heads alone, two lanes
    ([24700, 300], 64, 64, 64),                     # the same with slices that fill the chip: one lane
])
def test_host_entry_point_slices(lens, hq, hkv, D):
    """fcp_attn_fwd_bwd_host == the device calls, bit for bit where those are deterministic, on a first and a second call."""
    from paper_2602_21788_b200 import fcp
    from paper_2602_21788_b200.runner import DeviceState
    w = _wl(lens, [1] * len(lens), hq, hkv, D, seed=13)
    ds = DeviceState(w, *w.device_tensors(), partials=False)
    ds.forward_fused()
    ds.backward()
    torch.cuda.synchronize()
    ds.check_status()
    pin = lambda t: t.cpu().pin_memory()
    ins = [pin(t) for t in (ds.q, ds.k, ds.v, ds.do)]
    nbytes = ds.plan.host_workspace_bytes()
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        out = [torch.zeros(t.shape, dtype=t.dtype).pin_memory() for t in (ds.o, ds.lse, ds.dq, ds.dk, ds.dv)]
        fcp.fcp_attn_fwd_bwd_host(ds.plan, *ins, *out, ws, nbytes, torch.cuda.current_stream().cuda_stream)
        assert ds.plan.device_status()[0] == 0
        for got, ref in zip((out[0], out[1], out[3], out[4]), (ds.o, ds.lse, ds.dk, ds.dv)):
            assert torch.equal(got, ref.cpu())
        a, b = out[2].float(), ds.dq.float().cpu()
        assert (a - b).norm() <= 1e-2 * b.norm()


@pytest.mark.parametrize("lens,hq,hkv,D", [
    ([1000], 2, 1, 128),                 # 8 items on 148 SMs: the Q tiles of a unit are items of their own
    ([129, 128, 1], 3, 3, 64),           # units with one Q tile
    ([2560] * 9 + [70], 16, 2, 64),      # more items than SMs: both tiles of a unit together
])
def test_forward_with_split_and_whole_units(lens, hq, hkv, D):
    _check(_wl(lens, [1] * len(lens), hq, hkv, D, seed=17))


@pytest.mark.parametrize("hq", [65535, 65600])     # around the limit of a grid's second dimension
def test_backward_of_more_query_heads_than_a_grid_dimension_holds(hq):
    from paper_2602_21788_b200.runner import run_fwd_bwd
    w = _wl([2, 1], [1, 1], hq, 1, 64, seed=19)
    q, k, v, do = w.tensors()
    res = run_fwd_bwd(w, q, k, v, do, fused=True, want_o_f32=False)
    some = np.r_[0:3, hq - 67:hq - 62, hq - 2:hq]  # query heads that share the one KV head are independent
    dq_ref, _, _ = A.attention_bwd_packed(f64(q[:, some]), f64(k), f64(v), f64(do[:, some]), w.cu_seqlens)
    assert _rel(res["dq"][:, some], dq_ref) <= 2e-2


@pytest.mark.parametrize("n_seq", [3, 1500, 3200])    # one piece of the upload buffer, several, and a block that is not kept
def test_upload_in_pieces(n_seq):
    """A sequence's results do not depend on where its rows lie in the tables: span plans, whose tables grow with the tokens."""
    from paper_2602_21788_b200 import fcp
    kinds = [(500, [(10, 200), (210, 499)]), (129, []), (700, [(0, 700)])]
    some = sorted({0, 1, 2, n_seq // 2, n_seq - 2, n_seq - 1})
    lens = [kinds[i % 3][0] for i in range(n_seq)]
    cu = np.r_[0, np.cumsum(lens)]
    g = torch.Generator(device="cuda").manual_seed(29)
    q, k, v = (torch.randn((int(cu[-1]), 1, 64), dtype=torch.bfloat16, device="cuda", generator=g) for _ in range(3))
    st = torch.cuda.current_stream()
    plan = fcp.Plan(lens, [1] * n_seq, 1, 1, 64, spans=[kinds[i % 3][1] for i in range(n_seq)]).upload()
    small = fcp.Plan([5, 129], [1, 1], 1, 1, 64).upload()          # another one's tables go through the same buffer
    o, lse = _fused(plan, q, k, v, 1, st)
    _fused(small, q[:134], k[:134], v[:134], 1, st)
    assert plan.device_status()[0] == 0
    for i in some:
        a, b = int(cu[i]), int(cu[i + 1])
        alone = fcp.Plan([lens[i]], [1], 1, 1, 64, spans=[kinds[i % 3][1]]).upload()
        o1, lse1 = _fused(alone, *(t[a:b].contiguous() for t in (q, k, v)), 1, st)
        assert torch.equal(o[a:b], o1) and torch.equal(lse[a:b], lse1), i


@pytest.mark.parametrize("n_seq", [2, 300])     # tables in blocks of 64 KB: eight are kept; of 8 MB (spans): four
def test_more_plans_in_flight_than_blocks_are_kept(n_seq):
    """Twelve plans with queued work are dropped at once, so the list overflows with blocks in use and the uploads that follow
    find it full of them; results must come from the plan's own tables throughout."""
    from paper_2602_21788_b200 import fcp
    batches = [[2000 - 100 * i] + [2000] * (n_seq - 2) + [2000 + 100 * i] for i in range(12)]
    g = torch.Generator(device="cuda").manual_seed(31)
    q, k, v = (torch.randn((2000 * n_seq, 1, 64), dtype=torch.bfloat16, device="cuda", generator=g) for _ in range(3))
    st = torch.cuda.current_stream()
    make = lambda lens: fcp.Plan(lens, [1] * n_seq, 1, 1, 64, spans=[[(0, 500)]] * n_seq).upload()
    fcp.fcp_release_cached()
    want = []
    for lens in batches:
        want.append(_fused(make(lens), q, k, v, 1, st))
        torch.cuda.synchronize()
    busy = torch.zeros(1 << 28, device="cuda")
    got = []
    for _ in range(2):
        for _ in range(40):
            busy.add_(1.0)                              # the calls below stay queued for about 15 ms
        plans = [make(lens) for lens in batches]
        got += [_fused(plan, q, k, v, 1, st) for plan in plans]
        del plans
        got += [_fused(make(lens), q, k, v, 1, st) for lens in batches]
    torch.cuda.synchronize()
    for i, (o, lse) in enumerate(got):
        assert torch.equal(o, want[i % 12][0]) and torch.equal(lse, want[i % 12][1]), i


SHORT = [1, 2, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129]


@pytest.mark.parametrize("D,hq,hkv", [(64, 4, 2), (128, 2, 2)])
@pytest.mark.parametrize("spans", [False, True])
def test_short_sequences(D, hq, hkv, spans):
    """Lengths around 32, 64, 96 and 128, where column blocks, key rows and whole warps of a tile have nothing to do."""
    from oracle import span_attention_ref as S
    if not spans:
        return _check(_wl(SHORT + SHORT[::-1], [1] * (2 * len(SHORT)), hq, hkv, D, seed=37))
    from paper_2602_21788_b200.runner import run_fwd_bwd
    w = _wl(SHORT, [1] * len(SHORT), hq, hkv, D, seed=41)
    w.spans = [[] if n < 31 else [(0, 30)] if n < 64 else [(3, 33), (40, n)] for n in SHORT]
    q, k, v, do = w.tensors()
    res = run_fwd_bwd(w, q, k, v, do, fused=True)
    o_ref, lse_ref = S.span_attention_fwd_packed(f64(q), f64(k), f64(v), w.cu_seqlens, w.spans)
    e = np.abs(res["o_f32"] - o_ref)
    assert e.max() <= 1e-2 and e.mean() <= 1e-3 and np.abs(res["lse"] - lse_ref).max() <= 1e-3
    refs = S.span_attention_bwd_packed(f64(q), f64(k), f64(v), f64(do), w.cu_seqlens, w.spans)
    for name, ref in zip(("dq", "dk", "dv"), refs):
        assert _rel(res[name], ref) <= 2e-2, name


@pytest.mark.parametrize("D,deg", [(64, 1), (64, 5), (128, 3)])
def test_partial_path_of_short_sequences(D, deg):
    """Items of at most 64 keys, diagonal and full ones, and longer ones."""
    from paper_2602_21788_b200.runner import run_fwd_bwd
    lens = SHORT + [200, 331, 640]
    w = _wl(lens, [deg] * len(lens), 4, 2, D, seed=43)
    q, k, v, _ = w.tensors()
    res = run_fwd_bwd(w, q, k, v)
    o_ref, lse_ref = A.attention_fwd_packed(f64(q), f64(k), f64(v), w.cu_seqlens)
    e = np.abs(res["o_f32"] - o_ref)
    assert e.max() <= 1e-2 and e.mean() <= 1e-3 and np.abs(res["lse"] - lse_ref).max() <= 1e-3


@pytest.mark.parametrize("lens,hq,hkv,D", [([700, 130], 4, 2, 64), ([9000, 12000, 7000, 1001], 8, 4, 128)])
def test_host_entry_point_with_pageable_buffers(lens, hq, hkv, D):
    """One plan's calls with page-locked and pageable buffers in turn, and with one pageable buffer among page-locked ones."""
    from paper_2602_21788_b200 import fcp
    from paper_2602_21788_b200.runner import DeviceState
    w = _wl(lens, [1] * len(lens), hq, hkv, D, seed=47)
    ds = DeviceState(w, *w.device_tensors(), partials=False)
    ds.forward_fused()
    ds.backward()
    torch.cuda.synchronize()
    nbytes = ds.plan.host_workspace_bytes()
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    host = [t.cpu() for t in (ds.q, ds.k, ds.v, ds.do)]
    for locked in ("all", "none", "but dk", "all"):
        pin = lambda i, t: t.pin_memory() if locked == "all" or (locked == "but dk" and i != 7) else t
        ins = [pin(i, t) for i, t in enumerate(host)]
        out = [pin(4 + i, torch.zeros(t.shape, dtype=t.dtype)) for i, t in enumerate((ds.o, ds.lse, ds.dq, ds.dk, ds.dv))]
        fcp.fcp_attn_fwd_bwd_host(ds.plan, *ins, *out, ws, nbytes, torch.cuda.current_stream().cuda_stream)
        assert ds.plan.device_status()[0] == 0
        for got, ref in zip((out[0], out[1], out[3], out[4]), (ds.o, ds.lse, ds.dk, ds.dv)):
            assert torch.equal(got, ref.cpu()), locked
        assert (out[2].float() - ds.dq.float().cpu()).norm() <= 1e-2 * ds.dq.float().norm().item()


@pytest.mark.parametrize("lens,hq,hkv,D", [
    ([1000] * 33, 8, 8, 128),             # narrow rows, even runs: four runs of two passes
    ([4100] * 8, 4, 2, 64),               # the same with one pass
    ([20000] + [1000] * 13, 4, 4, 64),    # a sequence longer than two runs: heads first
])
def test_host_entry_point_cuts_copy_bound_batches_into_runs(lens, hq, hkv, D):
    test_host_entry_point_slices(lens, hq, hkv, D)


@pytest.mark.parametrize("lens,hq,hkv,D", [([700, 130, 1], 4, 2, 64), ([2300, 900, 64], 8, 2, 128)])
def test_captured_calls(lens, hq, hkv, D):
    """Forward and backward captured into a graph, replayed over new inputs while other plans are uploaded, run and dropped: the
    work counters come back to zero each time, and the captured plan's tables stay its own."""
    from paper_2602_21788_b200 import fcp
    from paper_2602_21788_b200.runner import DeviceState
    w = _wl(lens, [1] * len(lens), hq, hkv, D, seed=53)
    ds = DeviceState(w, *w.device_tensors(), partials=False)
    other = [fcp.Plan([500 + 100 * i, 77], [1, 1], hq, hkv, D) for i in range(3)]
    big = torch.randn((800, hq, D), device="cuda").bfloat16()
    small = torch.randn((800, hkv, D), device="cuda").bfloat16()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):                       # eager once, as before any capture
        ds.forward_fused(side)
        ds.backward(side)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ds.forward_fused()
        ds.backward()
    g = torch.Generator(device="cuda").manual_seed(59)
    for r in range(4):
        for t in (ds.q, ds.k, ds.v, ds.do):
            t.copy_(torch.randn(t.shape, device="cuda", generator=g))
        for t in (ds.o, ds.lse, ds.dq, ds.dk, ds.dv):
            t.zero_()
        graph.replay()
        if r < 3:
            plan = other[r].upload()
            _fused(plan, big, small, small, hq, torch.cuda.current_stream())
            other[r] = None
            del plan
        got = [t.clone() for t in (ds.o, ds.lse, ds.dk, ds.dv, ds.dq)]
        fresh = DeviceState(w, ds.q, ds.k, ds.v, ds.do, partials=False)
        fresh.forward_fused()
        fresh.backward()
        torch.cuda.synchronize()
        ds.check_status()
        for a, b in zip(got, (fresh.o, fresh.lse, fresh.dk, fresh.dv)):
            assert torch.equal(a, b), r
        assert (got[4].float() - fresh.dq.float()).norm() <= 1e-2 * fresh.dq.float().norm()
        del fresh
    del graph
