"""Two host threads, each with its own stream and buffers, whose calls need different amounts of shared memory in the
same kernels: every call succeeds and gives what it gives alone.  The calls go to the library directly, with
arguments made once, so that both threads are inside it nearly all the time."""

import ctypes as C
import threading

import pytest
import torch

import workload as wl

pytestmark = pytest.mark.gpu

CALLS = 4000


def _condense(wz, stream, T, D, dtype, relevance):
    X, Q = wl.random_video(T, 12, 11, D, 3, dtype=dtype, seed=T)
    X, Q = X.cuda(), Q.cuda()
    code = wz.DTYPE_F32 if dtype == "f32" else wz.DTYPE_BF16
    ws = torch.empty(wz.wz_condense_workspace_size(T, 12, 11, D, code, 0.1), dtype=torch.uint8, device="cuda")
    out = wz.wz_condense_ex(X, Q, 0.1, relevance=relevance, workspace=ws)
    a = wz.CondenseArgs()
    wz._lib.wz_condense_args_init(C.byref(a))
    a.features, a.T, a.H, a.W, a.D, a.dtype = X.data_ptr(), T, 12, 11, D, code
    a.query, a.Lq, a.ratio, a.relevance_mode = Q.data_ptr(), 3, 0.1, wz.RELEVANCE_MODES[relevance]
    a.workspace, a.workspace_bytes, a.stream = ws.data_ptr(), ws.numel(), stream.cuda_stream
    tokens, index = torch.zeros_like(out["tokens"]), torch.zeros_like(out["index"])
    a.out_tokens, a.out_index = tokens.data_ptr(), index.data_ptr()
    keep = (X, Q, ws, index)
    return (lambda: wz._lib.wz_condense_ex(C.byref(a))), tokens, out["tokens"], keep


def _dwt(wz, stream, H, W):
    X = torch.randn(2, H, W, 64, generator=torch.Generator().manual_seed(H)).cuda()
    want = torch.stack(wz.wz_dwt2d(X, 10))
    bands = torch.zeros_like(want)
    args = (X.data_ptr(), 2, H, W, 64, wz.DTYPE_F32, 10, 0, *[b.data_ptr() for b in bands], stream.cuda_stream)
    return (lambda: wz._lib.wz_dwt2d(*args)), bands, want, X


KINDS = {   # the call of thread k
    "simt": lambda wz, s, k: _condense(wz, s, (1500, 1900)[k], 64, "f32", "mean"),
    "tensor": lambda wz, s, k: _condense(wz, s, (7, 1800)[k], 64, "bf16", "mean"),
    "maxsim": lambda wz, s, k: _condense(wz, s, (7, 30)[k], (64, 3584)[k], "bf16", "maxsim"),
    "relevance": lambda wz, s, k: _condense(wz, s, (60, 50)[k], (320, 2304)[k], "bf16", "mean"),
    "dwt2d": lambda wz, s, k: _dwt(wz, s, (6, 40)[k], (7, 37)[k]),
}


@pytest.mark.parametrize("kind", KINDS)
def test_two_threads(kind):
    import paper_2607_23265_gb300 as wz
    codes, capacity = [set(), set()], wz.wz_graph_cache(0)["previous_capacity"]   # direct launches only
    try:
        streams = [torch.cuda.Stream() for _ in range(2)]
        calls = [KINDS[kind](wz, streams[k], k) for k in range(2)]
        torch.cuda.synchronize()
        start = threading.Barrier(2)

        def work(k):
            call = calls[k][0]
            start.wait()
            for _ in range(CALLS // 100):
                codes[k].update(call() for _ in range(100))
                streams[k].synchronize()   # bounds the launches in flight

        threads = [threading.Thread(target=work, args=(k,)) for k in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        torch.cuda.synchronize()
        assert codes == [{wz.OK}, {wz.OK}], codes
        for _, got, want, _ in calls:
            assert torch.equal(got, want)
    finally:
        wz.wz_graph_cache(capacity)
