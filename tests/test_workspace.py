"""The binding's default scratch buffer: calls that may run at the same time do not share one."""
import gc
import threading
import weakref

import numpy as np
import pytest

from oracle import qbp_oracle as O
from tests.util import random_codes, set_qparams, to_dev, to_host


@pytest.fixture(scope="module")
def B():
    import paper_1805_11046_b200.binding as binding
    return binding


def test_one_buffer_per_device_stream_and_thread(B, monkeypatch):
    import torch
    empty, now = torch.empty, {"device": 0, "stream": 0}
    monkeypatch.setattr(torch, "empty", lambda n, dtype=None, device=None: empty(n, dtype=dtype))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: now["device"])
    monkeypatch.setattr(B, "_workspaces", B._Workspaces())
    monkeypatch.setattr(B, "_raw_stream", lambda device: now["stream"])
    first = B.workspace(100)
    assert B.workspace(1 << 20) is first and B.workspace(100, "cuda") is first and B.workspace(100, "cuda:0") is first
    now["stream"] = 4096                                   # another stream of the same thread
    other = B.workspace(100)
    assert other is not first and B.workspace(100) is other
    now["stream"] = 0
    assert B.workspace(100) is first
    assert B.workspace(100, "cuda:1") is not first         # another device
    grown = B.workspace((1 << 20) + 1)
    assert grown is not first and grown.numel() > 1 << 20 and B.workspace(100) is grown
    theirs = []
    t = threading.Thread(target=lambda: theirs.append(weakref.ref(B.workspace(100))))
    t.start(); t.join()
    gc.collect()
    assert theirs[0]() is None                             # another thread's own, given back when it ended


@pytest.mark.gpu
def test_calls_on_two_streams_of_one_thread(B):
    """Products, weight gradients and quantisers enqueued in turn on two streams, each call with the default scratch, while
    the other stream's calls are running: the results of every call are those of the oracle."""
    import torch
    jobs = []
    for k, (M, N, K) in enumerate([(512, 512, 1024), (640, 528, 2048)]):
        A, Bm = random_codes((M, K), 91 + k), random_codes((K, N), 93 + k)
        G = np.random.Generator(np.random.PCG64(95 + k)).integers(-32768, 32768, (M, N)).astype(np.int16)
        hi, lo = O.limb_split(G)
        X = np.random.Generator(np.random.PCG64(97 + k)).standard_normal((M, K)).astype(np.float32) * np.float32(1 + k)
        q = lambda s, z: set_qparams(B.new_qparams(1), s, z)
        jobs.append(dict(A=to_dev(A), B=to_dev(Bm), hi=to_dev(hi), lo=to_dev(lo), X=to_dev(X), qa=q(0.5, 7 - k), qb=q(0.25, -19 + k), qg=q(0.125, 300 + k),
                         gemm=O.gemm_s8(A, 7 - k, Bm, -19 + k)[0], wgrad=O.gemm_s16s8(A, 7 - k, G, 300 + k)[0], quant=O.quantize(X, 8).q))
    streams = [torch.cuda.Stream() for _ in jobs]
    torch.cuda.synchronize()
    results = [[], []]
    for _ in range(20):
        for s, j, r in zip(streams, jobs, results):
            with torch.cuda.stream(s):
                r.append((B.qbp_gemm_s8(j["A"], j["qa"], j["B"], j["qb"], want_acc=True, want_out=False)[0],
                          B.qbp_wgrad_s16(j["A"], j["qa"], j["hi"], j["lo"], j["qg"], want_acc=True, want_out=False)[0],
                          B.qbp_quantize_s8(j["X"])[0]))
    torch.cuda.synchronize()
    for j, r in zip(jobs, results):
        for acc, grad, codes in r:
            assert np.array_equal(to_host(acc), j["gemm"]) and np.array_equal(to_host(grad), j["wgrad"]) and np.array_equal(to_host(codes), j["quant"])
