"""Calls from several host threads at once, each on its own stream: the bits of the same calls made alone and in plain order."""
import threading
from types import SimpleNamespace

import pytest
import torch

from paper_2602_22592_b200 import binding as pqb
from paper_2602_22592_b200 import inputs as I
from paper_2602_22592_b200.layer import PQLinear
from test_gpu_ffn import _pack, _pack8, _weights
from test_gpu_forward import check_status

pytestmark = pytest.mark.gpu
PER_THREAD = SimpleNamespace(cuda_stream=2)      # cudaStreamPerThread: one handle, another stream in every thread


def _ffn(T, Dm, F1, r):
    X, Wg, Wu, Wd, G, U, D = _weights(T, Dm, F1, r, seed=T)
    one = [_pack(W) for W in (Wg, Wu, Wd)]
    G8, D8, gd = _pack8(G, D)
    U8, _, ud = _pack8(U, D)
    hp = torch.stack([gd[0, 0], ud[0, 0], gd[0, 1]]).contiguous()
    d = pqb.make_ffn_desc(T, Dm, F1, r)
    ws = torch.empty(pqb.pq_ffn_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    Xd, al, be = torch.from_numpy(X).cuda().to(torch.bfloat16), torch.full((1,), 2.0, device="cuda"), torch.full((1,), 0.2, device="cuda")
    out = torch.empty((T, Dm), dtype=torch.bfloat16, device="cuda")
    return out, lambda Y, stream: pqb.pq_ffn_forward(d, Xd, *one[0], *one[1], *one[2], G8, U8, D8, hp, al, be, Y, ws, stream=stream)


def _dense(T, K, N, r):
    L = PQLinear(T, K, N, r, 1).load_case(I.make_linear_case(T, K, N, r, 1, seed=T, with_grad=False))
    L.pack()
    return L.Y, lambda Y, stream: pqb.pq_linear_forward(L.desc, L.X, L.w_bits, L.w_s8, L.w_scales, L.A, L.B, L.Wr, L.alpha, L.beta, Y, None,
                                                        L.ws_fwd, stream=stream)


def test_threads_on_the_per_thread_stream():
    # long and short calls side by side, so that one thread's fork and join fall between those of another
    work = [_ffn(700, 512, 2080, 48), _ffn(129, 256, 1056, 128), _dense(1000, 1056, 544, 64), _dense(130, 96, 64, 16)]
    rounds, want, got, failed = 30, [], [], []
    pqb.pq_set_option(pqb.PQ_OPT_SIDE_STREAM, 0)
    try:
        for out, call in work:
            call(out, None)
            want.append(out.clone())
    finally:
        pqb.pq_set_option(pqb.PQ_OPT_SIDE_STREAM, 1)
    for out, _ in work:
        got.append([torch.zeros_like(out) for _ in range(rounds)])
    torch.cuda.synchronize()
    start = threading.Barrier(len(work))

    def thread(i):
        try:
            start.wait(60)
            for Y in got[i]:
                work[i][1](Y, PER_THREAD)
        except Exception as e:  # noqa: BLE001 -- reported by the test
            failed.append(e)
    threads = [threading.Thread(target=thread, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    check_status()
    assert not failed
    for w, ys in zip(want, got):
        for Y in ys:
            assert torch.equal(Y, w)
