"""Edges of the kernels' own splits -- tiles, pairs of tiles, steps, blocks of tokens -- against the oracle, at sizes that
straddle them."""
import numpy as np
import pytest
import torch

from oracle import pquant_oracle as O
from paper_2602_22592_b200 import binding as pqb
from paper_2602_22592_b200 import inputs as I
from paper_2602_22592_b200.layer import PQLinear
from test_gpu_backward import check_backward, run_fwd_bwd
from test_gpu_ffn import test_ffn_decoupled_forward_matches_oracle as check_ffn
from test_gpu_forward import TOL_BF16, check_forward, check_status, f32, rel_err, run_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,K,E", [
    (1, 32, 2), (17, 288, 4),        # one token; one past a block of 16, one past a step of 256 elements
    (2369, 64, 5), (4737, 32, 9),    # one past 148 and past 2 x 148 blocks of tokens (one and two CTAs per SM); 8 / 16 experts
    (8209, 32, 16),                  # one past the 512 blocks of tokens that the scan takes in one go
])
def test_router_and_routing_tables(T, K, E):
    # indices, permutation and tables exact, gates and probabilities to the rounding of an fp32 softmax (check_forward)
    c = I.make_linear_case(T, K, 32, 16, E, seed=T + E, with_grad=False)
    check_forward(c, run_forward(c, False), O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"]))
    assert len(np.unique(O.router(c["X"], c["Wr"])["idx"])) >= min(T, 2)


@pytest.mark.parametrize("T,K,N,r,E,vector", [
    (1, 32, 32, 8, 1, False), (257, 288, 544, 72, 2, True),   # a lone tile of every kind; second tile of a pair with one row, r past 64
    (513, 544, 288, 128, 16, False),                          # experts that share tiles and pairs of tiles, most with few tokens
    (640, 4128, 96, 0, 0, False),                             # no HP branch: no dH tile to wait for; 17 column tiles, one feature tile
    (300, 64, 4128, 40, 1, True),                             # the longest contraction is dX's
])
def test_training_step_on_pairs_of_tiles(T, K, N, r, E, vector):
    # forward and every gradient, the tolerances of check_forward and check_backward
    c = I.make_linear_case(T, K, N, r, E, seed=T, scale_vector=vector, alpha=1.5, beta=0.5)
    f = O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    g = O.linear_backward(c["dY"], c["X"], f, c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    L = run_fwd_bwd(c, vector)
    check_forward(c, L, f)
    check_backward(c, L, f, g, vector)


@pytest.mark.parametrize("F1", [1056, 2080, 4128, 8224])
def test_ffn_rows_of_one_to_eight_warps(F1):
    # one past what one, two and four warps hold of a row in registers, and past what eight do; an odd number of rows.  Codes
    # and scales exact on the hidden activation the GPU made
    check_ffn(131, 96, F1, 16)


def test_forward_of_long_rows_uses_the_general_tile():
    # K = 32768: a sum of the 1-bit product no longer fits the short conversion to float; rows of equal signs reach |sum| ~ 128 K
    c = I.make_linear_case(40, 32768, 32, 8, 1, seed=3, with_grad=False)
    c["X"][:] = I.bf16_values(np.abs(c["X"]) + 4.0)
    c["W"][:16] = np.abs(c["W"][:16]) + 0.01
    f = O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    check_forward(c, run_forward(c, False), f)


def test_router_calls_of_two_threads_at_once():
    # the router asks for 116, 76 or 36 KB of shared memory by the number of blocks of tokens; the kernel's limit belongs to the
    # process, so a call must not lower it between another thread's look at it and that thread's launch
    import threading
    layers = []
    for T in (2048, 4096, 8192):
        c = I.make_linear_case(T, 64, 64, 16, 8, seed=T, with_grad=False)
        L = PQLinear(T, 64, 64, 16, 8).load_case(c)
        L.pack()
        L.forward()
        layers.append(L)
    torch.cuda.synchronize()
    want = [(L.Y.clone(), L.saved_view()["perm"].clone()) for L in layers]
    failed = []

    def calls(L):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(300):
                    L.forward()
        except Exception as e:      # noqa: BLE001 -- reported by the main thread
            failed.append(e)
    threads = [threading.Thread(target=calls, args=(L,)) for L in layers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    check_status()
    assert not failed
    for L, (y, perm) in zip(layers, want):
        assert torch.equal(L.Y, y) and torch.equal(L.saved_view()["perm"], perm)


def _decode_layers(shapes):
    layers = []
    for i, kw in enumerate(shapes):
        kw = dict(kw)
        hp8, stream = kw.pop("hp8", False), kw.pop("stream", True)
        c = I.make_linear_case(kw["T"], kw["K"], kw["N"], kw["r"], kw["E"], seed=60 + i, exact_quota=False, with_grad=False)
        L = PQLinear(c["T"], c["K"], c["N"], c["r"], c["E"], training=False, dump_acc=True).load_case(c)
        PQLinear.stream_decode = stream
        try:
            L.pack(bits_only=True)
        finally:
            PQLinear.stream_decode = True
        if hp8:
            L.pack_decode_hp8()
        layers.append((L, c))
    return layers


def check_decode_int8(c, L):
    # every integer the INT8 branch goes through, and the outputs, against the oracle
    mu, lam = O.weight_scales(c["W"])
    f = O.decode_forward(c["X"], O.pack_bits(O.binarize(c["W"], mu)), lam, c["A"], c["B"], c["Wr"], c["alpha"], c["beta"],
                         hp_int8=O.quantize_experts(c["A"], c["B"]))
    v = L.decode_view()
    for name, want in (("expert", f["idx"]), ("acc", f["acc"]), ("hp_h_int", f["h_int"]), ("hp_z_int", f["z_int"])):
        assert np.array_equal(v[name].cpu().numpy().astype(np.int64), want)
    assert rel_err(f32(L.Y), f["Y"]) <= TOL_BF16


@pytest.mark.parametrize("shapes", [
    *[[dict(T=M, K=256, N=96, r=32, E=4, hp8=hp8)] * n for n, M, hp8 in [(2, 9, False), (6, 4, False), (2, 9, True), (6, 2, True), (12, 8, True)]],
    # codes of a row too long to be in shared memory at once; one unit; ragged hidden widths; the INT8 branch beside linears
    # with and without the streaming layout
    [dict(T=16, K=16384, N=64, r=32, E=2)], [dict(T=16, K=16384, N=64, r=40, E=2, stream=False)],
    [dict(T=1, K=32, N=32, r=8, E=16), dict(T=8, K=4128, N=1056, r=48, E=2, hp8=True), dict(T=5, K=96, N=160, r=72, E=3, stream=False)],
])
def test_decode_small_groups(shapes):
    # the exact integers and the outputs of the oracle, in three launches
    from test_gpu_decode import check_decode
    layers = _decode_layers(shapes)
    before = pqb.pq_kernel_launches()
    pqb.pq_decode_batch(pqb.make_decode_items([L.decode_entry() for L, _ in layers]))
    assert pqb.pq_kernel_launches() - before == 3
    torch.cuda.synchronize()
    check_status()
    for (L, c), kw in zip(layers, shapes):
        (check_decode_int8 if kw.get("hp8") else check_decode)(c, L)


def _layers_alike(n, M, r, E, hp8):
    # n linears of 64 -> 8192 with the same weights and activations
    c = I.make_linear_case(M, 64, 8192, r, E, seed=71, exact_quota=False, with_grad=False)
    layers = []
    for _ in range(n):
        L = PQLinear(M, 64, 8192, r, E, training=False, dump_acc=True).load_case(c)
        L.pack(bits_only=True)
        if hp8:
            L.pack_decode_hp8()
        layers.append(L)
    return c, layers


def _linears_for(units_per_sm):
    return -(-units_per_sm * torch.cuda.get_device_properties(0).multi_processor_count * 16 // 8192)


@pytest.mark.parametrize("M,r,E,hp8,least", [
    # units of 16 features per SM from which the streaming kernel takes a batch: by tokens and kind of branch
    (1, 16, 4, False, 19), (1, 16, 4, True, 19), (2, 16, 4, False, 29), (3, 16, 2, False, 40), (4, 16, 4, True, 44), (6, 16, 4, False, 75),
    (1, 16, 1, False, 19), (2, 16, 1, False, 50), (1, 0, 0, False, 37), (2, 0, 0, False, 65), (7, 16, 4, False, None),
])
def test_decode_dispatch_on_both_sides_of_its_lines(M, r, E, hp8, least):
    from test_gpu_decode import check_decode
    n = 48 if least is None else _linears_for(least)
    c, layers = _layers_alike(n, M, r, E, hp8)
    for take, launches in ((n - 1, 3 if r else 2), (n, (3 if r else 2) if least is None else 1)):
        for L in layers:
            L.Y.zero_()
            L.ws_decode.zero_()
        before = pqb.pq_kernel_launches()
        pqb.pq_decode_batch(pqb.make_decode_items([L.decode_entry() for L in layers[:take]]))
        assert pqb.pq_kernel_launches() - before == launches
        torch.cuda.synchronize()
        check_status()
        (check_decode_int8 if hp8 else check_decode)(c, layers[take - 1])
        assert all(torch.equal(L.Y, layers[0].Y) for L in layers[1:take])


@pytest.mark.parametrize("plain,launches", [
    ([0], 3 + 1), ([1], 3 + 1), ([2], 3 + 1),             # linears without the layout, alone or after one or two with it: up to the run that pays
    ([-1], 1 + 3), ([0, -1], 3 + 1 + 3),
])
def test_decode_batch_of_a_run_that_pays_and_linears_without_the_layout(plain, launches):
    n = _linears_for(19)
    c, layers = _layers_alike(n + len(plain) + max(plain[0], 0), 1, 16, 4, False)
    entries = [list(L.decode_entry()) for L in layers]
    for k in plain:
        entries[k][13] = entries[k][14] = None
    before = pqb.pq_kernel_launches()
    pqb.pq_decode_batch(pqb.make_decode_items([tuple(e) for e in entries]))
    assert pqb.pq_kernel_launches() - before == launches
    torch.cuda.synchronize()
    check_status()
    from test_gpu_decode import check_decode
    for k in (0, len(layers) // 2, -1):
        check_decode(c, layers[k])


@pytest.mark.parametrize("mode", [0, 2])
def test_decode_output_that_starts_at_an_odd_element(mode):
    # outputs are stored two features at a time where the output allows it, else one by one
    M, N = 5, 96
    c = I.make_linear_case(M, 256, N, 32, 4, seed=11, exact_quota=False, with_grad=False)
    L = PQLinear(M, 256, N, 32, 4, training=False).load_case(c)
    L.pack(bits_only=True)
    buf = torch.full((M * N + 2,), 7.0, dtype=torch.bfloat16, device="cuda")
    pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, mode)
    try:
        L.decode()
        L.decode(Y=buf[1:-1])
        torch.cuda.synchronize()
    finally:
        pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, 1)
    check_status()
    assert torch.equal(buf[1:-1].view(M, N), L.Y) and buf[0] == 7.0 and buf[-1] == 7.0


def _decode_case(T, K, N, r, E, norm, seed=17):
    c = I.make_linear_case(T, K, N, r, E, seed=seed, exact_quota=False, with_grad=False)
    L = PQLinear(T, K, N, r, E, training=False, dump_acc=True).load_case(c)
    w = None
    if norm:
        w = I.bf16_values(1.0 + 0.1 * np.random.default_rng(5).standard_normal(K).astype(np.float32))
        L.norm_weight, L.norm_eps = torch.from_numpy(w).cuda().to(torch.bfloat16), 1e-5
    L.pack(bits_only=True)
    return c, L, w


def _check_long_row(c, L, w):
    mu, lam = O.weight_scales(c["W"])
    f = O.decode_forward(c["X"], O.pack_bits(O.binarize(c["W"], mu)), lam, c["A"], c["B"], c["Wr"], c["alpha"], c["beta"],
                         **(dict(norm_weight=w, norm_eps=1e-5) if w is not None else {}))
    v = L.decode_view()
    assert np.array_equal(v["expert"].cpu().numpy(), f["idx"])
    assert np.array_equal(v["code_sum"].cpu().numpy(), f["q"].astype(np.int64).sum(axis=1))
    assert np.array_equal(v["acc"].cpu().numpy().astype(np.int64), f["acc"])
    assert rel_err(f32(L.Y), f["Y"]) <= TOL_BF16


@pytest.mark.parametrize("K,E,norm", [
    (25600, 16, True), (25632, 16, True),     # token, two router rows and gains: as many as fit, and one group of 32 values more
    (34112, 16, False), (34112, 8, True), (34144, 8, True), (32768, 1, True),
])
def test_decode_of_rows_that_fill_shared_memory(K, E, norm):
    c, L, w = _decode_case(3, K, 64, 16, E, norm)
    L.decode()
    torch.cuda.synchronize()
    check_status()
    _check_long_row(c, L, w)


@pytest.mark.parametrize("shapes", [
    [(1, 32768, 32, 16, 1, True), (16, 64, 32, 16, 16, False)],        # the longest row, the most experts and the norm in different linears
    [(1, 100000, 32, 16, 1, False), (16, 64, 32, 256, 2, False)],      # no room for both in one launch
])
def test_decode_batch_of_linears_that_fit_one_by_one(shapes):
    layers = [_decode_case(*s, seed=18 + i)[1] for i, s in enumerate(shapes)]
    pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, 0)
    try:
        for L in layers:
            L.decode()
        torch.cuda.synchronize()
        want = [L.Y.clone() for L in layers]
        for L in layers:
            L.Y.zero_()
        pqb.pq_decode_batch(pqb.make_decode_items([L.decode_entry() for L in layers]))
        torch.cuda.synchronize()
    finally:
        pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, 1)
    check_status()
    assert all(torch.equal(L.Y, y) for L, y in zip(layers, want))


@pytest.mark.parametrize("mode", [0, 2])
def test_decode_expert_when_the_first_logit_is_not_a_number(mode):
    # one logit is compared after the other, from expert 0 on: nothing is greater than a logit that is not a number
    c = I.make_linear_case(3, 256, 96, 16, 4, seed=23, exact_quota=False, with_grad=False)
    c["Wr"][0, 5] = np.nan
    D = PQLinear(3, 256, 96, 16, 4, training=False).load_case(c)
    L = PQLinear(3, 256, 96, 16, 4).load_case(c)
    pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, mode)
    try:
        D.pack(bits_only=True)
        D.decode()
        L.pack()
        L.forward()
        torch.cuda.synchronize()
    finally:
        pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, 1)
    check_status()
    assert D.decode_view()["expert"].tolist() == L.saved_view()["expert"].tolist() == [0, 0, 0]


@pytest.mark.parametrize("T,K,N,r,E,vector", [
    (1, 32, 32, 8, 1, False), (257, 1024, 544, 72, 2, True),   # a lone tile; the longest contraction on single CTAs, rows left over in both forms
    (257, 1056, 544, 72, 2, False),                            # the shortest on pairs
    (513, 128, 288, 128, 16, False), (640, 512, 96, 0, 0, True),
])
def test_forward_on_single_ctas_and_on_pairs(T, K, N, r, E, vector):
    c = I.make_linear_case(T, K, N, r, E, seed=T, scale_vector=vector, alpha=1.5, beta=0.5, with_grad=False)
    f = O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    check_forward(c, run_forward(c, vector), f)


@pytest.mark.parametrize("M,K,N,r,E", [
    (4, 1056, 7552, 160, 8), (14, 1056, 7552, 160, 8),      # short rows of sign bits: more expert rows in a pass than those would hold
    (16, 8640, 3200, 256, 8), (16, 3200, 8640, 160, 8),     # codes, sign bits and expert rows that do not fit at once
    (1, 32, 37888, 8, 1), (9, 64, 4768, 8, 16),             # many units in a pass; a unit more than two for each SM
])
def test_decode_shapes_of_a_pass(M, K, N, r, E):
    from test_gpu_decode import check_decode
    c, L, _ = _decode_case(M, K, N, r, E, False, seed=31)
    others = [_decode_case(M, 8640, 512, r, E, False, seed=32)[1], _decode_case(M, 96, 2048, r, E, False, seed=33)[1]]
    pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, 0)
    try:
        L.decode()
        torch.cuda.synchronize()
        check_decode(c, L)
        y = L.Y.clone()
        for beside in (others[:1], others):     # other splits of shared memory, the same bits
            L.Y.zero_()
            pqb.pq_decode_batch(pqb.make_decode_items([L.decode_entry()] + [o.decode_entry() for o in beside]))
            torch.cuda.synchronize()
            assert torch.equal(L.Y, y)
    finally:
        pqb.pq_set_option(pqb.PQ_OPT_DECODE_STREAM, 1)
    check_status()


@pytest.mark.parametrize("hp8", [False, True])
@pytest.mark.parametrize("T,K,N,r,E", [(1, 32, 32, 16, 1), (129, 1056, 96, 32, 4), (300, 512, 544, 128, 16), (300, 2080, 64, 0, 0)])
def test_forward_that_keeps_nothing_for_a_backward(T, K, N, r, E, hp8):
    # without a saved buffer the operands of the backward are not written: the same output
    if hp8 and r == 0:
        pytest.skip("needs experts")
    c = I.make_linear_case(T, K, N, r, E, seed=T + K, with_grad=False)
    L = PQLinear(T, K, N, r, E).load_case(c)
    L.pack()
    if hp8:
        L.pack_experts()
        L.forward_hp8()
    else:
        L.forward()
    Y = torch.zeros_like(L.Y)
    ws = torch.full((pqb.pq_workspace_bytes(L.desc, pqb.PQ_PHASE_FWD) + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    if hp8:
        pqb.pq_linear_forward_hp8(L.desc, L.X, L.w_s8, L.w_scales, L.A8, L.B8, L.hp_scales, L.Wr, L.alpha, L.beta, Y, None, ws[:-4096])
    else:
        pqb.pq_linear_forward(L.desc, L.X, L.w_bits, L.w_s8, L.w_scales, L.A, L.B, L.Wr, L.alpha, L.beta, Y, None, ws[:-4096])
    torch.cuda.synchronize()
    check_status()
    assert torch.equal(Y, L.Y) and bool((ws[-4096:] == 0xA5).all())


@pytest.mark.parametrize("T,K,N,r,E,vector", [
    (100, 1056, 288, 72, 16, False),      # sixteen experts to a tile
    (129, 96, 64, 16, 3, True), (4100, 64, 96, 24, 2, False), (16640, 64, 96, 24, 1, False),   # a tile more than one; many tiles of an expert
])
def test_gradients_of_experts_over_their_items(T, K, N, r, E, vector):
    # dB and dA contract over an expert's items in one run: from its first tile on, in the tokens and in the hidden planes
    c = I.make_linear_case(T, K, N, r, E, seed=T + E, scale_vector=vector, alpha=1.5, beta=0.5)
    f = O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    g = O.linear_backward(c["dY"], c["X"], f, c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    check_backward(c, run_fwd_bwd(c, vector), f, g, vector)


@pytest.mark.parametrize("T", [128, 256, 300])        # whole tiles: the experts behind the last token then start a tile beyond it
def test_gradients_beside_experts_without_tokens(T):
    c = I.make_linear_case(T, 96, 160, 24, 8, seed=T)
    planted = np.array([1, 2, 5])[np.arange(T) % 7 % 3]    # none for the first, the last two and two in the middle
    c["X"] = I.bf16_values(np.random.default_rng(T).standard_normal((T, 96)).astype(np.float32) + 8 * c["Wr"][planted])
    f = O.linear_forward(c["X"], c["W"], c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    g = O.linear_backward(c["dY"], c["X"], f, c["A"], c["B"], c["Wr"], c["alpha"], c["beta"])
    tokens = np.bincount(f["idx"], minlength=8)
    assert np.array_equal(np.flatnonzero(tokens == 0), [0, 3, 4, 6, 7])
    L = run_fwd_bwd(c, False)
    check_backward(c, L, f, g, False)
    for e in (0, 3, 4, 6, 7):
        assert not bool(L.dA[e].any()) and not bool(L.dB[e].any())


@pytest.mark.parametrize("T,K,N,r,E", [(129, 96, 64, 16, 1), (300, 1056, 96, 32, 4), (200, 8704, 64, 0, 0)])
def test_normalised_forward_that_keeps_nothing(T, K, N, r, E):
    # the up-projection reads the normalised rows, which the quantiser leaves in the workspace then
    c = I.make_linear_case(T, K, N, r, E, seed=T, with_grad=False)
    L = PQLinear(T, K, N, r, E, fused_rmsnorm=True).load_case(c)
    L.norm_weight, L.norm_eps = (1 + 0.1 * torch.randn(K, device="cuda")).to(torch.bfloat16), 1e-5
    L.pack()
    L.forward()
    Y = torch.zeros_like(L.Y)
    ws = torch.full((pqb.pq_workspace_bytes(L.desc, pqb.PQ_PHASE_FWD) + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    pqb.pq_linear_forward_rms(L.desc, L.X, L.norm_weight, L.norm_eps, L.w_s8, L.w_scales, L.A, L.B, L.Wr, L.alpha, L.beta, Y, None, ws[:-4096])
    torch.cuda.synchronize()
    check_status()
    assert torch.equal(Y, L.Y) and bool((ws[-4096:] == 0xA5).all())


def test_all_experts_forward_that_keeps_nothing():
    T, K, N, r, E = 129, 256, 320, 16, 8
    c = I.make_linear_case(T, K, N, r, E, seed=5, with_grad=False)
    L = PQLinear(T, K, N, r, E).load_case(c)
    L.pack()
    d = pqb.make_desc(T, K, N, r, E, top_k=E, unit_gates=True)
    saved = torch.empty(pqb.pq_saved_bytes(d), dtype=torch.uint8, device="cuda")
    ws = torch.full((pqb.pq_workspace_bytes(d, pqb.PQ_PHASE_FWD) + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    out = []
    for keep in (saved, None):
        out.append(torch.zeros_like(L.Y))
        pqb.pq_linear_forward(d, L.X, L.w_bits, L.w_s8, L.w_scales, L.A, L.B, None, L.alpha, L.beta, out[-1], keep, ws[:-4096])
        torch.cuda.synchronize()
    check_status()
    assert torch.equal(*out) and bool(out[0].any()) and bool((ws[-4096:] == 0xA5).all())
