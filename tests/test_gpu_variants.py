"""Alternative code paths behind switches, checked against the default path on the GPU:
the CUDA-core debug kernels, the dense (all experts) search, and replay of a captured CUDA
graph of moe_forward."""
import os

import numpy as np
import pytest
import torch

from oracle import moe_oracle as O
from paper_2402_14800_b200 import binding, build, synth
from tests import parity as P

pytestmark = pytest.mark.gpu

H, F, E = 128, 448, 8
DEV = "cuda:0"


@pytest.fixture(scope="module")
def weights():
    build.build()
    W = synth.make_layer_weights(H, F, E, seed=0)
    return [t.to(DEV) for t in (W.W_gate, W.W1, W.W3, W.W2)]


def layer_with_env(weights, kept=0xFF, **env):
    """The switches are read when a handle is created."""
    old = {k: os.environ.get(k) for k in env}
    os.environ.update({k: str(v) for k, v in env.items()})
    try:
        return binding.MoeLayer(*weights, kept)
    finally:
        for k, v in old.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v


def rel_l2(a, b):
    """Worst per-token relative L2 distance between two bf16 outputs."""
    a, b = a.double().cpu().numpy(), b.double().cpu().numpy()
    return float((np.linalg.norm(a - b, axis=1) / np.linalg.norm(b, axis=1)).max())


@pytest.mark.parametrize("T", [40, 700])
def test_debug_cuda_core_kernels_agree_with_tensor_core_path(weights, T):
    x = synth.make_tokens(T, H, seed=3).to(DEV)
    ref = binding.MoeLayer(*weights, 0b11011101)
    dbg = layer_with_env(weights, 0b11011101, MOE_DEBUG_SIMT=1)
    y0, y1 = ref.forward(x, 0.4), dbg.forward(x, 0.4)
    torch.cuda.synchronize()
    assert rel_l2(y1, y0) < 5e-3  # different summation orders, same rounding points
    ref.close()
    dbg.close()


@pytest.mark.parametrize("T", [1, 5, 40, 150, 256])
def test_both_small_batch_gemms_at_every_size(weights, T):
    # by default the batch size picks the kernel of a small batch; each one is forced here over
    # the whole range and compared with the CUDA-core kernels
    x = synth.make_tokens(T, H, seed=6).to(DEV)
    dbg = layer_with_env(weights, 0b01111011, MOE_DEBUG_SIMT=1)
    y0 = dbg.forward(x, 0.3)
    for kernel in ("wm", "td"):
        lay = layer_with_env(weights, 0b01111011, MOE_DECODE_KERNEL=kernel)
        y1 = lay.forward(x, 0.3)
        y2 = lay.forward(x, 0.3)
        torch.cuda.synchronize()
        assert rel_l2(y1, y0) < 5e-3
        assert torch.equal(y1, y2)
        assert lay.device_status() == 0
        lay.close()
    dbg.close()


@pytest.mark.parametrize("beta", [0.0, 0.6])
def test_single_token_kernels_agree_with_gemm_path(weights, beta):
    # T = 1 runs matrix-vector kernels by default; MOE_SINGLE_KERNEL=gemm keeps the grouped GEMMs
    gemv = binding.MoeLayer(*weights, 0b11110110)
    gemm = layer_with_env(weights, 0b11110110, MOE_SINGLE_KERNEL="gemm")
    for seed in range(8):
        x = synth.make_tokens(1, H, seed=50 + seed).to(DEV)
        res = synth.make_tokens(1, H, seed=90 + seed).to(DEV) if seed % 2 else None
        y0 = gemm.forward(x, beta, residual=res)
        y1 = gemv.forward(x, beta, residual=res)
        y2 = gemv.forward(x, beta, residual=res)
        torch.cuda.synchronize()
        assert rel_l2(y1, y0) < 5e-3  # different summation orders, same rounding points
        assert torch.equal(y1, y2)
    assert gemv.device_status() == 0 and gemm.device_status() == 0
    gemv.close()
    gemm.close()


@pytest.mark.parametrize("r", [6, 4, 7])
def test_dense_search_equals_pruned_work_search(weights, r):
    x = synth.make_tokens(777, H, seed=4).to(DEV)
    fast = binding.MoeLayer(*weights)
    dense = layer_with_env(weights, MOE_SEARCH_DENSE=1)
    l0, b0 = fast.prune_search(x, r)
    l1, b1 = dense.prune_search(x, r)
    fast.close()
    dense.close()
    np.testing.assert_allclose(l0, l1, rtol=1e-6)
    assert b0 == b1


@pytest.mark.parametrize("T", [1, 16, 600])
def test_forward_replays_from_a_cuda_graph(weights, T):
    layer = binding.MoeLayer(*weights)
    x = synth.make_tokens(T, H, seed=6).to(DEV)
    y = torch.empty_like(x)
    s = torch.cuda.Stream(DEV)
    layer.set_stream(s)
    with torch.cuda.stream(s):
        layer.forward(x, 0.4, y=y)          # first call grows the scratch, outside the capture
        s.synchronize()
        want = y.clone()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            layer.forward(x, 0.4, y=y)
        x2 = synth.make_tokens(T, H, seed=7).to(DEV)
        y.zero_()
        g.replay()
        s.synchronize()
        assert torch.equal(y, want)
        x.copy_(x2)                          # same buffers, new contents
        g.replay()
        s.synchronize()
        fresh = layer.forward(x2, 0.4)
        s.synchronize()
        assert torch.equal(y, fresh)
    layer.close()


@pytest.mark.parametrize("T", [1, 2, 8, 40, 128, 600])
def test_back_to_back_calls_with_changing_inputs_equal_isolated_calls(weights, T):
    # Serving pattern: the same buffers, new contents every step, the calls queued without a
    # synchronisation in between (the kernels of consecutive calls overlap through programmatic
    # dependent launch).  Every step must give what the same input gives in an isolated call.
    n = 12
    layer = binding.MoeLayer(*weights, 0b11110111)
    xs = [synth.make_tokens(T, H, seed=200 + i).to(DEV) for i in range(n)]
    want = []
    for x in xs:
        want.append(layer.forward(x, 0.4).clone())
        torch.cuda.synchronize()
    x_buf = torch.empty_like(xs[0])
    ys = [torch.empty_like(xs[0]) for _ in range(n)]
    for rep in range(3):
        for i in range(n):
            x_buf.copy_(xs[i])
            layer.forward(x_buf, 0.4, y=ys[i])
        torch.cuda.synchronize()
        for i in range(n):
            assert torch.equal(ys[i], want[i]), "step %d of round %d differs from the isolated call" % (i, rep)
    assert layer.device_status() == 0
    layer.close()


STACK_SPECS = [(20, 0xFF, 0.0), (21, 0b10111011, 0.4), (22, 0b00111100, 0.5)]


@pytest.fixture(scope="module")
def stack_layers():
    build.build()
    layers = []
    for seed, kept, _ in STACK_SPECS:
        W = synth.make_layer_weights(H, F, E, seed=seed)
        layers.append(binding.MoeLayer(W.W_gate.to(DEV), W.W1.to(DEV), W.W3.to(DEV), W.W2.to(DEV), kept))
    for l in layers[1:]:
        l.share_scratch(layers[0])
    yield layers
    for l in reversed(layers):
        l.close()


@pytest.mark.parametrize("T", [1, 16, 128, 600])
def test_queued_stack_steps_equal_isolated_calls(stack_layers, T):
    # Three layers out of one set of scratch, every kernel a programmatic dependent of the one
    # before, the state buffer read as the residual and overwritten by the same launch from the
    # second layer on.  Steps are queued without synchronising, once on one refilled input buffer
    # and once on separate inputs with no other kernel between two steps; each must reproduce the
    # isolated call bit for bit.
    n = 8
    betas = [s[2] for s in STACK_SPECS]
    xs = [synth.make_tokens(T, H, seed=400 + i).to(DEV) for i in range(n)]
    want = []
    for x in xs:
        want.append(binding.stack_forward(stack_layers, x, betas, 1e-5).clone())
        torch.cuda.synchronize()
    x_buf = torch.empty_like(xs[0])
    ys = [torch.empty_like(xs[0]) for _ in range(n)]
    for rep in range(6 if T <= 128 else 3):
        for i in range(n):
            if rep % 2 == 0:
                x_buf.copy_(xs[i])
                binding.stack_forward(stack_layers, x_buf, betas, 1e-5, y=ys[i])
            else:
                binding.stack_forward(stack_layers, xs[i], betas, 1e-5, y=ys[i])
        torch.cuda.synchronize()
        for i in range(n):
            assert torch.equal(ys[i], want[i]), "step %d of round %d differs from the isolated call" % (i, rep)
        for y in ys:
            y.zero_()
    assert stack_layers[0].device_status() == 0


@pytest.mark.parametrize("T", [1, 16, 128, 600])
def test_queued_residual_steps_with_y_aliasing_the_residual(weights, T):
    # state <- state + MoE(x) in place (y and residual are the same buffer), queued steps
    n = 8
    layer = binding.MoeLayer(*weights, 0b11110111)
    xs = [synth.make_tokens(T, H, seed=500 + i).to(DEV) for i in range(n)]
    s0 = synth.make_tokens(T, H, seed=599).to(DEV)
    want, state = [], s0.clone()
    for x in xs:
        state = layer.forward(x, 0.4, residual=state).clone()   # separate output buffer, isolated
        torch.cuda.synchronize()
        want.append(state)
    for rep in range(4):
        state = s0.clone()
        snaps = []
        for i in range(n):
            layer.forward(xs[i], 0.4, residual=state, y=state)
            if rep % 2 == 0:
                snaps.append(state.clone())
        torch.cuda.synchronize()
        assert torch.equal(state, want[-1]), "round %d" % rep
        for i, snap in enumerate(snaps):
            assert torch.equal(snap, want[i]), "step %d of round %d" % (i, rep)
    assert layer.device_status() == 0
    layer.close()


@pytest.mark.parametrize("T", [2, 5, 16, 64, 128])
def test_small_batches_repeat_many_queued_steps(weights, T):
    # the small-batch sequences (router, permutation + gather, two GEMMs, combine: five programmatic
    # dependents per step on the same scratch addresses) queued 200 steps deep on alternating inputs
    layer = binding.MoeLayer(*weights, 0b11110111)
    xa, xb = (synth.make_tokens(T, H, seed=s).to(DEV) for s in (610, 611))
    wa, wb = layer.forward(xa, 0.4).clone(), layer.forward(xb, 0.4).clone()
    torch.cuda.synchronize()
    ya, yb = torch.empty_like(xa), torch.empty_like(xa)
    bad = torch.zeros((), dtype=torch.int32, device=DEV)
    for i in range(200):
        if i % 2 == 0:
            layer.forward(xa, 0.4, y=ya)
            bad += (~torch.eq(ya, wa)).any().int()
        else:
            layer.forward(xb, 0.4, y=yb)
            bad += (~torch.eq(yb, wb)).any().int()
    torch.cuda.synchronize()
    assert int(bad.item()) == 0
    assert layer.device_status() == 0
    layer.close()


def test_reserve_makes_later_calls_allocation_free(weights):
    # after moe_reserve(T_max) no forward call with T <= T_max grows the scratch, so a capture
    # needs no warm-up call
    layer = binding.MoeLayer(*weights)
    layer.reserve(700)
    held = layer.scratch_bytes
    assert held > 0
    s = torch.cuda.Stream(DEV)
    layer.set_stream(s)
    with torch.cuda.stream(s):
        x = synth.make_tokens(700, H, seed=6).to(DEV)
        y = torch.empty_like(x)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):       # first forward call of the handle, inside a capture
            layer.forward(x, 0.4, y=y)
        g.replay()
        s.synchronize()
        got = y.clone()
        for T in (1, 2, 40, 256, 257, 700):
            layer.forward(x[:T].contiguous(), 0.4)
        s.synchronize()
        assert layer.scratch_bytes == held
        assert torch.equal(layer.forward(x, 0.4), got)
        s.synchronize()
    with pytest.raises(binding.MoeError):
        layer.reserve(0)
    layer.close()


@pytest.mark.parametrize("T", [1, 40, 700])
def test_plain_stream_order_gives_the_same_bits(weights, T):
    # MOE_NO_PDL=1: every kernel in plain stream order instead of as a programmatic dependent;
    # the overlap of launches must not change a single bit
    x = synth.make_tokens(T, H, seed=8).to(DEV)
    ref = binding.MoeLayer(*weights, 0b11011101)
    want = ref.forward(x, 0.4).clone()
    ref.close()
    plain = layer_with_env(weights, 0b11011101, MOE_NO_PDL=1)
    try:
        got = plain.forward(x, 0.4).clone()
        torch.cuda.synchronize()
        assert plain.device_status() == 0
    finally:
        plain.close()
        layer_with_env(weights, MOE_NO_PDL=0).close()  # the switch is process-wide: back to the default
    assert torch.equal(got, want)


@pytest.mark.parametrize("h,f,E,kept,T", [
    # two kept experts and no skipping: both groups hold exactly T tokens, so T walks the edges of
    # the token tiles (grain 32, at most 256 a tile) and, above 1536, the other large-batch kernel
    (128, 448, 8, 0b00100100, 257), (128, 448, 8, 0b00100100, 287), (128, 448, 8, 0b00100100, 288),
    (128, 448, 8, 0b00100100, 289), (128, 448, 8, 0b00100100, 512), (128, 448, 8, 0b00100100, 513),
    (128, 448, 8, 0b00100100, 1536), (128, 448, 8, 0b00100100, 1537),
    # many small ragged groups; one k-block; weight rows just above one item of 512
    (128, 448, 8, 0xFF, 259), (64, 64, 16, 0xFFFF, 300), (64, 320, 3, 0b111, 333), (576, 64, 4, 0b1111, 700),
])
def test_large_batch_gemm_at_the_edges_of_its_tiles(h, f, E, kept, T):
    build.build()
    W = synth.make_layer_weights(h, f, E, seed=5, device=DEV)
    w = (W.W_gate, W.W1, W.W3, W.W2)
    x = synth.make_tokens(T, h, seed=6, device=DEV)
    lay, dbg = binding.MoeLayer(*w, kept), layer_with_env(w, kept, MOE_DEBUG_SIMT=1)
    y0, y1, y2 = dbg.forward(x), lay.forward(x), lay.forward(x)
    torch.cuda.synchronize()
    assert rel_l2(y1, y0) < 5e-3  # different summation orders, same rounding points
    assert torch.equal(y1, y2)
    assert lay.device_status() == 0
    lay.close()
    dbg.close()


@pytest.mark.parametrize("h,f,E,kept,T,k", [
    # expert counts between the instantiations, slices of a row that do not fill a warp, router rows
    # beyond the shared memory (8192 x 13), a last unit of one token, batches beyond the permutation
    # that counts for itself
    (64, 64, 3, 0b111, 257, 2), (576, 64, 5, 0b11111, 300, 3), (128, 64, 16, 0xFFFF, 513, 5),
    (8192, 64, 13, 0x1FFF, 300, 4), (128, 64, 13, 0x1FFF, 8193, 3), (128, 64, 2, 0b11, 9001, 2),
    (320, 64, 12, 0b111111111111, 8192, 8),
    # top-k calls just above the 64 pairs per expert up to which the weight-major GEMM runs beyond 256 tokens
    (128, 64, 16, 0xFFFF, 300, 4), (1024, 256, 16, 0xFFFF, 270, 4),
])
def test_routing_and_permutation_of_large_batches_equal_small_ones(h, f, E, kept, T, k):
    # the same tokens through the small-batch sequences, at most 256 at a time
    build.build()
    W = synth.make_layer_weights(h, f, E, seed=8, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2, kept)
    x = synth.make_tokens(T, h, seed=9, device=DEV)
    stats = binding.RoutingStats(T, E, DEV)
    y = layer.forward(x, 0.5, stats=stats)
    yk, idx, wn, n_active = layer.forward_topk(x, k, 0.2, record=True)
    torch.cuda.synchronize()
    counts = torch.zeros_like(stats.count)
    logits = (x.double() @ W.W_gate.double().T).sort(dim=1, descending=True)
    clear = (logits.values[:, :-1] - logits.values[:, 1:]).min(dim=1).values > 1e-4 if E > 1 else None
    p = torch.exp(logits.values - logits.values[:, :1])
    far = (p[:, 1] - 0.5).abs() > 1e-4
    assert torch.equal(stats.idx[clear].long(), logits.indices[clear, :2])
    assert torch.equal(stats.skipped[clear & far].bool(), p[clear & far, 1] < 0.5)
    assert torch.equal(idx[clear].long(), logits.indices[clear, :k])
    assert torch.allclose(stats.ratio.double(), p[:, 1], atol=1e-4)
    for slot in (0, 1):
        on = stats.idx[:, slot][(stats.skipped == 0) | (slot == 0)]
        counts[:, slot] = torch.bincount(on.long(), minlength=E).to(counts.dtype)
    assert torch.equal(stats.count, counts)
    assert int(stats.n_skipped) == int(stats.skipped.sum())
    assert int(stats.n_experts_touched) == int((counts.sum(1) > 0).sum())
    starts = [0, (T // 512) * 256, T - min(T, 200)]
    for t0 in starts:
        xs = x[t0:t0 + 200].contiguous()
        s = binding.RoutingStats(xs.shape[0], E, DEV)
        ys = layer.forward(xs, 0.5, stats=s)
        yks, idxs, _, nas = layer.forward_topk(xs, k, 0.2, record=True)
        torch.cuda.synchronize()
        same = (s.idx == stats.idx[t0:t0 + 200]).all(1) & (s.skipped == stats.skipped[t0:t0 + 200])
        assert same.float().mean() > 0.95 and rel_l2(ys[same], y[t0:t0 + 200][same]) < 5e-3
        same = (idxs == idx[t0:t0 + 200]).all(1) & (nas == n_active[t0:t0 + 200])
        assert same.float().mean() > 0.95 and rel_l2(yks[same], yk[t0:t0 + 200][same]) < 5e-3
    assert layer.device_status() == 0
    layer.close()


@pytest.mark.parametrize("T,distinct", [(1, 1), (2, 2), (257, 257), (8192, 8192), (8193, 8193), (16385, 16385),
                                        (32769, 32769), (5000, 3), (5001, 1), (40000, 2)])
def test_calibrated_beta_is_the_exact_median_of_the_ratios(weights, T, distinct):
    # repeated tokens make the middle values equal, or put both sides of the middle on two values
    layer = binding.MoeLayer(*weights)
    x = synth.make_tokens(distinct, H, seed=11, device=DEV).repeat((T + distinct - 1) // distinct, 1)[:T].contiguous()
    got = layer.calibrate_beta(x)
    stats = binding.RoutingStats(T, E, DEV)
    layer.forward(x, 0.0, stats=stats)
    r = stats.ratio.double().sort().values
    want = float(((r[(T - 1) // 2] + r[T // 2]) / 2).float())
    # up to 256 tokens forward adds its logits in another order: a few units in the last place
    assert abs(got - want) <= (2e-6 if T <= 256 else 0.0)
    layer.close()


def wide_router_layer(h, offset, narrow, f=64):
    """A layer of width h whose router rows are zero but for `narrow`'s columns, from column `offset` on."""
    E, hn = narrow.shape
    W = synth.make_layer_weights(h, f, E, seed=21, device=DEV)
    Wg = torch.zeros_like(W.W_gate)
    Wg[:, offset:offset + hn] = narrow
    return binding.MoeLayer(Wg, W.W1, W.W3, W.W2), Wg


@pytest.mark.parametrize("E", [3, 5, 8, 16])
@pytest.mark.parametrize("T", [5, 300, 10000])
def test_router_rows_longer_than_shared_memory(E, T):
    # rows of 16384 columns (2 to 8 parts) that are zero but for 1024 columns: a lane's chain of
    # multiply-adds is that of a layer of 1024 columns with zeros added before and behind, so the
    # weights are the same bits wherever the columns lie (first part, across parts, last part), as long
    # as they lie at a multiple of the 512 columns after which the top-k router closes a chain.  The
    # first part ends at column 7680 with 3 experts, 4608 with 5, 2816 with 8 and 2304 with 16 (top-k
    # router: whole rows, 7936, 4864 and 2304).
    # 10000 tokens are several rounds of a block, whose first part then comes round again.
    build.build()
    hn, h, k = 1024, 16384, 3 if T <= 300 else 2
    Wn = synth.make_layer_weights(hn, 64, E, seed=20, device=DEV)
    ref = binding.MoeLayer(Wn.W_gate, Wn.W1, Wn.W3, Wn.W2)
    xn = synth.make_tokens(T, hn, seed=22, device=DEV)
    want = ref.forward_topk(xn, k, 0.1, record=True)[1:]
    beta = ref.calibrate_beta(xn)
    x = torch.ones((T, h), dtype=torch.bfloat16, device=DEV)
    for offset in (0, 2048, 4096, 7168, h - hn):
        layer, Wg = wide_router_layer(h, offset, Wn.W_gate)
        x[:, offset:offset + hn] = xn
        got = layer.forward_topk(x, k, 0.1, record=True)[1:]
        for a, b in zip(got, want):
            assert torch.equal(a, b)
        if T == 300:
            s, sn = binding.RoutingStats(T, E, DEV), binding.RoutingStats(T, E, DEV)
            layer.forward(x, 0.5, stats=s)
            ref.forward(xn, 0.5, stats=sn)
            for name in ("idx", "wn", "ratio", "skipped", "count"):
                assert torch.equal(getattr(s, name), getattr(sn, name))
        assert layer.calibrate_beta(x) == beta
        assert binding.calibrate_beta_noalloc(Wg, x) == beta
        x[:, offset:offset + hn] = 1.0
        assert layer.device_status() == 0
        layer.close()
    ref.close()


def test_allocation_free_calibration_reads_rows_written_just_before(weights):
    # the router rows are the caller's: here a kernel of the stream, which lets its dependents start
    # early, writes other ones before every call; widths on both sides of the shared memory
    for h in (4096, 8192):
        x = synth.make_tokens(500, h, seed=30, device=DEV)
        rows = torch.empty((8, h), dtype=torch.bfloat16, device=DEV)
        src = [synth.make_layer_weights(h, 64, 8, seed=31 + i, device=DEV).W_gate for i in range(6)]
        want = []
        for w in src:
            binding.rmsnorm(w, out=rows)
            torch.cuda.synchronize()
            want.append(binding.calibrate_beta_noalloc(rows, x))
        assert len(set(want)) == len(want)
        for i in list(range(6)) * 4:
            binding.rmsnorm(src[i], out=rows)
            assert binding.calibrate_beta_noalloc(rows, x) == want[i]


@pytest.mark.parametrize("h", [4096, 8192])
@pytest.mark.parametrize("call", ["forward_8192", "topk_333"])
def test_routing_weights_against_64_bits(h, call):
    # A logit of 2 to 4 rounded to fp32 is off by up to 1.2e-7, and what else the weights lose depends on
    # how long the chains of the sum are: 1.2e-7 to 1.4e-7 (2-norm over the batch) with chains of up to 32
    # products, 1.5e-7 and 2.0e-7 with one chain of h / 32 per lane.
    build.build()
    got_err = []
    for seed in range(3):
        W = synth.make_layer_weights(h, 64, 8, seed=50 + seed, device=DEV)
        layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
        T = 8192 if call == "forward_8192" else 333
        x = synth.make_tokens(T, h, seed=90 + seed, device=DEV)
        ranked = (x.double() @ W.W_gate.double().T).sort(dim=1, descending=True)
        if call == "forward_8192":
            k, stats = 2, binding.RoutingStats(T, 8, DEV)
            layer.forward(x, 0.0, stats=stats)
            idx, wn = stats.idx, stats.wn
        else:
            k = 4
            _, idx, wn, _ = layer.forward_topk(x, k, 0.0, record=True)
        same = (idx.long() == ranked.indices[:, :k]).all(1)
        assert same.float().mean() > 0.99
        p = torch.softmax(ranked.values[same, :k], 1)
        got_err.append(float((wn[same].double() - p).norm() / p.norm()))
        assert layer.device_status() == 0
        layer.close()
    assert np.mean(got_err) < 1.45e-7, got_err


def test_long_enumerations_with_one_and_two_tokens_per_warp():
    # 12870 subsets: 512 tokens go one to a warp, 1024 two; the squared losses of the halves add up
    # (fp32 sums of squares of at most two tokens, then fp64: 2e-7 relative)
    build.build()
    W = synth.make_layer_weights(64, 64, 16, seed=41, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    x = synth.make_tokens(1024, 64, seed=42, device=DEV)
    whole, a, b = (np.array(layer.prune_search(t.contiguous(), 8)[0], np.float64) for t in (x, x[:512], x[512:]))
    np.testing.assert_allclose(whole ** 2, a ** 2 + b ** 2, rtol=2e-6)
    layer.close()


@pytest.mark.parametrize("h,f,E,T,k,skew", [
    # up to 64 pairs per expert beyond 256 tokens: the weight-major GEMM, at the line and just beyond it,
    # K-sliced (contraction of 1024) and not, on few experts, and with every token on one expert (three tiles)
    (64, 64, 6, 384, 1, False), (64, 64, 6, 385, 1, False), (128, 448, 5, 257, 1, False), (128, 64, 16, 257, 3, False),
    (1024, 256, 16, 270, 3, False), (128, 448, 6, 384, 1, True), (1024, 1024, 6, 300, 1, True),
])
def test_topk_calls_with_few_pairs_per_expert(h, f, E, T, k, skew):
    build.build()
    W = synth.make_layer_weights(h, f, E, seed=13, device=DEV)
    x = synth.make_tokens(T, h, seed=14, device=DEV)
    if skew:
        W.W_gate[:, 0] = 0
        W.W_gate[2, 0] = 1.0
        x[:, 0] = 64.0
    layers = [binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2),
              layer_with_env((W.W_gate, W.W1, W.W3, W.W2), (1 << E) - 1, MOE_DECODE_KERNEL="td"),
              layer_with_env((W.W_gate, W.W1, W.W3, W.W2), (1 << E) - 1, MOE_DEBUG_SIMT=1)]
    got = [l.forward_topk(x, k, 0.2, record=True) for l in layers]
    again = layers[0].forward_topk(x, k, 0.2)
    torch.cuda.synchronize()
    if skew:
        assert int((got[0][1] == 2).sum()) == T
    assert torch.equal(got[0][0], again)
    for l, g in zip(layers, got):
        for a, b in zip(g[1:], got[0][1:]):
            assert torch.equal(a, b)
        assert rel_l2(got[0][0], g[0]) < 5e-3  # different summation orders, same rounding points
        assert l.device_status() == 0
        l.close()


def test_results_in_pinned_words_with_many_handles_and_threads(weights):
    # more handles than the process' pinned words have slots for, then handles that come and go in threads
    import threading
    x = synth.make_tokens(300, H, seed=51, device=DEV)
    layers = [binding.MoeLayer(*weights) for _ in range(70)]
    want, found = layers[0].calibrate_beta(x), layers[0].prune_search_multi(x, [6, 4])
    for l in layers + layers[60:]:
        assert l.calibrate_beta(x) == want
    for l in layers[::3] + layers[60:]:
        assert l.prune_search_multi(x, [6, 4]) == found
        assert l.calibrate_beta(x) == want and l.device_status() == 0
    for l in layers:
        l.close()
    wrong = []

    def work(seed):
        stream = torch.cuda.Stream(DEV)
        with torch.cuda.stream(stream):
            for i in range(8):
                l = binding.MoeLayer(*weights)
                l.set_stream(stream)
                if any(l.calibrate_beta(x) != want for _ in range(3)) or (i % 3 == seed % 3 and l.prune_search_multi(x, [6, 4]) != found):
                    wrong.append((seed, i))
                l.close()

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def forced(layer, kernel, cap=0):
    assert binding.load_library().moe_test_large_batch(layer._h, kernel, cap) == 0
    return layer


@pytest.mark.parametrize("cap", [0, 1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("h,f", [(128, 448), (576, 320), (1024, 64)])
def test_pair_gemm_equals_the_token_major_one_for_every_token_tile(cap, h, f):
    # Both add up a contraction in the same order, so the bits are the same whatever the tile.  Two kept
    # experts and no skipping: two groups of T tokens, at n tiles of 32 cap tokens, one less and one more
    # (and in between, where the tiles are uneven); weight rows that end inside an item of 512.
    build.build()
    W = synth.make_layer_weights(h, f, 3, seed=61, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2, 0b101)
    step = 32 * (cap or 8)
    n = -(-257 // step)
    sizes = sorted({T for m in (n, n + 1) for T in (m * step - 1, m * step, m * step + 1, m * step + 17) if T > 256})
    x = synth.make_tokens(sizes[-1], h, seed=62, device=DEV)
    for T in sizes:
        xs = x[:T].contiguous()
        want = forced(layer, 2).forward(xs)
        got = forced(layer, 1, cap).forward(xs)
        assert torch.equal(got, want), T
        assert torch.equal(forced(layer, 1, cap).top2_distance(xs), forced(layer, 2).top2_distance(xs))
    assert layer.device_status() == 0
    layer.close()
    # bf16 outputs (the search), ragged groups of all experts
    full = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    for T in (257, 300, 777):
        xs = x[:T].contiguous()
        for r in (2, 3):  # r = 2 evaluates every expert on every token, r = 3 two experts of a token
            assert forced(full, 1, cap).prune_search(xs, r) == forced(full, 2).prune_search(xs, r)
    full.close()


@pytest.mark.parametrize("cap", [0, 1, 5, 8])
@pytest.mark.parametrize("beta", [0.0, 2.0])
def test_pair_gemm_on_skewed_groups(cap, beta):
    # every token on the same two experts of eight (beta = 2: on the first of them alone): groups of 6000
    # tokens beside empty ones, more token tiles than sweep the weight tiles together
    build.build()
    h, f, E, T = 192, 640, 8, 6000
    W = synth.make_layer_weights(h, f, E, seed=63, device=DEV)
    x = synth.make_tokens(T, h, seed=64, device=DEV)
    W.W_gate[:, 0] = 0
    W.W_gate[2, 0], W.W_gate[5, 0] = 2.0, 1.0
    x[:, 0] = 128.0
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    stats = binding.RoutingStats(T, E, DEV)
    got = forced(layer, 1, cap).forward(x, beta, stats=stats)
    torch.cuda.synchronize()
    assert int(stats.count[2, 0]) == T and int(stats.count[5, 1]) == (T if beta == 0 else 0)
    assert torch.equal(got, forced(layer, 2).forward(x, beta))
    dbg = layer_with_env((W.W_gate, W.W1, W.W3, W.W2), MOE_DEBUG_SIMT=1)
    assert rel_l2(got, dbg.forward(x, beta)) < 5e-3
    assert torch.equal(forced(layer, 0).forward(x, beta), got)
    assert layer.device_status() == 0
    layer.close()
    dbg.close()


def test_large_batch_hook_rejects_what_it_does_not_know(weights):
    layer = binding.MoeLayer(*weights)
    lib = binding.load_library()
    for kernel, cap in ((-1, 0), (3, 0), (1, -1), (1, 9)):
        assert lib.moe_test_large_batch(layer._h, kernel, cap) == -1
    assert lib.moe_test_large_batch(None, 0, 0) == -1
    layer.close()


def test_forward_kernel_names_the_kernel_that_runs(weights):
    eight, four = binding.MoeLayer(*weights), binding.MoeLayer(*weights, 0x0F)
    names = [(eight, 1, "gemv_route_gate_up_kernel"), (eight, 2, "gemm_weights_m_kernel"), (eight, 256, "gemm_weights_m_kernel"),
             (four, 79, "gemm_weights_m_kernel"), (four, 80, "gemm_tokens_d_kernel"), (four, 257, "gemm_pair_n_kernel"),
             (eight, 6144, "gemm_pair_n_kernel"), (eight, 6145, "gemm_tokens_m_kernel"), (eight, 0, "")]
    for layer, T, name in names:
        assert layer.forward_kernel(T) == name, T
    eight.close()
    four.close()


def overflow_one_logit(Wg, x):
    """Makes the last expert's logit infinite in fp32, and no other one, on every 16th token (3e38 times 2; the column
    is zero for everyone else).  Returns the mask of those tokens."""
    mask = torch.arange(x.shape[0], device=DEV) % 16 == 7
    Wg[:, 5], x[:, 5] = 0.0, 0.0
    Wg[-1, 5], x[mask, 5] = 2.0, 3e38
    logits = x.float() @ Wg.float().T
    assert torch.isinf(logits[mask, -1]).all()
    assert torch.isfinite(logits[:, :-1]).all() and torch.isfinite(logits[~mask]).all()
    return mask


@pytest.mark.parametrize("h,E,T", [
    # one team per block with tiles of 8 and of 16 tokens, four teams: the lines between them (1184 tokens, 4736, rows
    # of 2048 columns), tiles that end inside a warp's tokens; rows of one block of 64 columns, of fewer blocks than
    # warps, of one more than a round of them; router rows just within shared memory and just beyond it
    (64, 2, 300), (64, 3, 1185), (320, 16, 8200), (1984, 5, 1184), (1984, 7, 1193), (2048, 8, 4736), (2048, 8, 4737),
    (4160, 6, 9473), (4416, 16, 1185), (4480, 16, 1199), (4480, 16, 300), (10944, 4, 1201),
])
def test_router_at_the_edges_of_its_tiles_against_64_bits(h, E, T):
    # A logit of 2 to 4 rounded to fp32 is off by up to 1.2e-7, which is most of what the weights lose; sums of 64
    # products by the tensor core add little to it (0.7e-7 to 1.1e-7 seen, 2-norm over the batch).
    build.build()
    W = synth.make_layer_weights(h, 64, E, seed=70, device=DEV)
    x = synth.make_tokens(T, h, seed=71, device=DEV)
    infinite = overflow_one_logit(W.W_gate, x)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    ranked = (x.double() @ W.W_gate.double().T).sort(dim=1, descending=True)
    k = min(E, 4)
    _, idx, wn, n_active = layer.forward_topk(x, k, 0.0, record=True)
    same = (idx.long() == ranked.indices[:, :k]).all(1)
    # the infinite logit leads, and the others rank behind it as ever (its weight is exp(inf - inf))
    assert (idx[infinite, 0] == E - 1).all() and same[infinite].float().mean() > 0.98
    finite = ~infinite
    assert same[finite].float().mean() > 0.99 and torch.isfinite(wn[finite]).all() and int(n_active.min()) >= 1
    same &= finite
    want = torch.softmax(ranked.values[same, :k], 1)
    assert float((wn[same].double() - want).norm() / want.norm()) < 1.45e-7
    # the median of the ratios: two logits of up to 8 in magnitude, whose last bit is 4.8e-7; the infinite ones have
    # a ratio of 0 (one token in 16: with any other ratio there the median would lie some per cent off)
    ratio = torch.exp(ranked.values[:, 1] - ranked.values[:, 0])
    assert float(ratio[infinite].max()) == 0.0
    s = ratio.sort().values
    want = float((s[(T - 1) // 2] + s[T // 2]) / 2)
    assert abs(layer.calibrate_beta(x) - want) <= 2e-6 * want
    assert layer.device_status() == 0
    layer.close()


@pytest.mark.parametrize("h,r,T", [(8, 2, 300), (72, 5, 1300), (1032, 8, 5000), (4456, 16, 1201)])
def test_allocation_free_calibration_of_ragged_rows_against_64_bits(h, r, T):
    # rows that end inside a block of 64 columns; an infinite logit has a ratio of 0
    Wg = synth.make_layer_weights(max(64, -(-h // 64) * 64), 64, 16, seed=72, device=DEV).W_gate[:r, :h].contiguous()
    x = synth.make_tokens(T, h, seed=73, device=DEV)
    infinite = overflow_one_logit(Wg, x)
    top = (x.double() @ Wg.double().T).sort(dim=1, descending=True).values
    ratio = torch.exp(top[:, 1] - top[:, 0])
    assert float(ratio[infinite].max()) == 0.0
    s = ratio.sort().values
    want = float((s[(T - 1) // 2] + s[T // 2]) / 2)
    got = binding.calibrate_beta_noalloc(Wg, x)
    # of logits of up to 8 in magnitude, whose last bit is 4.8e-7
    assert abs(got - want) <= 2e-6 * want


@pytest.mark.parametrize("h,kept,T,forward_bits", [
    # on either side of the lines of few experts: 74 MiB of tokens with 3 and 4, 2368 tokens with 2, never with 5
    (4096, 4, 9472, False), (4096, 4, 9473, True), (8192, 3, 4737, True), (1536, 2, 2368, False), (1536, 2, 2369, True),
    (4096, 2, 16384, True), (4096, 5, 9473, False), (1024, 3, 40000, False)])
def test_calibration_with_few_experts_takes_the_faster_router(h, kept, T, forward_bits):
    # The forward router's ratios do not depend on the batch; calls of at most 4000 tokens record them.  Both routers
    # give the median within the last bits, the forward router to the bit.
    build.build()
    W = synth.make_layer_weights(h, 64, 8, seed=84, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2, (1 << kept) - 1)
    equal = 0
    for seed in range(85, 90):
        x = synth.make_tokens(T, h, seed=seed, device=DEV)
        ratio = []
        for part in x.tensor_split(-(-T // 4000)):
            stats = binding.RoutingStats(part.shape[0], 8, DEV)
            layer.forward(part.contiguous(), 0.0, stats=stats)
            ratio.append(stats.ratio)
        r = torch.cat(ratio).double().sort().values
        want = float(((r[(T - 1) // 2] + r[T // 2]) / 2).float())
        got = layer.calibrate_beta(x)
        assert abs(got - want) <= 2e-6 * want
        if T <= 16384:
            assert binding.calibrate_beta_noalloc(W.W_gate[:kept].contiguous(), x) == got
        equal += got == want
    assert (equal == 5) if forward_bits else (equal < 5)
    layer.close()


@pytest.mark.parametrize("scale", [1.0, 2.0 ** -6, 2.0 ** -16, 0.0])
@pytest.mark.parametrize("T", [2, 1000, 8193, 20000])
def test_median_of_crowded_ratios(weights, T, scale):
    # the smaller the router's weights the nearer to 1 the ratios: a few candidates per bin, thousands of different
    # values in one bin, one value
    Wg = weights[0] * scale
    layer = binding.MoeLayer(Wg, *weights[1:])
    x = synth.make_tokens(T, H, seed=74, device=DEV)
    stats = binding.RoutingStats(max(T, 300), E, DEV)
    if T < 300:  # the forward call that uses the same router
        x = torch.cat([x, synth.make_tokens(300 - T, H, seed=75, device=DEV)])
    layer.forward(x, 0.0, stats=stats)
    r = stats.ratio[:T].double().sort().values
    assert layer.calibrate_beta(x[:T].contiguous()) == float(((r[(T - 1) // 2] + r[T // 2]) / 2).float())
    layer.close()


def test_subsets_that_travel_with_the_launch_and_subsets_in_memory():
    # 1001 and 1015 subsets go along with the launch, 1092 through memory; six ranked experts a token each time
    build.build()
    W = synth.make_layer_weights(128, 64, 14, seed=76, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    x = synth.make_tokens(300, 128, seed=77, device=DEV)
    alone = layer.prune_search(x, 10)
    for sizes in ([10, 13], [10, 12], [13, 10]):
        found = dict(zip(sizes, layer.prune_search_multi(x, sizes)))
        assert found[10] == alone
    # an expired wait is reported through the losses' way, once
    lib = binding.load_library()
    assert lib.moe_test_wait_expiry(layer._h, 1000, 0) == 0
    with pytest.raises(binding.MoeError):
        layer.prune_search(x, 10)
    assert layer.prune_search(x, 10) == alone
    layer.close()


@pytest.mark.parametrize("E,r,T", [(4, 3, 1), (6, 4, 33), (13, 9, 130), (14, 10, 4100), (14, 9, 37), (16, 12, 129), (16, 8, 5)])
def test_enumerations_of_every_list_length_against_the_oracle(E, r, T):
    # 4 and 15 subsets (less than and not a multiple of the 8 that a block reduces), 715 and 1001 with the launch,
    # 1820 through memory, 2002 and 12870 through memory and pair by pair; 1 to 1025 partial sums per subset
    build.build()
    W = synth.make_layer_weights(128, 64, E, seed=95)
    layer = binding.MoeLayer(*(t.to(DEV) for t in (W.W_gate, W.W1, W.W3, W.W2)))
    x = synth.make_tokens(T, 128, seed=96)
    losses, best = layer.prune_search(x.to(DEV), r)
    b = synth.bf16_bits
    P.check_search(losses, best, O.prune_search_allexperts(b(x), b(W.W_gate), b(W.W1), b(W.W3), b(W.W2), r))
    assert layer.prune_search(x.to(DEV), r) == (losses, best)
    layer.close()


@pytest.mark.parametrize("h,E,T", [(1024, 8, 4095), (1024, 8, 4096), (1600, 4, 2700), (2560, 8, 2047), (2560, 8, 2049), (4096, 8, 1025)])
def test_host_calls_in_column_slabs_equal_the_device_call(h, E, T):
    # below the line, two and four slabs, slabs of different widths, a last slab that ends inside a weight tile
    build.build()
    W = synth.make_layer_weights(h, 1024, E, seed=78, device=DEV)  # (with fewer features the line is at 8 Mi values)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    x = synth.make_tokens(T, h, seed=79, device=DEV)
    want = layer.forward(x, 0.3).cpu()
    pinned, pageable = (torch.zeros_like(want).pin_memory(), torch.zeros_like(want))
    for y in (pinned, pageable, pinned):
        y.zero_()
        assert torch.equal(layer.forward_host(x.cpu().pin_memory(), 0.3, y), want)
    assert layer.device_status() == 0
    layer.close()


@pytest.mark.parametrize("h,f,E,sizes", [
    # (tokens, slabs): 4 Mi values with many features, 8 Mi with few; two and four slabs, fewer tiles than four, a last
    # slab that ends inside a weight tile, more pairs per expert than the pair kernel's down projection takes
    (1024, 1024, 2, [(4095, 1), (4096, 2), (4097, 1)]), (1600, 1024, 4, [(2621, 1), (2622, 3)]),
    (2560, 1024, 8, [(1638, 1), (1639, 2), (2047, 2), (2048, 4)]), (2560, 960, 8, [(2560, 1), (3277, 4)]),
    (448, 1024, 8, [(9400, 1)])])
def test_lines_of_the_column_slabs(h, f, E, sizes):
    build.build()
    W = synth.make_layer_weights(h, f, E, seed=93, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    for T, slabs in sizes:
        assert binding.load_library().moe_test_host_slabs(layer._h, T) == slabs, T
        x = synth.make_tokens(T, h, seed=94, device=DEV)
        y = torch.zeros_like(x, device="cpu").pin_memory()
        assert torch.equal(layer.forward_host(x.cpu().pin_memory(), 0.3, y), layer.forward(x, 0.3).cpu()), T
    assert layer.device_status() == 0
    layer.close()


def test_stage_times_of_host_calls_in_column_slabs():
    # every slab has a down GEMM and a combine of its own.  Four slabs of a layer whose down GEMM (0.25 TFLOP, 0.15 ms
    # and more) takes several times what the combine (0.05 GB) does: with the GEMMs of three slabs in its stage, the
    # combine would seem three times as long as the GEMM.
    build.build()
    W = synth.make_layer_weights(2048, 14336, 2, seed=82, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2)
    x = synth.make_tokens(2100, 2048, seed=83, device=DEV)
    xh, yh = x.cpu().pin_memory(), torch.empty(x.shape, dtype=x.dtype).pin_memory()
    layer.forward(x)
    layer.forward_host(xh, 0.0, yh)
    for call in (lambda: layer.forward(x), lambda: layer.forward_host(xh, 0.0, yh)):
        layer.profile_enable(True)
        for _ in range(5):
            call()
        ms, calls = layer.profile_read()
        assert calls == 5 and min(ms[:4]) > 0
        assert ms[3] < 0.8 * ms[2], ms
        assert layer.profile_read()[1] == 0   # a window of its own
    layer.profile_enable(False)
    layer.close()


@pytest.mark.parametrize("h", [448, 512])
def test_large_groups_on_either_side_of_the_width_line(h):
    # two kept experts, no skipping: groups of T tokens beyond the line of the narrow layers
    build.build()
    W = synth.make_layer_weights(h, 192, 3, seed=80, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2, 0b110)
    line = 8192 if h >= 512 else 1536
    assert layer.forward_kernel(line) == "gemm_pair_n_kernel" and layer.forward_kernel(line + 1) == "gemm_tokens_m_kernel"
    for T in (1537, 2400, 4096, 4097, 8193):  # from 4097 to 8192 on the wide rows: gate/up on the pairs alone
        x = synth.make_tokens(T, h, seed=81, device=DEV)
        want = layer.forward(x)
        for kernel in (1, 2, 0):
            assert torch.equal(forced(layer, kernel).forward(x), want)
    assert layer.device_status() == 0
    layer.close()


@pytest.mark.parametrize("f,line", [(64, 4096), (128, 4096), (192, 8192)])
def test_large_groups_of_experts_with_few_features(f, line):
    # two kept experts, no skipping: groups of T tokens; beyond the line everything is the token-major kernel's
    build.build()
    W = synth.make_layer_weights(512, f, 3, seed=91, device=DEV)
    layer = binding.MoeLayer(W.W_gate, W.W1, W.W3, W.W2, 0b011)
    assert layer.forward_kernel(line) == "gemm_pair_n_kernel" and layer.forward_kernel(line + 1) == "gemm_tokens_m_kernel"
    for T in (4096, 4097, 4225):
        x = synth.make_tokens(T, 512, seed=92, device=DEV)
        want = layer.forward(x)
        for kernel in (1, 2, 0):
            assert torch.equal(forced(layer, kernel).forward(x), want)
    assert layer.device_status() == 0
    layer.close()
