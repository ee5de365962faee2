"""GPU parity: the CUDA path, called through the C ABI, against the CPU oracle on the same seeded
inputs.  Integers (X_q, W_q, Int32 accumulators, scales' bits) must match exactly; fp32 outputs
within 1e-5 of the output magnitude."""
import gc

import numpy as np
import pytest
import torch

from oracle import q8_oracle as o
from paper_1910_06188_b200 import binding as q8
from paper_1910_06188_b200 import synth
from tests.gpu_util import REL_TOL, assert_close_fp, check_linear, dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _no_garbage_left_behind():
    """Tensors that earlier tests left in reference cycles are freed here, not while another test counts allocations."""
    yield
    gc.collect()


# ------------------------------------------------------------------ quantiser (Eq. 1, Eq. 3, Sec. 4.1)
@pytest.mark.parametrize("n", [1, 3, 4, 5, 15, 16, 17, 1023, 4096, 100_003, 1 << 20])
def test_quantize_dynamic_bit_exact(n):
    x = synth.activation(1, n, seed=100 + n).reshape(-1)
    xq, S = q8.q8_quantize_activation(dev(x))
    S_ref, _ = o.scale_from_absmax(o.absmax(x))
    assert S.cpu().numpy()[0] == S_ref
    assert np.array_equal(xq.cpu().numpy(), o.quantize(x, S_ref))


def test_quantize_static_scale_ties_clamp_and_nonfinite():
    x = np.concatenate([
        np.arange(-300, 301, dtype=np.float32) * 0.5,
        np.array([np.nan, np.inf, -np.inf, 1e30, -1e30, 0.0, -0.0], np.float32),
        synth.activation(1, 5000, seed=5).reshape(-1) * 20,
    ]).astype(np.float32)
    for S in (1.0, 0.5, 3.1875, float(np.float32(1) / np.float32(3))):
        Sd = dev(np.array([S], np.float32))
        xq, _ = q8.q8_quantize_activation(dev(x), Sd)
        got = xq.cpu().numpy()
        assert np.array_equal(got, o.quantize(x, S))
        assert got.min() >= -127


def test_quantize_unaligned_pointer_uses_scalar_kernel():
    x = synth.activation(1, 1000, seed=9).reshape(-1)
    buf = torch.zeros(1001, dtype=torch.float32, device="cuda")
    buf[1:] = dev(x)
    xq, S = q8.q8_quantize_activation(buf[1:])
    S_ref, _ = o.scale_from_absmax(o.absmax(x))
    assert S.cpu().numpy()[0] == S_ref
    assert np.array_equal(xq.cpu().numpy(), o.quantize(x, S_ref))


def test_zero_tensor_flags_scale():
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    x = torch.zeros(1000, dtype=torch.float32, device="cuda")
    xq, S = q8.q8_quantize_activation(x, dev_status=status)
    code, bits = q8.q8_poll_status(status)
    assert code == q8.Q8_ERR_SCALE and bits == 1 << q8.Q8_ERR_SCALE
    assert S.cpu().numpy()[0] == 1.0 and not xq.any()
    assert q8.q8_poll_status(status) == (q8.Q8_OK, 0)  # polling clears the word


@pytest.mark.parametrize("shape", [(1, 1), (7, 13), (768, 768), (3072, 768)])
def test_quantize_weight(shape):
    W = synth.weight(shape[0], shape[1], seed=200 + shape[0])
    Wq, S_w = q8.q8_quantize_weight(dev(W))
    Wq_ref, S_ref, _ = o.quantize_weight(W)
    assert S_w.cpu().numpy()[0] == S_ref
    assert np.array_equal(Wq.cpu().numpy(), Wq_ref)


# ------------------------------------------------------------------ Eq. 4
def test_calibrate_matches_oracle_ema():
    state = q8.new_calibrate_state()
    ref = o.EmaState()
    decay = 0.9999
    for i in range(6):
        x = synth.activation(64, 96, seed=300 + i) * np.float32(1.0 + 0.3 * i)
        q8.q8_calibrate(dev(x), decay, state)
        ref.update(o.absmax(x), decay)
        words = state.cpu()
        ema, S_x = words.view(torch.float32)[0].item(), words.view(torch.float32)[1].item()
        assert np.float32(ema) == ref.ema[0] and np.float32(S_x) == ref.S_x
        assert words[2].item() == i + 1 and words[4].item() == 0
    assert q8.calibrate_S_x(state).cpu().numpy()[0] == ref.S_x


def test_calibrate_decay_zero_is_dynamic_and_zero_batch_flags():
    state = q8.new_calibrate_state()
    ref = o.EmaState()
    for i, g in enumerate((3.0, 0.5, 7.0)):
        x = synth.activation(8, 40, seed=310 + i) * np.float32(g)
        q8.q8_calibrate(dev(x), 0.0, state)
        ref.update_batch(x, 0.0)
        got = state.view(torch.float32)[1].item()
        # decay 0 keeps no history: exactly the dynamic scale of Sec. 4.1 for this batch
        assert np.float32(got) == ref.S_x == np.float32(127.0) / o.absmax(x)
    # an empty batch is no observation: state (ema, S_x, n_batches) unchanged, nothing launched
    before = state.clone()
    q8.q8_calibrate(torch.empty(0, device="cuda"), 0.5, state)
    assert q8.q8_last_launch_info()["launches"] == 0 and torch.equal(state, before)
    assert ref.update_batch(np.zeros(0, np.float32), 0.5) == np.float32(state.view(torch.float32)[1].item())
    state = q8.new_calibrate_state()
    q8.q8_calibrate(torch.zeros(100, device="cuda"), 0.9, state)
    assert state[4].item() == 1 << q8.Q8_ERR_SCALE and state.view(torch.float32)[1].item() == 1.0


# ------------------------------------------------------------------ quantised FC, small / ragged / tile-boundary shapes
SHAPES = [
    (1, 8, 16), (1, 1, 16), (5, 3, 32), (128, 128, 128), (129, 130, 144), (127, 255, 48), (256, 64, 16),
    (300, 200, 400), (33, 257, 272), (260, 520, 1040), (1000, 96, 2064),
]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("mode", ["dynamic", "static"])
def test_linear_small_shapes(M, N, K, mode):
    X = synth.activation(M, K, seed=400 + M + N + K)
    W = synth.weight(N, K, seed=401 + M + N + K)
    b = synth.bias(N, seed=402 + M + N + K)
    S_x = None if mode == "dynamic" else float(np.float32(127.0) / np.float32(6.0))  # clamps the x8 outliers
    info = check_linear(X, W, b, act=(M + N) % 2, S_x=S_x)
    assert info["gemm_kernel"] == 1, "K % 16 == 0 shapes must run the tcgen05 kernel"


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (3, 5, 7), (64, 64, 100), (130, 70, 33), (17, 200, 1001)])
def test_linear_generic_shapes(M, N, K):
    X = synth.activation(M, K, seed=500 + M)
    W = synth.weight(N, K, seed=501 + M)
    b = synth.bias(N, seed=502 + M)
    info = check_linear(X, W, b, act=1)
    assert info["gemm_kernel"] == 2, "K % 16 != 0 must fall back to the generic kernel"


def test_linear_no_bias_and_forced_generic_agree():
    X = synth.activation(200, 256, seed=600)
    W = synth.weight(300, 256, seed=601)
    check_linear(X, W, None, act=0)
    check_linear(X, W, None, act=1, fn=q8.q8_linear_generic)


def test_linear_integer_inputs_reduce_to_exact_matmul():
    rng = np.random.default_rng(5)
    M, N, K = 150, 90, 160
    X = rng.integers(-127, 128, size=(M, K)).astype(np.float32)
    Wq = rng.integers(-127, 128, size=(N, K), dtype=np.int8)
    b = rng.integers(-1000, 1000, size=N).astype(np.float32)
    one = dev(np.ones(1, np.float32))
    acc = torch.empty((M, N), dtype=torch.int32, device="cuda")
    Y = q8.q8_linear(dev(X), dev(Wq), one, one, dev(b), 0, dbg_acc=acc)
    want = X.astype(np.int64) @ Wq.astype(np.int64).T + b.astype(np.int64)
    assert np.array_equal(acc.cpu().numpy().astype(np.int64), want)
    assert np.array_equal(Y.cpu().numpy().astype(np.float64), want.astype(np.float64))


def test_linear_saturated_accumulator():
    # all-127 rows: acc = 16129 * K, the largest value the path can produce for this K
    M, N, K = 128, 64, 4096
    X = np.full((M, K), 127.0, np.float32)
    X[1::2] *= -1
    Wq = np.full((N, K), 127, np.int8)
    one = dev(np.ones(1, np.float32))
    acc = torch.empty((M, N), dtype=torch.int32, device="cuda")
    q8.q8_linear(dev(X), dev(Wq), one, one, None, 0, dbg_acc=acc)
    got = acc.cpu().numpy()
    assert np.all(got[0::2] == 66064384) and np.all(got[1::2] == -66064384)


def test_linear_q_matches_linear():
    M, N, K = 256, 384, 512
    X = synth.activation(M, K, seed=700)
    W = synth.weight(N, K, seed=701)
    b = synth.bias(N, seed=702)
    Wq, S_w = q8.q8_quantize_weight(dev(W))
    Xq, S_x = q8.q8_quantize_activation(dev(X))
    Y1 = q8.q8_linear_q(Xq, S_x, Wq, S_w, dev(b), 1)
    Y2 = q8.q8_linear(dev(X), Wq, S_w, None, dev(b), 1)
    assert torch.equal(Y1, Y2)


def test_linear_is_deterministic():
    X, W, b = synth.activation(512, 768, 800), synth.weight(768, 768, 801), synth.bias(768, 802)
    Wq, S_w = q8.q8_quantize_weight(dev(W))
    Xd, bd = dev(X), dev(b)
    Y1 = q8.q8_linear(Xd, Wq, S_w, None, bd, 1).clone()
    Y2 = q8.q8_linear(Xd, Wq, S_w, None, bd, 1)
    assert torch.equal(Y1, Y2)


def test_device_side_errors_are_returned_as_codes():
    X = torch.zeros((8, 16), device="cuda")
    Wq = torch.ones((4, 16), dtype=torch.int8, device="cuda")
    S_w = torch.ones(1, device="cuda")
    ws = q8.new_workspace(8, 4, 16)
    Y = q8.q8_linear(X, Wq, S_w, None, None, 0, workspace=ws)      # max|X| == 0
    assert q8.q8_poll_status(ws)[0] == q8.Q8_ERR_SCALE and not Y.any()
    # a caller-supplied static scale that is zero, negative, NaN or infinite is reported the same way
    Xr = torch.randn((8, 16), device="cuda")
    for bad in (0.0, -3.0, float("nan"), float("inf")):
        q8.q8_linear(Xr, Wq, S_w, torch.full((1,), bad, device="cuda"), None, 0, workspace=ws)
        assert q8.q8_poll_status(ws)[0] == q8.Q8_ERR_SCALE, bad
        st = torch.zeros(1, dtype=torch.int32, device="cuda")
        q8.q8_quantize_activation(Xr, torch.full((1,), bad, device="cuda"), dev_status=st)
        assert q8.q8_poll_status(st)[0] == q8.Q8_ERR_SCALE, bad
    q8.q8_linear(Xr, Wq, S_w, torch.full((1,), 2.5, device="cuda"), None, 0, workspace=ws)
    assert q8.q8_poll_status(ws) == (q8.Q8_OK, 0)
    with pytest.raises(q8.Q8Error) as e:
        q8.q8_linear(X, Wq, S_w, None, None, 0, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    assert e.value.status == q8.Q8_ERR_WORKSPACE
    with pytest.raises(q8.Q8Error) as e:
        q8.q8_linear(X, Wq, S_w, None, None, 3)
    assert e.value.status == q8.Q8_ERR_ARG


@pytest.mark.parametrize("M,K,N", [(128, 768, 768), (256, 768, 96), (1, 16, 8), (37, 96, 40), (4, 48, 32), (255, 768, 64)])
def test_small_dynamic_layer_is_two_launches_and_matches_the_oracle(M, K, N):
    """A small activation (up to 256 x 768 values) is abs-maxed, scaled and quantised by one cluster in one launch
    (Sec. 4.1 + Eq. 1), so the whole dynamic layer is two kernels; same bits as the oracle, call after call."""
    X = synth.activation(M, K, seed=700 + M)
    W = synth.weight(N, K, seed=701 + M)
    b = synth.bias(N, seed=702 + M)
    for _ in range(2):
        info = check_linear(X, W, b, act=1)
        assert info["launches"] == 2
    # all-zero and non-finite activations: scale forced to 1, flagged, no NaN in the Int8 tensor
    Wq, S_w = q8.q8_quantize_weight(dev(W))
    ws = q8.new_workspace(M, N, K)
    xq = torch.empty((M, K), dtype=torch.int8, device="cuda")
    q8.q8_linear(torch.zeros((M, K), device="cuda"), Wq, S_w, None, dev(b), 0, workspace=ws, dbg_Xq=xq)
    assert q8.q8_poll_status(ws)[0] == q8.Q8_ERR_SCALE and not xq.any()
    Xi = dev(X).clone()
    Xi[0, 0] = float("inf")
    Xi[0, 1] = float("nan")
    q8.q8_linear(Xi, Wq, S_w, None, dev(b), 0, workspace=ws, dbg_Xq=xq)
    assert q8.q8_poll_status(ws)[0] == q8.Q8_ERR_SCALE
    assert np.array_equal(xq.cpu().numpy(), o.quantize(Xi.cpu().numpy(), 1.0))
    q8.q8_linear(dev(X), Wq, S_w, None, dev(b), 0, workspace=ws)        # and the next call starts clean
    assert q8.q8_poll_status(ws) == (q8.Q8_OK, 0)


# ------------------------------------------------------------------ the paper-shaped configurations
def test_config_single_layer_dynamic():
    """X [128 x 768] with x8 outliers, W [768 x 768], bias; dynamic S_x (Sec. 4.1)."""
    X = synth.activation(128, 768, synth.seed_for(1, 0))
    W = synth.weight(768, 768, synth.seed_for(1, 1))
    b = synth.bias(768, synth.seed_for(1, 2))
    info = check_linear(X, W, b, act=0)
    assert info["gemm_kernel"] == 1


@pytest.mark.parametrize("name,K,N,act", synth.fc_set(768, 3072))
def test_config_bert_base_fc_set(name, K, N, act):
    """BERT-Base FC set at 32 x 128 tokens, S_x from one seeded calibration batch (Eq. 4)."""
    M = 4096
    idx = [n for n, *_ in synth.fc_set(768, 3072)].index(name)
    X = synth.activation(M, K, synth.seed_for(2, 10 * idx))
    calib = synth.activation(M, K, synth.seed_for(2, 10 * idx + 1))
    W = synth.weight(N, K, synth.seed_for(2, 10 * idx + 2))
    b = synth.bias(N, synth.seed_for(2, 10 * idx + 3))
    state = q8.new_calibrate_state()
    q8.q8_calibrate(dev(calib), 0.9999, state)
    ref = o.EmaState()
    S_x = ref.update(o.absmax(calib), 0.9999)
    assert q8.calibrate_S_x(state).cpu().numpy()[0] == S_x
    info = check_linear(X, W, b, act=act, S_x=float(S_x), canary=False)
    assert info["gemm_kernel"] == 1


# ------------------------------------------------------------------ embedding (Sec. 3)
@pytest.mark.parametrize("V,H,T", [(50, 24, 31), (1000, 768, 4096), (77, 10, 200), (30522, 1024, 3000)])
def test_embedding(V, H, T):
    E = synth.embedding_table(V, H, seed=900 + H)
    ids = synth.token_ids(T, V, seed=901 + H)
    Eq, S_e = q8.q8_quantize_weight(dev(E))
    Eq_ref, S_ref, _ = o.quantize_weight(E)
    assert np.array_equal(Eq.cpu().numpy(), Eq_ref) and S_e.cpu().numpy()[0] == S_ref
    rows = torch.empty((T, H), dtype=torch.int8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = q8.q8_embedding(dev(ids), Eq, S_e, rows_q=rows, dev_status=status)
    rows_ref, out_ref, bad = o.embedding(ids, Eq_ref, S_ref)
    assert bad == 0 and q8.q8_poll_status(status) == (q8.Q8_OK, 0)
    assert np.array_equal(rows.cpu().numpy(), rows_ref)
    assert_close_fp(out.cpu().numpy(), out_ref, "embedding")


def test_embedding_bad_ids_are_flagged_and_zeroed():
    V, H, T = 40, 32, 20
    E = synth.embedding_table(V, H, seed=950)
    ids = synth.token_ids(T, V, seed=951)
    ids[3], ids[11] = -1, V
    Eq, S_e = q8.q8_quantize_weight(dev(E))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = q8.q8_embedding(dev(ids), Eq, S_e, dev_status=status)
    assert q8.q8_poll_status(status)[0] == q8.Q8_ERR_INDEX
    rows_ref, out_ref, bad = o.embedding(ids, Eq.cpu().numpy(), S_e.cpu().numpy()[0])
    assert bad == 2
    got = out.cpu().numpy()
    assert not got[3].any() and not got[11].any()
    assert_close_fp(got, out_ref, "embedding with bad ids")


# ------------------------------------------------------------------ training-mode pieces (Sec. 2.2, Eq. 5)
@pytest.mark.parametrize("n", [1, 7, 4096, 100_003])
def test_fake_quantize_and_ste(n):
    x = synth.activation(1, n, seed=1300 + n).reshape(-1)
    state = q8.new_calibrate_state()
    q8.q8_calibrate(dev(x), 0.9, state)                       # the EMA update training does on every forward
    S = q8.calibrate_S_x(state)
    xh = q8.q8_fake_quantize(dev(x), S).cpu().numpy()
    S_ref, _ = o.scale_from_absmax(o.absmax(x))
    assert S.item() == S_ref
    ref = o.fake_quantize(x, S_ref)
    assert np.abs(xh - ref).max() <= 1e-6 * max(np.abs(ref).max(), 1e-30)
    # the fake-quantised values sit exactly on the Int8 grid of the real quantiser
    assert np.array_equal(np.rint(xh.astype(np.float64) * float(S_ref)).astype(np.int8), o.quantize(x, S_ref))
    g = synth.normal((n,), 1.0, 1400 + n)
    assert np.array_equal(q8.q8_ste_backward(dev(g)).cpu().numpy(), g)
    gd = dev(g)
    assert q8.q8_ste_backward(gd, gd).data_ptr() == gd.data_ptr()


@pytest.mark.parametrize("n", [3, 2049, 100_003])
def test_straight_through_copy_by_kernel_and_by_the_runtime(n):
    """One launch for aligned memory of the device, also where a stream is captured; addresses off 16 bytes on either side and pinned host
    memory go to the runtime's copy, which counts as no launch."""
    g = dev(synth.normal((n,), 1.0, 1450))
    assert torch.equal(q8.q8_ste_backward(g), g) and q8.q8_last_launch_info()["launches"] == 1
    for off_in, off_out in ((1, 0), (0, 1), (2, 2), (3, 1)):
        src, room = torch.zeros(n + 4, device="cuda"), torch.full((n + 8,), 9.0, device="cuda")
        src[off_in:off_in + n] = g
        q8.q8_ste_backward(src[off_in:off_in + n], room[off_out:off_out + n])
        assert q8.q8_last_launch_info()["launches"] == 0
        assert torch.equal(room[off_out:off_out + n], g)
        assert bool((room[:off_out] == 9.0).all()) and bool((room[off_out + n:] == 9.0).all())
    pinned, out = torch.empty(n, pin_memory=True), torch.zeros(n, device="cuda")
    pinned.copy_(g)
    torch.cuda.synchronize()
    assert q8.load().q8_ste_backward(pinned.data_ptr(), n, out.data_ptr(), torch.cuda.current_stream().cuda_stream) == q8.Q8_OK
    assert torch.equal(out, g)
    graph, moved, off = torch.cuda.CUDAGraph(), torch.zeros(n, device="cuda"), torch.zeros(n + 1, device="cuda")
    with torch.cuda.graph(graph):
        q8.q8_ste_backward(g, moved)
        q8.q8_ste_backward(g, off[1:])
    g.mul_(-3.0)
    graph.replay()
    assert torch.equal(moved, g) and torch.equal(off[1:], g)


# ------------------------------------------------------------------ one weight scale per fused layer (Eq. 3 per layer)
@pytest.mark.parametrize("M,H,seg,act", [(300, 128, 128, 0), (515, 256, 256, 1), (64, 40, 40, 0)])
def test_fused_projection_with_per_layer_scales_equals_separate_layers(M, H, seg, act):
    """Q, K and V stored as one [3H, H] matrix with one S_w per block of H rows must give what three separate
    quantised FC layers give (the paper's model has three layers, each with its own Eq. 3 scale)."""
    X = synth.activation(M, H, seed=1500 + M)
    Ws = [synth.normal((H, H), 0.02 * (1 + 2 * i), 1501 + M + i) for i in range(3)]   # different ranges per layer
    bs = [synth.bias(H, 1510 + M + i) for i in range(3)]
    W, b = np.concatenate(Ws), np.concatenate(bs)
    Wq, S_w = q8.q8_quantize_weight_segments(dev(W), seg)
    acc = torch.empty((M, 3 * H), dtype=torch.int32, device="cuda")
    Y = q8.q8_linear_wseg(dev(X), Wq, S_w, seg, None, dev(b), act, dbg_acc=acc)
    info = q8.q8_last_launch_info()
    assert info["gemm_kernel"] == (1 if seg % 32 == 0 else 2)
    for i in range(3):
        Wq_ref, S_ref, _ = o.quantize_weight(Ws[i])
        assert S_w[i].item() == S_ref and np.array_equal(Wq[i * H:(i + 1) * H].cpu().numpy(), Wq_ref)
        ref = o.linear(X, Wq_ref, S_ref, None, bs[i], act)
        assert np.array_equal(acc[:, i * H:(i + 1) * H].cpu().numpy(), ref["acc"])
        assert_close_fp(Y[:, i * H:(i + 1) * H].cpu().numpy(), ref["y"], f"segment {i}")
    Xq, S_x = q8.q8_quantize_activation(dev(X))
    assert torch.equal(q8.q8_linear_q_wseg(Xq, S_x, Wq, S_w, seg, dev(b), act), Y)


# ------------------------------------------------------------------ routes of the dynamic scale
@pytest.mark.parametrize("n", [1, 3, 4, 4095, 196607, 196608, 196612, 300001, 1 << 20, (2 << 20) - 1, 2 << 20, (2 << 20) + 5,
                               (4 << 20) - 1, 4 << 20, (4 << 20) + 5, 148 * 8 * 4096 + 5, 2 * 148 * 8 * 4096 + 12343])
@pytest.mark.parametrize("peak_at", ["first", "last"])
def test_dynamic_quantisation_in_one_or_several_launches(n, peak_at):
    """One cluster, one cooperative grid or separate passes (by size): the same integers, the same scale, and the largest
    value is found wherever it lies; a zero tensor flags the scale without clearing the caller's status word."""
    x = synth.normal((n,), 1.0, 9000 + n % 1000)
    x[0 if peak_at == "first" else -1] = -9.0
    xq, s = q8.q8_quantize_activation(dev(x))
    s_ref, _ = o.scale_from_absmax(o.absmax(x))
    assert s.cpu().numpy()[0] == s_ref
    assert np.array_equal(xq.cpu().numpy(), o.quantize(x, s_ref))
    word = torch.full((1,), 1 << 20, dtype=torch.int32, device="cuda")
    zq, zs = q8.q8_quantize_activation(torch.zeros(n, device="cuda"), dev_status=word)
    assert zs.item() == 1.0 and not zq.any() and word.item() == (1 << 20) | (1 << q8.Q8_ERR_SCALE)


@pytest.mark.parametrize("n", [196612, 1 << 20, (2 << 20) - 1])
def test_dynamic_quantisation_where_the_cooperative_launch_is_refused(n):
    """As in a process that may use a part of the SMs only: the separate passes give the same values, and no error stays behind."""
    x = dev(synth.normal((n,), 1.0, 9050))
    want, s_want = q8.q8_quantize_activation(x)
    assert q8.q8_last_launch_info()["launches"] == 1
    try:  # (an SM holds 2048 threads, eight of its CTAs: nine for each SM are refused before anything is launched)
        q8.q8_tune_quantize_grid(9 * torch.cuda.get_device_properties(0).multi_processor_count)
        got, s_got = q8.q8_quantize_activation(x)
        assert q8.q8_last_launch_info()["launches"] == 3
        assert torch.equal(got, want) and torch.equal(s_got, s_want)
        Wq, S_w = q8.q8_quantize_weight(x.view(1, n))
        assert torch.equal(Wq.view(-1), want) and torch.equal(S_w, s_want)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):  # (a launch that is refused would end the capture)
            captured, s_captured = q8.q8_quantize_activation(x)
        graph.replay()
        assert torch.equal(captured, want) and torch.equal(s_captured, s_want)
    finally:
        q8.q8_tune_quantize_grid(0)
    torch.cuda.synchronize()
    assert torch.equal(q8.q8_quantize_activation(x)[0], want)


@pytest.mark.parametrize("M,K", [(1, 13), (3, 65537), (257, 768), (1000, 300), (4096, 1040), (8192, 1024), (8192, 1040),
                                 (7168, 1024), (7169, 1024), (9000, 1040), (14300, 1024)])
def test_dynamic_linear_finds_the_peak_of_every_share(M, K):
    """The partial maxima of the abs-max pass: the scale is that of the largest value, in whichever CTA's share it lies."""
    W = synth.weight(16, K, 9100)
    for at in (0, M * K // 2, M * K - 1):
        x = synth.normal((M, K), 1.0, 9101)
        x.flat[at] = 11.0
        Wq, S_w = q8.q8_quantize_weight(dev(W))
        buf = torch.empty(M * K + 1, device="cuda")
        for off in (0, 1):  # (off 16 bytes a thread loads a value at a time)
            X = buf[off:M * K + off].view(M, K)
            X.copy_(torch.from_numpy(x))
            ws = q8.new_workspace(M, 16, K)
            q8.q8_linear(X, Wq, S_w, None, None, 0, workspace=ws)
            assert ws[4:8].view(torch.float32).item() == np.float32(127.0) / np.float32(11.0)
            assert q8.q8_poll_status(ws) == (q8.Q8_OK, 0)


@pytest.mark.parametrize("n", [1, 5, 1023, 4096, 1 << 20, (1 << 20) + 3])
def test_calibration_leaves_its_counter_at_zero_and_fake_quantisation_divides_exactly(n):
    x = synth.activation(1, n, 9200)[0]
    state = q8.new_calibrate_state()
    for _ in range(3):
        q8.q8_calibrate(dev(x), 0.9999, state)
    words = state.cpu().numpy()
    assert words[2] == 3 and words[3] == 0 and not words[4:].any()
    S = np.float32(127.0) / np.abs(x).max()
    assert q8.calibrate_S_x(state).item() == S
    got = q8.q8_fake_quantize(dev(x), q8.calibrate_S_x(state)).cpu().numpy()
    assert np.array_equal(got, o.quantize(x, S).astype(np.float32) / S)


# ------------------------------------------------------------------ operands that TMA cannot fetch
@pytest.mark.parametrize("K", [8, 24, 56, 72, 4, 20, 132, 1, 3, 63, 65, 129, 1001])
@pytest.mark.parametrize("M,N", [(1, 1), (63, 65), (65, 130), (1700, 1665)])
def test_generic_gemm_pieces_and_tile_edges(M, N, K):
    """Pieces of 8, 4 and single bytes of K, both tile sizes (1700 x 1665: more than 148 of 128 x 128), ragged everywhere."""
    rng = np.random.default_rng(K * 7 + M)
    Xq, Wq = (rng.integers(-127, 128, size=(n, K), dtype=np.int8) for n in (M, N))
    acc = torch.empty((M, N), dtype=torch.int32, device="cuda")
    q8.q8_linear_q(dev(Xq), torch.ones(1, device="cuda"), dev(Wq), torch.ones(1, device="cuda"), None, 0, dbg_acc=acc)
    assert q8.q8_last_launch_info()["gemm_kernel"] == 2
    assert np.array_equal(acc.cpu().numpy(), Xq.astype(np.int32) @ Wq.astype(np.int32).T)


@pytest.mark.parametrize("N,tile", [(1, 64), (64, 64), (65, 64), (128, 64), (129, 128)])
def test_generic_gemm_tall_and_narrow(N, tile):
    M, K = 20003, 20
    rng = np.random.default_rng(N)
    Xq, Wq = (rng.integers(-127, 128, size=(n, K), dtype=np.int8) for n in (M, N))
    acc = torch.empty((M, N), dtype=torch.int32, device="cuda")
    q8.q8_linear_q(dev(Xq), torch.ones(1, device="cuda"), dev(Wq), torch.ones(1, device="cuda"), None, 0, dbg_acc=acc)
    info = q8.q8_last_launch_info()
    assert (info["gemm_kernel"], info["block_n"]) == (2, tile)
    assert np.array_equal(acc.cpu().numpy(), Xq.astype(np.int32) @ Wq.astype(np.int32).T)


@pytest.mark.parametrize("offset_x,offset_w", [(8, 0), (4, 8), (1, 0), (0, 3), (2, 1)])
def test_generic_gemm_pointers_at_any_byte(offset_x, offset_w):
    M, N, K = 70, 66, 96
    rng = np.random.default_rng(77)
    Xq, Wq = (rng.integers(-127, 128, size=(n, K), dtype=np.int8) for n in (M, N))

    def at(a, offset):
        buf = torch.empty(a.size + offset, dtype=torch.int8, device="cuda")
        buf[offset:] = dev(a).reshape(-1)
        return buf[offset:].view(a.shape)

    acc = torch.empty((M, N), dtype=torch.int32, device="cuda")
    Y = torch.empty(M * N + 1, device="cuda")[1:].view(M, N)  # 4-byte aligned output: no 8-byte stores
    one = torch.ones(1, device="cuda")
    q8.q8_linear_q(at(Xq, offset_x), one, at(Wq, offset_w), one, None, 0, Y=Y, dbg_acc=acc)
    ref = Xq.astype(np.int32) @ Wq.astype(np.int32).T
    assert np.array_equal(acc.cpu().numpy(), ref) and np.array_equal(Y.cpu().numpy(), ref.astype(np.float32))


# ------------------------------------------------------------------ native marshalling and its Python form
def _both_forms():
    M, K, N, S, heads = 20, 64, 96, 10, 1
    g = torch.Generator(device="cuda").manual_seed(3)
    r = lambda *shape: torch.randn(shape, generator=g, device="cuda")
    X, b, x64, qkv = r(M, K), r(N), r(M, 64), r(2 * S, 192)
    Wq, S_w = q8.q8_quantize_weight(r(N, K))
    Xq = torch.randint(-127, 128, (M, K), generator=g, device="cuda", dtype=torch.int8)
    s, word = torch.full((1,), 20.0, device="cuda"), lambda: torch.zeros(1, dtype=torch.int32, device="cuda")
    ids = torch.randint(0, N, (7,), generator=g, device="cuda", dtype=torch.int32)
    state, peak = q8.new_calibrate_state(), X.abs().max().reshape(1).view(torch.int32)
    return [
        (q8.q8_linear, (X, Wq, S_w, s, b, 1)), (q8.q8_linear, (X, Wq, S_w)), (q8.q8_linear_q, (Xq, s, Wq, S_w, b)),
        (q8.q8_linear_requant, (X, Wq, S_w, s, b, 1, s)), (q8.q8_linear_q_requant, (Xq, s, Wq, S_w, b, 1, s)),
        (q8.q8_linear_dyn, (X, peak, Wq, S_w, b)), (q8.q8_embedding, (ids, Wq, S_w)), (q8.q8_add_layernorm, (x64, x64)),
        (q8.q8_add_layernorm_quant, (x64, x64, None, s)), (q8.q8_add_layernorm_absmax, (x64, word())),
        (q8.q8_attention, (qkv, 2, S, heads)), (q8.q8_attention_quant, (qkv, 2, S, heads, s)),
        (q8.q8_attention_absmax, (qkv, 2, S, heads, word())), (q8.q8_quantize_weight, (X,)),
        (q8.q8_fake_quantize, (X, s)), (q8.q8_ste_backward, (X,)), (q8.q8_calibrate, (X, 0.5, state)),
    ]


def test_native_and_python_forms_of_a_call_agree():
    """A given stream selects the Python form; without one the same arguments take the native form."""
    for fn, args in _both_forms():
        native, python = fn(*args), fn(*args, stream=torch.cuda.current_stream())
        for a, b in zip(*(v if isinstance(v, tuple) else (v,) for v in (native, python))):
            assert a is None and b is None or torch.equal(a, b), fn.__name__
        out = native[0] if isinstance(native, tuple) else native
        if out is not None and fn not in (q8.q8_quantize_weight,):
            name = {torch.int8: {"q8_linear_requant": "Yq", "q8_linear_q_requant": "Yq", "q8_add_layernorm_quant": "out_q",
                                 "q8_attention_quant": "ctx_q"},
                    torch.float32: {"q8_embedding": "out", "q8_fake_quantize": "Xhat", "q8_ste_backward": "grad_in"}}[out.dtype]
            key = name.get(fn.__name__) or ("Y" if "linear" in fn.__name__ else "ctx" if "attention" in fn.__name__ else "out")
            into = torch.empty_like(out)
            assert fn(*args, **{key: into}) is into and torch.equal(into, out), fn.__name__


def test_native_calls_refuse_what_the_python_form_refuses():
    for fn, args in _both_forms():
        for bad in (lambda t: t.cpu(), lambda t: t.double(), lambda t: torch.stack([t, t], -1)[..., 0]):
            broken = (bad(args[0]),) + args[1:]
            with pytest.raises(TypeError):
                fn(*broken, stream=torch.cuda.current_stream())
            with pytest.raises(TypeError):
                fn(*broken)
    X = torch.zeros((4, 32), device="cuda")
    Wq, S_w = q8.q8_quantize_weight(torch.ones((8, 48), device="cuda"))
    with pytest.raises(ValueError, match="X is"):
        q8.q8_linear(X, Wq, S_w)
    with pytest.raises(q8.Q8Error, match="q8_linear: q8_status 10"):
        q8.q8_linear(X, Wq[:, :32].contiguous(), S_w, act=7)
    with pytest.raises(q8.Q8Error, match="q8_status 7"):
        q8.q8_linear(X, Wq[:, :32].contiguous(), S_w, workspace=torch.empty(256, dtype=torch.uint8, device="cuda"))


def test_operands_that_do_not_fit_together_are_refused():
    """In both forms of a call, before anything is launched: shapes under which a kernel would read past an operand, or read it as
    something that it is not."""
    f32 = lambda *shape: torch.ones(shape, device="cuda")
    i8 = lambda *shape: torch.ones(shape, dtype=torch.int8, device="cuda")
    s, word, b = f32(1), torch.zeros(1, dtype=torch.int32, device="cuda"), f32(8)
    X, Xq, ids = f32(4, 32), i8(4, 32), torch.zeros(6, dtype=torch.int32, device="cuda")
    cases = []
    for W in (i8(8, 16), i8(8, 48)):
        cases += [(q8.q8_linear, (X, W, s)), (q8.q8_linear_generic, (X, W, s)), (q8.q8_linear_q, (Xq, s, W, s)),
                  (q8.q8_linear_requant, (X, W, s, s, b, 0, s)), (q8.q8_linear_q_requant, (Xq, s, W, s, b, 0, s)),
                  (q8.q8_linear_dyn, (X, word, W, s)), (q8.q8_linear_wseg, (X, W, s, 32)), (q8.q8_linear_q_wseg, (Xq, s, W, s, 32))]
    for qkv, B, S, heads in ((f32(20, 192), 3, 10, 1), (f32(20, 192), 2, 10, 2), (f32(20, 384), 2, 10, 1)):
        cases += [(q8.q8_attention, (qkv, B, S, heads)), (q8.q8_attention_quant, (qkv, B, S, heads, s)),
                  (q8.q8_attention_absmax, (qkv, B, S, heads, word))]
    for extra in ((f32(3, 32),), (None, f32(4, 31)), (None, None, f32(31)), (None, None, None, f32(31))):
        extra = tuple(extra) + (None,) * (4 - len(extra))
        cases += [(q8.q8_add_layernorm, (X,) + extra), (q8.q8_add_layernorm_absmax, (X, word) + extra),
                  (q8.q8_add_layernorm_quant, (X, extra[0], extra[1], s, None, None, extra[2], extra[3]))]
    for pos, typ in ((i8(9, 16), i8(2, 32)), (i8(9, 32), i8(2, 16)), (i8(9, 32), i8(0, 32))):
        cases.append((q8.q8_embed_layernorm, (ids, 3, i8(9, 32), s, pos, s, typ, s)))
    for fn, args in cases:
        for stream in (None, torch.cuda.current_stream()):
            with pytest.raises(ValueError):
                fn(*args, stream=stream)
    # larger ones than needed stay as they were
    x, r, qkv = torch.randn((4, 32), device="cuda"), torch.randn((5, 32), device="cuda"), torch.randn((21, 192), device="cuda")
    assert torch.equal(q8.q8_add_layernorm(x, r), q8.q8_add_layernorm(x, r[:4].contiguous()))
    assert torch.equal(q8.q8_attention_quant(qkv, 2, 10, 1, s), q8.q8_attention_quant(qkv[:20].contiguous(), 2, 10, 1, s))


# ------------------------------------------------------------------ K split over a cluster
@pytest.mark.parametrize("M,N,K", [(1, 32, 2048), (37, 90, 2064), (128, 768, 3072), (129, 500, 4096), (128, 1184, 2048),
                                   (300, 1000, 2176), (512, 1152, 2048), (16, 33, 16400)])
@pytest.mark.parametrize("act", [0, 1])
def test_split_k_layers_bit_exact(M, N, K, act):
    """Four CTAs per 128 x 32 tile (up to 37 tiles) and two per 128 x 64 tile: integers, fp32, and every output form."""
    X, W, b = synth.activation(M, K, 9300 + M), synth.weight(N, K, 9301), synth.bias(N, 9302)
    info = check_linear(X, W, b, act)
    assert info["gemm_kernel"] == 1 and (info["block_n"], info["grid"]) in (
        (32, 4 * ((M + 127) // 128) * ((N + 31) // 32)), (64, 2 * ((M + 127) // 128) * ((N + 63) // 64)))
    Wq, S_w = q8.q8_quantize_weight(dev(W))
    Xq, S_x = q8.q8_quantize_activation(dev(X))
    S_y = torch.full((1,), 25.0, device="cuda")
    peak = torch.zeros(1, dtype=torch.int32, device="cuda")
    top = torch.tensor([float(np.abs(X).max())], device="cuda").view(torch.int32)
    Y = q8.q8_linear_q(Xq, S_x, Wq, S_w, dev(b), act)
    Y2 = torch.empty_like(Y)
    both = q8.q8_linear_q_requant(Xq, S_x, Wq, S_w, dev(b), act, S_y, Y=Y2)
    only = q8.q8_linear_q_requant(Xq, S_x, Wq, S_w, dev(b), act, S_y)
    dyn = q8.q8_linear_dyn(dev(X), top, Wq, S_w, dev(b), act, y_absmax=peak)
    assert torch.equal(Y2, Y) and torch.equal(both, only) and torch.equal(dyn, Y)
    assert np.array_equal(only.cpu().numpy(), o.quantize(Y.cpu().numpy(), np.float32(25.0)))
    assert peak.view(torch.float32).item() == Y.abs().max().item()


@pytest.mark.parametrize("M,N,K,block_n,ctas", [(1, 32, 2048, 32, 4), (300, 1000, 2176, 64, 2)])
def test_split_k_reports_the_ctas_of_a_tile(M, N, K, block_n, ctas):
    Xq, Wq = (torch.ones((n, K), dtype=torch.int8, device="cuda") for n in (M, N))
    one = torch.ones(1, device="cuda")
    q8.q8_linear_q(Xq, one, Wq, one)
    info = q8.q8_last_launch_info()
    assert (info["block_n"], info["ctas"]) == (block_n, ctas)


@pytest.mark.parametrize("M,N,K", [(1, 1, 16), (129, 193, 144), (300, 500, 272)])
def test_192_wide_tiles_can_be_asked_for(M, N, K):
    try:
        q8.q8_tune_gemm_tile(192, 1)
        info = check_linear(synth.activation(M, K, 9450), synth.weight(N, K, 9451), synth.bias(N, 9452), 1)
    finally:
        q8.q8_tune_gemm_tile(0, 0)
    assert (info["gemm_kernel"], info["block_n"], info["ctas"]) == (1, 192, 1)


@pytest.mark.parametrize("M,N,K", [(4096, 768, 256), (4000, 700, 144), (2900, 1024, 272)])
def test_192_wide_tiles_bit_exact(M, N, K):
    X, W, b = synth.activation(M, K, 9400 + N), synth.weight(N, K, 9401), synth.bias(N, 9402)
    info = check_linear(X, W, b, 1)
    assert (info["gemm_kernel"], info["block_n"], info["ctas"]) == (1, 192, 1)
    Wq, S_w = q8.q8_quantize_weight(dev(W))
    Xq, S_x = q8.q8_quantize_activation(dev(X))
    S_y = torch.full((1,), 25.0, device="cuda")
    Y = q8.q8_linear_q(Xq, S_x, Wq, S_w, dev(b), 1)
    only = q8.q8_linear_q_requant(Xq, S_x, Wq, S_w, dev(b), 1, S_y)
    assert np.array_equal(only.cpu().numpy(), o.quantize(Y.cpu().numpy(), np.float32(25.0)))


@pytest.mark.parametrize("block_n", [128, 192, 256])
@pytest.mark.parametrize("M,N,K", [(1, 32, 16), (130, 260, 272), (511, 1000, 1040), (40000, 384, 48)])
def test_one_cta_tiles_in_every_output_mode(block_n, M, N, K):
    """Tiles of one CTA have 12 or 16 epilogue warps with GELU and 8 without: ragged rows and columns, several tiles to a CTA, fp32, Int8,
    both, and with the running maximum."""
    X, W, b = synth.activation(M, K, 9460), synth.weight(N, K, 9461), synth.bias(N, 9462)
    S_y = torch.full((1,), 25.0, device="cuda")
    try:
        q8.q8_tune_gemm_tile(block_n, 1)
        for act in (0, 1):
            info = check_linear(X, W, b, act)
            assert (info["gemm_kernel"], info["block_n"], info["ctas"]) == (1, block_n, 1)
            Wq, S_w = q8.q8_quantize_weight(dev(W))
            Xd = dev(X)
            Xq, S_x = q8.q8_quantize_activation(Xd)
            Y = q8.q8_linear_q(Xq, S_x, Wq, S_w, dev(b), act)
            want = o.quantize(Y.cpu().numpy(), np.float32(25.0))
            assert np.array_equal(q8.q8_linear_q_requant(Xq, S_x, Wq, S_w, dev(b), act, S_y).cpu().numpy(), want)
            Y2 = torch.empty_like(Y)
            assert np.array_equal(q8.q8_linear_q_requant(Xq, S_x, Wq, S_w, dev(b), act, S_y, Y=Y2).cpu().numpy(), want)
            word = torch.zeros(1, dtype=torch.int32, device="cuda")
            Y3 = q8.q8_linear_dyn(Xd, Xd.abs().max().view(torch.int32).reshape(1), Wq, S_w, dev(b), act, y_absmax=word)
            assert torch.equal(Y2, Y) and torch.equal(Y3, Y) and word.view(torch.float32).item() == Y.abs().max().item()
    finally:
        q8.q8_tune_gemm_tile(0, 0)


@pytest.mark.parametrize("block_n,ctas,warps", [(64, 1, 0), (128, 1, 0), (192, 1, 0), (256, 1, 0), (256, 2, 8), (256, 2, 16)])
def test_gelu_to_int8_at_any_scale(block_n, ctas, warps):
    """Eq. 1 on GELU's output at scales on both sides of the line from which its lowest value (-0.17) needs the lower clamp, and at scales
    that are not positive (-128 never appears), infinite or NaN: the integers of the fp32 output, whatever the tile."""
    M, N, K = 515, 1040, 272
    Wq, S_w = q8.q8_quantize_weight(dev(synth.weight(N, K, 9480)))
    b = dev(synth.bias(N, 9481))
    Xq, S_x = q8.q8_quantize_activation(dev(synth.activation(M, K, 9482)))
    try:
        q8.q8_tune_gemm_tile(block_n, ctas)
        q8.q8_tune_gemm_epilogue_warps(warps)
        for scale_x in (S_x, torch.zeros_like(S_x)):  # (a zero product scale: every value is NaN or infinite)
            Y = q8.q8_linear_q(Xq, scale_x, Wq, S_w, b, 1)
            if scale_x is S_x:
                assert Y.min().item() < -0.1699 and Y.max().item() > 0.3  # (-0.17 x 760 is beyond -127.5, 0.3 x 1000 beyond 127)
            for S in (25.0, 699.0, 700.0, 701.0, 760.0, 5000.0, 0.0, -1.0, -1000.0, np.inf, -np.inf, np.nan):
                got = q8.q8_linear_q_requant(Xq, scale_x, Wq, S_w, b, 1, dev(np.array([S], np.float32)))
                assert np.array_equal(got.cpu().numpy(), o.quantize(Y.cpu().numpy(), np.float32(S))), S
    finally:
        q8.q8_tune_gemm_epilogue_warps(0)
        q8.q8_tune_gemm_tile(0, 0)


@pytest.mark.parametrize("block_n", [64, 128, 192, 256])
@pytest.mark.parametrize("M,N,K", [(1, 33, 16), (127, 63, 64), (161, 1001, 272), (20000, 257, 48)])
def test_one_cta_tiles_of_widths_that_tma_does_not_store(block_n, M, N, K):
    """Rows that are no multiple of 16 bytes leave in a loop over the block's rows: fp32 alone, with the integers, with the maximum."""
    X, W, b = synth.activation(M, K, 9470), synth.weight(N, K, 9471), synth.bias(N, 9472)
    S_y = torch.full((1,), 25.0, device="cuda")
    try:
        q8.q8_tune_gemm_tile(block_n, 1)
        for act in (0, 1):
            info = check_linear(X, W, b, act)
            assert (info["gemm_kernel"], info["block_n"], info["ctas"]) == (1, block_n, 1)
            Wq, S_w = q8.q8_quantize_weight(dev(W))
            Xd = dev(X)
            Xq, S_x = q8.q8_quantize_activation(Xd)
            Y = q8.q8_linear_q(Xq, S_x, Wq, S_w, dev(b), act)
            Y2 = torch.full((M * N + 64,), 7.0, device="cuda")
            Yq = q8.q8_linear_q_requant(Xq, S_x, Wq, S_w, dev(b), act, S_y, Y=Y2[: M * N].view(M, N))
            assert np.array_equal(Yq.cpu().numpy(), o.quantize(Y.cpu().numpy(), np.float32(25.0)))
            assert torch.equal(Y2[: M * N].view(M, N), Y) and bool((Y2[M * N :] == 7.0).all())
            word = torch.zeros(1, dtype=torch.int32, device="cuda")
            Y3 = q8.q8_linear_dyn(Xd, Xd.abs().max().view(torch.int32).reshape(1), Wq, S_w, dev(b), act, y_absmax=word)
            assert torch.equal(Y3, Y) and word.view(torch.float32).item() == Y.abs().max().item()
    finally:
        q8.q8_tune_gemm_tile(0, 0)


@pytest.mark.parametrize("N,off,K,ctas", [(1024, 0, 64, 2), (1023, 0, 64, 1), (1022, 0, 64, 1), (1024, 1, 64, 1), (1024, 2, 64, 1),
                                          (1022, 0, 2064, 2), (1022, 1, 2064, 1), (1023, 0, 2064, 1)])
def test_layers_whose_output_pairs_cannot_store_take_one_cta_tiles(N, off, K, ctas):
    """A grid full of pairs: fp32 rows that neither TMA nor the paired 8-byte stores take (K > 2048 for these) leave through one-CTA tiles;
    the Int8 output does not ask."""
    M = 9500
    Xq, S_x = q8.q8_quantize_activation(dev(synth.activation(M, K, 9490)))
    Wq, S_w = q8.q8_quantize_weight(dev(synth.weight(N, K, 9491)))
    b = dev(synth.bias(N, 9492))
    room = torch.full((M * N + 64,), 7.0, device="cuda")
    Y = room[off:M * N + off].view(M, N)
    q8.q8_linear_q(Xq, S_x, Wq, S_w, b, 0, Y=Y)
    assert q8.q8_last_launch_info()["ctas"] == ctas
    assert bool((room[:off] == 7.0).all()) and bool((room[M * N + off:] == 7.0).all())
    q8.q8_linear_q_requant(Xq, S_x, Wq, S_w, b, 0, torch.full_like(S_x, 25.0))
    assert q8.q8_last_launch_info()["ctas"] == 2
    acc = Xq.double() @ Wq.double().T + torch.round(b * (S_x * S_w)).double()  # exact: below 2^53
    inv = torch.ones_like(S_x) / (S_x * S_w)
    assert torch.equal(Y, acc.float() * inv)


# ------------------------------------------------------------------ the streaming passes at the ends of their runs
@pytest.mark.parametrize("n", [1, 5, 511, 2047, 2048, 2049, 4 * 2048 - 3, 16 * 148 * 512 + 7, 148 * 8 * 2048, 148 * 8 * 2048 + 1,
                               148 * 8 * 4096 + 5, 2 * 148 * 8 * 4096 + 12343])
@pytest.mark.parametrize("peak_at", [0, -1])
def test_streaming_passes_at_the_ends_of_their_runs(n, peak_at):
    """Quantise, abs-max with the Eq. 4 update, fake quantise and the straight-through copy: a CTA's run is 4 x 128 float4 (4 x 256
    of the abs-max, whose 8 CTAs per SM take a second and a third run on the two largest), the last run is ragged and up to three values
    are left over."""
    x = synth.normal((n,), 1.0, 9100 + n % 1000)
    x[peak_at] = 7.5  # the largest value is the first or the last one
    xd, S = dev(x), dev(np.array([12.7], np.float32))
    assert np.array_equal(q8.q8_quantize_activation(xd, S)[0].cpu().numpy(), o.quantize(x, np.float32(12.7)))
    state = q8.new_calibrate_state()
    q8.q8_calibrate(xd, 0.5, state)
    assert state.view(torch.float32)[0].item() == 7.5
    assert torch.equal(q8.q8_ste_backward(xd), xd)
    want = o.quantize(x, np.float32(12.7)).astype(np.float32) / np.float32(12.7)
    assert np.array_equal(q8.q8_fake_quantize(xd, S).cpu().numpy(), want)
    inplace = xd.clone()
    assert np.array_equal(q8.q8_fake_quantize(inplace, S, inplace).cpu().numpy(), want)


@pytest.mark.parametrize("S", [2.0 ** -125, 1e-25, 2.0 ** -60, 1.0000001, 12.7, 1e9 / 3, 2.0 ** 60, 1e25, 3.4e38])
def test_fake_quantise_quotient_is_rounded_to_nearest(S):
    """Every integer of -127..127 over S, at the ends of the range where the quotient comes from a reciprocal and beyond."""
    S = np.float32(S)
    q = np.arange(-127, 128, dtype=np.float32)
    with np.errstate(over="ignore"):
        x = (q / S).astype(np.float32)
        want = o.quantize(x, S).astype(np.float32) / S
    got = q8.q8_fake_quantize(dev(x), dev(np.array([S], np.float32))).cpu().numpy()
    assert np.array_equal(got, want)


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (65, 66, 300), (100, 130, 301), (64, 1201, 72), (1000, 1200, 300), (2050, 1930, 100),
                                   (2049, 1931, 104), (3000, 700, 77), (40000, 4, 100)])
def test_generic_gemm_with_and_without_the_other_outputs(M, N, K):
    """A call that wants the fp32 output only has its own form of the generic kernel: same bits as the one that also copies the Int32
    accumulator, for pieces of 8, 4 and 1 bytes, both tiles, ragged edges, odd widths and an output that takes no pairs."""
    X, W, b = dev(synth.activation(M, K, 9700)), dev(synth.weight(N, K, 9701)), dev(synth.bias(N, 9702))
    Wq, S_w = q8.q8_quantize_weight(W)
    ws, acc = q8.new_workspace(M, N, K), torch.empty((M, N), dtype=torch.int32, device="cuda")
    for act in (0, 1):
        for bias in (b, None):
            want = q8.q8_linear_generic(X, Wq, S_w, None, bias, act, workspace=ws, dbg_acc=acc)
            assert torch.equal(q8.q8_linear_generic(X, Wq, S_w, None, bias, act, workspace=ws), want)
            room = torch.full((M * N + 3,), 5.0, device="cuda")
            q8.q8_linear_generic(X, Wq, S_w, None, bias, act, Y=room[1:1 + M * N].view(M, N), workspace=ws)
            assert torch.equal(room[1:1 + M * N].view(M, N), want) and room[0] == 5.0 and (room[1 + M * N:] == 5.0).all()
