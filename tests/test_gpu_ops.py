"""GPU parity: every lpdt entry point against the CPU oracle on the same seeded
inputs, through the C ABI.  Integer results bit-exact; fp32 results within
1e-5 relative / 1e-6 absolute."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_09389_b200 import api, workloads as wlmod

pytestmark = pytest.mark.gpu

RTOL, ATOL = 1e-5, 1e-6


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def close(got, want, rtol=RTOL, atol=ATOL):
    got = got.cpu().numpy() if isinstance(got, torch.Tensor) else got
    want = np.asarray(want, dtype=np.float64)
    err = np.abs(got.astype(np.float64) - want)
    ok = err <= atol + rtol * np.abs(want)
    assert ok.all(), f"{(~ok).sum()} of {ok.size} outside tolerance, worst {err.max():.3e}"


def ws_bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


# ------------------------------------------------------------------ quantizer
@pytest.mark.parametrize("nodes,n", [(1, 1), (3, 7), (4, 4096), (2, 100003), (16, 98304), (1, 1 << 22)])
@pytest.mark.parametrize("rounding", [0, 1])
def test_quantize_sym(nodes, n, rounding):
    rng = np.random.default_rng(n + rounding)
    x = (rng.standard_normal((nodes, n)) * rng.uniform(0.01, 100, (nodes, 1))).astype(np.float32)
    q_ref, s_ref = oracle.quantize_sym_s8(x, rounding, seed=(9 << 32) | 77, ctr_offset=3)
    xd = dev(x)
    q = torch.empty(nodes, n, dtype=torch.int8, device="cuda")
    s = torch.empty(nodes, dtype=torch.float32, device="cuda")
    ws = ws_bytes(api.lpdt_quantize_workspace_size(nodes))
    api.lpdt_quantize(xd, nodes, n, n, q, s, ws, mode=0, rounding=rounding, seed=(9 << 32) | 77, ctr_offset=3)
    assert np.array_equal(s.cpu().numpy(), s_ref)
    assert np.array_equal(q.cpu().numpy(), q_ref)
    y = torch.empty(nodes, n, dtype=torch.float32, device="cuda")
    api.lpdt_dequantize(q, nodes, n, s, y)
    assert np.array_equal(y.cpu().numpy(), oracle.dequantize(q_ref, s_ref))


@pytest.mark.parametrize("n", [4096, 4099])          # words of four codes, single ones
def test_stochastic_rounding_at_its_edges(n):
    """Integers, values just below and above them, denormals: the oracle's codes exactly; values beyond a caller's range,
    infinities and NaN: the clamp's codes."""
    rng = np.random.default_rng(n)
    x = rng.uniform(-127, 127, (2, n)).astype(np.float32)
    x[:, 0] = 127.0
    x[:, 1:256] = np.arange(-127, 128)
    x[:, 256:511] = np.nextafter(x[:, 1:256], np.float32(-200))
    x[:, 511:766] = np.nextafter(x[:, 1:256], np.float32(200))
    x[:, 766:1024] = np.clip(x[:, 766:1024], -126, 126) * np.float32(1e-30)
    x[:, 1024:1280] = np.exp2(rng.uniform(-149, -20, (2, 256))).astype(np.float32) * rng.choice([-1, 1], (2, 256))
    x = np.clip(x, -127, 127).astype(np.float32)
    q_ref, _ = oracle.quantize_sym_s8(x, 1, seed=5, ctr_offset=1)
    amax = dev(np.abs(x).max(1).astype(np.float32))
    beyond = np.array([3e38, -3e38, np.inf, -np.inf, np.nan, 4194303.75, -4194304.5, 8388609, -1.3e7, 200.5, -128.25], np.float32)
    clamped = np.array([127, -127, 127, -127, -127, 127, -127, 127, -127, 127, -127], np.int8)
    x[:, 2000:2000 + len(beyond)] = beyond
    q_ref[:, 2000:2000 + len(beyond)] = clamped
    q = torch.empty(2, n, dtype=torch.int8, device="cuda")
    s = torch.empty(2, dtype=torch.float32, device="cuda")
    api.lpdt_quantize_with_range(dev(x), 2, n, n, amax, q, s, rounding=1, seed=5, ctr_offset=1)
    assert np.array_equal(q.cpu().numpy(), q_ref)


def test_quantize_strided_rows_zero_tensor_and_ties():
    # rows inside a wider flat vector (odd stride -> scalar path), an all-zero node, exact ties
    rng = np.random.default_rng(0)
    nodes, n, stride = 3, 432, 1001
    flat = rng.standard_normal((nodes, stride)).astype(np.float32)
    flat[1, 5:5 + n] = 0.0
    flat[2, 5:5 + n] = np.round(flat[2, 5:5 + n] * 4) / 8      # many .5 ties once scaled
    flat[2, 5] = 127.0 / 2
    q_ref, s_ref = oracle.quantize_sym_s8(flat[:, 5:5 + n])
    fd = dev(flat)
    q = torch.empty(nodes, n, dtype=torch.int8, device="cuda")
    s = torch.empty(nodes, dtype=torch.float32, device="cuda")
    api.lpdt_quantize(fd[:, 5:], nodes, n, stride, q, s, ws_bytes(256))
    assert np.array_equal(q.cpu().numpy(), q_ref) and np.array_equal(s.cpu().numpy(), s_ref)
    assert s_ref[1] == 1.0 and not q_ref[1].any()


@pytest.mark.parametrize("nodes,n", [(2, 1001), (3, 65536)])
def test_quantize_affine(nodes, n):
    rng = np.random.default_rng(n)
    x = rng.uniform(-1, 3, (nodes, n)).astype(np.float32)
    x[-1] = np.abs(x[-1]) + 0.5                                  # one-sided node
    q_ref, s_ref, z_ref = oracle.quantize_affine_u8(x)
    q = torch.empty(nodes, n, dtype=torch.int8, device="cuda")
    s = torch.empty(nodes, dtype=torch.float32, device="cuda")
    zp = torch.empty(nodes, dtype=torch.int32, device="cuda")
    api.lpdt_quantize(dev(x), nodes, n, n, q, s, ws_bytes(256), mode=1, zero_point=zp)
    assert np.array_equal(q.cpu().numpy().view(np.uint8), q_ref)
    assert np.array_equal(s.cpu().numpy(), s_ref) and np.array_equal(zp.cpu().numpy(), z_ref)
    y = torch.empty(nodes, n, dtype=torch.float32, device="cuda")
    api.lpdt_dequantize(q, nodes, n, s, y, zero_point=zp)
    assert np.array_equal(y.cpu().numpy(), oracle.dequantize(q_ref, s_ref, z_ref))


def test_quantize_batch_matches_per_tensor_calls():
    rng = np.random.default_rng(11)
    nodes, d = 5, 20011
    params = (rng.standard_normal((nodes, d)) * rng.uniform(0.01, 3, (nodes, 1))).astype(np.float32)
    src = [0, 432, 433, 5000, 15003]; size = [432, 1, 2304, 9216, 5008]
    params[2, 432] = 0.0                                   # an all-zero single-element tensor on one node
    dst, off = [], 0
    for n in size:
        dst.append(off); off += (nodes * n + 255) // 256 * 256
    q = torch.full((off,), 99, dtype=torch.int8, device="cuda")
    sc = torch.zeros(len(size), nodes, device="cuda")
    ws = ws_bytes(api.lpdt_quantize_batch_workspace_size(nodes, len(size)))
    api.lpdt_quantize_batch(dev(params), nodes, d, src, size, dst, q, sc, ws)
    qh, sh = q.cpu().numpy(), sc.cpu().numpy()
    for t, (o, n, do) in enumerate(zip(src, size, dst)):
        q_ref, s_ref = oracle.quantize_sym_s8(params[:, o:o + n])
        assert np.array_equal(sh[t], s_ref)
        assert np.array_equal(qh[do:do + nodes * n].reshape(nodes, n), q_ref)
    assert sh[1, 2] == 1.0


@pytest.mark.parametrize("words", [1, 2, 3, 4, 5, 1023, 1024, 16383, 16384, 16385])
@pytest.mark.parametrize("first", [0, 1, 2, 3])
def test_fill_zero_at_every_alignment(words, first):
    t = torch.full((words + 8,), 7, dtype=torch.int32, device="cuda")
    api.lpdt_fill_zero(t[first:first + words])
    assert not t[first:first + words].any() and (t[:first] == 7).all() and (t[first + words:] == 7).all()
    b = t.view(torch.uint8)                       # not whole words
    b.fill_(3)
    api.lpdt_fill_zero(b[first:first + 4 * words - 1])
    assert not b[first:first + 4 * words - 1].any() and (b[:first] == 3).all() and (b[first + 4 * words - 1:] == 3).all()


def test_fill_zero_leaves_other_memory_to_the_runtime():
    """A kernel fills memory of the device; what lies elsewhere (here pinned host memory) goes to the runtime's fill, which
    checks it."""
    stream = torch.cuda.current_stream().cuda_stream
    for t, kernels in ((torch.ones(64, device="cuda"), 1), (torch.ones(64).pin_memory(), 0)):
        before = api.lpdt_launch_count()
        assert api.lib().lpdt_fill_zero(t.data_ptr(), 256, stream) == 0
        assert api.lpdt_launch_count() - before == kernels
        torch.cuda.synchronize()
        assert not t.any()


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 8193])
@pytest.mark.parametrize("mode", [0, 1])
def test_quantize_with_a_workspace_that_holds_anything(n, mode):
    """Short tensors store their range, longer ones gather it in words that the call clears."""
    rng = np.random.default_rng(n)
    x = rng.standard_normal((3, n)).astype(np.float32)
    q = torch.empty(3, n, dtype=torch.uint8 if mode else torch.int8, device="cuda")
    s, z = torch.empty(3, device="cuda"), torch.zeros(3, dtype=torch.int32, device="cuda")
    ws = ws_bytes(api.lpdt_quantize_workspace_size(3)).fill_(255)
    api.lpdt_quantize(dev(x), 3, n, n, q, s, ws, mode=mode, zero_point=z if mode else None)
    ref = oracle.quantize_affine_u8(x) if mode else oracle.quantize_sym_s8(x)
    assert np.array_equal(q.cpu().numpy(), ref[0]) and np.array_equal(s.cpu().numpy(), ref[1])
    if mode:
        assert np.array_equal(z.cpu().numpy(), ref[2])
    else:
        q2, s2 = torch.empty_like(q), torch.empty(1, 3, device="cuda")
        ws = ws_bytes(api.lpdt_quantize_batch_workspace_size(3, 1)).fill_(255)
        api.lpdt_quantize_batch(dev(x), 3, n, [0], [n], [0], q2, s2, ws)
        assert torch.equal(q2, q) and torch.equal(s2[0], s)


def test_quantize_argument_errors():
    x = torch.zeros(8, device="cuda")
    q = torch.zeros(8, dtype=torch.int8, device="cuda")
    s = torch.zeros(1, device="cuda")
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_quantize(x, 1, 8, 8, q, s, None)
    assert e.value.code == 3
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_quantize(None, 1, 8, 8, q, s, ws_bytes(256))
    assert e.value.code == 1
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_quantize(x, 1, 8, 8, q, s, ws_bytes(256), mode=1)     # affine without zero_point
    assert e.value.code == 1
    api.lpdt_quantize(x, 0, 8, 8, q, s, None)                          # empty: no-op


# ------------------------------------------------------------------ contractions
CONV_CASES = [
    # nodes, B, H, W, Cin, Cout, R, S, stride, pad
    (4, 8, 16, 16, 16, 16, 3, 3, 1, 1),      # the single-layer workload
    (2, 3, 32, 32, 3, 16, 3, 3, 1, 1),       # first layer of the networks
    (2, 2, 16, 16, 16, 32, 3, 3, 2, 1),      # strided stage transition
    (1, 2, 9, 7, 5, 6, 3, 3, 1, 1),          # ragged everything
    (2, 4, 8, 8, 64, 64, 3, 3, 1, 1),
    (1, 1, 12, 12, 32, 48, 1, 1, 1, 0),      # 1x1
    (3, 32, 1, 1, 64, 10, 1, 1, 1, 0),       # classifier
    (1, 5, 4, 4, 8, 8, 3, 3, 1, 0),          # no padding
    (1, 2, 40, 24, 128, 64, 3, 3, 1, 1),
    (2, 3, 32, 32, 32, 64, 3, 3, 2, 1),      # strided, tensor-core path
    (1, 2, 15, 13, 16, 16, 3, 3, 2, 1),      # strided with odd image sizes
    (1, 2, 16, 16, 32, 32, 1, 1, 2, 0),      # strided 1x1: three of four input parities get no tap
    (1, 1, 56, 56, 64, 64, 3, 3, 1, 1),      # image width that no power-of-two tile divides
    (1, 3, 7, 7, 16, 32, 5, 5, 1, 2),        # 5x5 filter
    (2, 40, 1, 1, 256, 128, 1, 1, 1, 0),     # linear layer on the tensor-core path
    (1, 130, 1, 1, 512, 272, 1, 1, 1, 0),    # linear: ragged row tile, two N tiles (272 = 16*17)
    (1, 1, 4, 4, 512, 512, 3, 3, 1, 1),      # wide channels on a tiny map
    (3, 5, 32, 32, 16, 16, 3, 3, 1, 1),      # 16-channel halo-tile path, several nodes per CTA range
    (2, 3, 19, 13, 16, 48, 3, 3, 1, 1),      # halo path: ragged image, 16 -> 48 channels
    (2, 2, 20, 20, 48, 16, 3, 3, 1, 1),      # halo path on the backward-data side (Cout = 16)
    (1, 2, 17, 9, 16, 16, 5, 4, 1, 2),       # halo path: 5x4 filter (even tap count), asymmetric padding effect
    (1, 2, 12, 12, 16, 32, 1, 1, 1, 0),      # halo path with a single tap
    (2, 2, 10, 10, 16, 16, 3, 3, 1, 0),      # halo path without padding
    (2, 3, 16, 16, 32, 32, 3, 3, 1, 1),      # halo path with two 16-channel chunks
    (2, 5, 8, 8, 64, 64, 3, 3, 1, 1),        # halo path: 8x8 maps (half of each tile is outside the image)
    (1, 2, 13, 11, 96, 32, 3, 3, 1, 1),      # halo path: 6 chunks forward, 2 chunks backward
    (1, 2, 9, 20, 128, 128, 3, 3, 1, 1),     # halo path at its channel limit
]


def _conv_inputs(case, seed=0):
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    rng = np.random.default_rng(seed)
    A = wlmod.random_s8(rng, (nodes, B, H, W, Cin))
    Wq = wlmod.random_s8(rng, (nodes, Cout, R, S, Cin))
    Ho, Wo = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - S) // stride + 1
    E = wlmod.random_s8(rng, (nodes, B, Ho, Wo, Cout))
    s1 = rng.uniform(0.001, 0.1, nodes).astype(np.float32)
    s2 = rng.uniform(0.001, 0.1, nodes).astype(np.float32)
    return A, Wq, E, s1, s2


@pytest.mark.parametrize("case", CONV_CASES)
def test_qconv_fwd_affine(case):
    """Zero-point operands (Section 3's scheme) on every forward shape: int32 sums bit-exact, fp32 as dequant_acc."""
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    rng = np.random.default_rng(77)
    A = rng.integers(0, 256, (nodes, B, H, W, Cin), dtype=np.uint8)
    Wq = rng.integers(0, 256, (nodes, Cout, R, S, Cin), dtype=np.uint8)
    zA = rng.integers(0, 256, nodes).astype(np.int32)
    zW = rng.integers(0, 256, nodes).astype(np.int32)
    zA[0], zW[0] = 255, 0                                   # extreme zero points on one node
    s1 = rng.uniform(0.001, 0.1, nodes).astype(np.float32)
    s2 = rng.uniform(0.001, 0.1, nodes).astype(np.float32)
    acc_ref, ovf = oracle.qconv_fwd_affine(A, zA, Wq, zW, stride, pad)
    assert ovf == 0
    desc = api.conv_desc(*case)
    ws = ws_bytes(api.lpdt_qconv_fwd_affine_workspace_size(desc))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    bias = rng.standard_normal((nodes, Cout)).astype(np.float32)
    Y = torch.empty(acc_ref.shape, dtype=torch.float32, device="cuda")
    Yacc = torch.empty(acc_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_fwd_affine(desc, dev(A), dev(s1), dev(zA), dev(Wq), dev(s2), dev(zW), Y=Y, Yacc=Yacc,
                              bias=dev(bias), bias_node_stride=Cout, ws=ws, dev_status=status)
    assert int(status.item()) == 0
    assert np.array_equal(Yacc.cpu().numpy(), acc_ref)
    assert np.array_equal(Y.cpu().numpy(), oracle.dequant_acc(acc_ref, s1, s2, bias))


@pytest.mark.parametrize("case", CONV_CASES)
def test_qconv_bwd_affine(case):
    """Both backward products on zero-point operands, every shape: int32 sums bit-exact, fp32 as dequant_acc;
    the weight gradient also into a strided destination."""
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    rng = np.random.default_rng(78)
    Ho, Wo = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - S) // stride + 1
    A = rng.integers(0, 256, (nodes, B, H, W, Cin), dtype=np.uint8)
    Wq = rng.integers(0, 256, (nodes, Cout, R, S, Cin), dtype=np.uint8)
    E = rng.integers(0, 256, (nodes, B, Ho, Wo, Cout), dtype=np.uint8)
    zA, zW, zE = (rng.integers(0, 256, nodes).astype(np.int32) for _ in range(3))
    zE[0], zW[0], zA[0] = 255, 0, 255                       # extreme zero points on one node
    sA, sW, sE = (rng.uniform(0.001, 0.1, nodes).astype(np.float32) for _ in range(3))
    dA_ref, o1 = oracle.qconv_bwd_data_affine(E, zE, Wq, zW, H, W, stride, pad)
    dW_ref, o2 = oracle.qconv_bwd_weight_affine(E, zE, A, zA, R, S, stride, pad)
    assert o1 == 0 and o2 == 0
    desc = api.conv_desc(*case)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Ed, Wd, Ad = dev(E), dev(Wq), dev(A)
    dA = torch.empty(dA_ref.shape, dtype=torch.float32, device="cuda")
    dAacc = torch.empty(dA_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_bwd_data_affine(desc, Ed, dev(sE), dev(zE), Wd, dev(sW), dev(zW), dA=dA, dAacc=dAacc,
                                   ws=ws_bytes(api.lpdt_qconv_bwd_data_affine_workspace_size(desc)), dev_status=status)
    assert np.array_equal(dAacc.cpu().numpy(), dA_ref)
    assert np.array_equal(dA.cpu().numpy(), oracle.dequant_acc(dA_ref, sE, sW))
    wn = Cout * R * S * Cin
    stride_w = wn + 12
    dW = torch.zeros(nodes, stride_w, dtype=torch.float32, device="cuda")
    dWacc = torch.empty(dW_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_bwd_weight_affine(desc, Ed, dev(sE), dev(zE), Ad, dev(sA), dev(zA), dW=dW, dw_node_stride=stride_w,
                                     dWacc=dWacc, ws=ws_bytes(api.lpdt_qconv_bwd_weight_affine_workspace_size(desc)),
                                     dev_status=status)
    assert int(status.item()) == 0
    assert np.array_equal(dWacc.cpu().numpy(), dW_ref)
    assert np.array_equal(dW[:, :wn].cpu().numpy(), oracle.dequant_acc(dW_ref, sE, sA).reshape(nodes, wn))
    assert not dW[:, wn:].any()


@pytest.mark.parametrize("nodes,Cin,Cout,R,stride", [(1, 1, 3, 3, 1), (2, 4, 4, 1, 1), (2, 12, 5, 3, 2), (3, 64, 16, 3, 1),
                                                     (2, 132, 8, 3, 1), (2, 160, 32, 1, 2)])
def test_qconv_bwd_weight_affine_destinations(nodes, Cin, Cout, R, stride):
    """Weight gradients of zero-point operands at every alignment of their destination (four channels a store or one)
    and node stride: int32 sums exact, fp32 as dequant_acc, nothing written beside them."""
    B, H, pad = 3, 9, R // 2
    rng = np.random.default_rng(79)
    Ho = (H + 2 * pad - R) // stride + 1
    A = rng.integers(0, 256, (nodes, B, H, H, Cin), dtype=np.uint8)
    E = rng.integers(0, 256, (nodes, B, Ho, Ho, Cout), dtype=np.uint8)
    zA, zE = (rng.integers(0, 256, nodes).astype(np.int32) for _ in range(2))
    sA, sE = (rng.uniform(0.001, 0.1, nodes).astype(np.float32) for _ in range(2))
    ref, ovf = oracle.qconv_bwd_weight_affine(E, zE, A, zA, R, R, stride, pad)
    assert ovf == 0
    wn = Cout * R * R * Cin
    want = oracle.dequant_acc(ref, sE, sA).reshape(nodes, wn)
    desc = api.conv_desc(nodes, B, H, H, Cin, Cout, R, R, stride, pad)
    ws = ws_bytes(api.lpdt_qconv_bwd_weight_affine_workspace_size(desc))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for offset, more in ((0, 0), (0, 1), (1, 4), (4, 4), (2, 2)):
        step = wn + more
        flat = torch.full((offset + nodes * step + 8,), 7.0, device="cuda")
        accs = torch.full((offset + nodes * wn + 8,), 7, dtype=torch.int32, device="cuda")
        api.lpdt_qconv_bwd_weight_affine(desc, dev(E), dev(sE), dev(zE), dev(A), dev(sA), dev(zA), dW=flat[offset:],
                                         dw_node_stride=step, dWacc=accs[offset:], ws=ws, dev_status=status)
        got = flat[offset:offset + nodes * step].view(nodes, step)
        assert np.array_equal(got[:, :wn].cpu().numpy(), want)
        assert np.array_equal(accs[offset:offset + nodes * wn].cpu().numpy(), ref.reshape(-1))
        assert (got[:, wn:] == 7).all() and (flat[:offset] == 7).all() and (flat[offset + nodes * step:] == 7).all()
        assert (accs[:offset] == 7).all() and (accs[offset + nodes * wn:] == 7).all()
    assert int(status.item()) == 0


# channel counts that no 16-byte row holds, or that end inside a box of the tensor-core kernels.  (cc): forward products so
# small that they run on the CUDA cores; backward-weight takes the tensor cores all the same
RAGGED_CASES = [
    (2, 130, 1, 1, 200, 270, 1, 1, 1, 0),    # linear: 200 = 128 + 72 inputs, results in rows of 270 (no 16-byte rows)
    (1, 300, 1, 1, 1001, 17, 1, 1, 1, 0),    # odd on both sides, three row tiles
    (1, 5, 9, 11, 7, 21, 3, 3, 1, 1),        # cc
    (2, 3, 13, 10, 33, 50, 3, 3, 2, 1),      # strided, both ragged
    (2, 2, 16, 16, 3, 24, 3, 3, 2, 1),       # strided first layer (cc)
    (1, 2, 8, 8, 130, 36, 3, 3, 1, 1),
    (1, 2, 6, 6, 16, 15, 3, 3, 1, 1),        # whole input rows, one result short of a row (cc)
    (1, 3, 5, 5, 20, 16, 5, 5, 1, 2),
    (1, 2, 12, 12, 144, 80, 3, 3, 1, 1),     # multiples of 16 whose last box is part zeros
    (2, 3, 7, 7, 272, 400, 1, 1, 1, 0),      # several N tiles, the last one part empty
    (1, 2, 9, 9, 48, 336, 3, 3, 2, 1),
    (3, 1, 4, 4, 1, 1, 3, 3, 1, 1),          # a single channel (cc)
]


@pytest.mark.parametrize("case", RAGGED_CASES)
def test_qconv_ragged_channels(case):
    test_qconv_all_three(case)
    test_qconv_fwd_affine(case)
    test_qconv_bwd_affine(case)


# group widths of backward-weight: the narrowest that give every SM one tile (16, 32, 64 channels, with a part-empty last
# group), loops of up to four blocks with wide groups of 32-byte rows, split loops; channel counts that end inside 16
@pytest.mark.parametrize("nodes,rows,cin,cout", [(2, 815, 128, 304), (2, 2008, 32, 272), (3, 21, 32, 416), (1, 7, 16, 17), (8, 43, 64, 160),
                                                 (2, 100, 700, 1001), (6, 20, 704, 3360), (6, 20, 704, 3345), (1, 5000, 64, 250),
                                                 (1, 2500, 30, 10), (5, 128, 512, 512)])
def test_backward_weight_group_widths(nodes, rows, cin, cout):
    rng = np.random.default_rng(rows)
    A, E = wlmod.random_s8(rng, (nodes, rows, cin)), wlmod.random_s8(rng, (nodes, rows, cout))
    s1, s2 = rng.uniform(0.001, 0.1, (2, nodes)).astype(np.float32)
    desc = api.conv_desc(nodes, rows, 1, 1, cin, cout, 1, 1, 1, 0)
    ws = ws_bytes(api.lpdt_qconv_workspace_size(desc, 2))
    acc = torch.full((nodes, cout, cin), 77, dtype=torch.int32, device="cuda")
    dW = torch.full((nodes, cout * cin + 5), 9.0, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_bwd_weight(desc, dev(E), dev(s1), dev(A), dev(s2), dW=dW, dw_node_stride=cout * cin + 5, dWacc=acc, ws=ws,
                              dev_status=status)
    assert api.lpdt_last_kernel().endswith("conv_wgrad_kernel") and int(status.item()) == 0
    ref = torch.from_numpy(E).cuda().double().transpose(1, 2) @ torch.from_numpy(A).cuda().double()
    assert torch.equal(acc.double(), ref)
    want = oracle.dequant_acc(acc.cpu().numpy().reshape(nodes, -1), s1, s2)
    only = torch.full_like(dW, 9.0)
    api.lpdt_qconv_bwd_weight(desc, dev(E), dev(s1), dev(A), dev(s2), dW=only, dw_node_stride=cout * cin + 5, ws=ws)
    for got in (dW, only):
        assert np.array_equal(got[:, :cout * cin].cpu().numpy(), want) and bool((got[:, cout * cin:] == 9.0).all())


# strided backward-data: pixels that no tap reaches (1x1 of stride 2, and a filter of two rows), results in rows of 16 bytes
# and not, tiles of every row width, more tiles than one wave
STRIDED_CASES = [(2, 3, 9, 9, 352, 48, 1, 1, 2, 0), (1, 2, 8, 8, 30, 16, 1, 1, 2, 0), (2, 2, 7, 11, 21, 33, 1, 1, 2, 0), (1, 40, 28, 28, 80, 32, 1, 1, 2, 0),
                 (2, 3, 8, 8, 400, 128, 3, 3, 2, 1), (1, 2, 9, 12, 272, 96, 2, 1, 2, 0), (1, 1, 1, 1, 64, 64, 1, 1, 2, 0), (1, 2, 5, 5, 16, 20, 1, 1, 2, 2)]


@pytest.mark.parametrize("case", STRIDED_CASES)
def test_qconv_strided(case):
    test_qconv_all_three(case)
    test_qconv_fwd_affine(case)
    test_qconv_bwd_affine(case)
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    A, Wq, E, s1, s2 = _conv_inputs(case)
    desc = api.conv_desc(*case)
    addend = np.random.default_rng(3).standard_normal(A.shape).astype(np.float32)
    dA = torch.full(A.shape, float("nan"), dtype=torch.float32, device="cuda")
    ws = ws_bytes(api.lpdt_qconv_workspace_size(desc, 1))
    api.lpdt_qconv_bwd_data(desc, dev(E), dev(s1), dev(Wq), dev(s2), dA=dA, ws=ws, addend=dev(addend))
    ref = oracle.residual_add_bwd(addend, oracle.dequant_acc(oracle.qconv_bwd_data(E, Wq, H, W, stride, pad)[0], s1, s2))
    assert np.array_equal(dA.cpu().numpy(), ref)


# maps of odd sizes with few images: every split of the 128 pixels of a tile, boxes that reach past the map on two axes
@pytest.mark.parametrize("case", [(2, 5, 27, 27, 32, 48, 3, 3, 1, 1), (1, 3, 25, 13, 48, 32, 3, 3, 2, 1), (2, 12, 7, 7, 64, 80, 3, 3, 1, 1),
                                  (1, 5, 39, 11, 16, 16, 5, 5, 1, 2), (1, 2, 33, 28, 20, 36, 3, 3, 1, 1), (1, 3, 1, 29, 16, 130, 1, 3, 1, 1),
                                  (1, 1, 131, 3, 64, 32, 3, 3, 1, 1), (3, 1, 6, 130, 32, 16, 1, 1, 2, 0)])
def test_qconv_odd_maps(case):
    test_qconv_all_three(case)
    test_qconv_fwd_affine(case)
    test_qconv_bwd_affine(case)


@pytest.mark.parametrize("rows,cin,skew", [(300 * 1024, 3, 0), (300 * 1024 + 1, 3, 1), (100 * 1024 - 3, 33, 0), (100 * 1024 + 1, 33, 3),
                                           (303104, 5, 0), (303103, 5, 0), (303103, 1, 2), (7, 17, 1)])
def test_padded_copies_of_many_rows(rows, cin, skew):
    """Operands whose rows no TMA can address, at every byte offset, on both sides of the size from which a thread copies
    several pieces; the last row ends the allocation."""
    rng = np.random.default_rng(rows + cin)
    A, Wq = wlmod.random_s8(rng, (rows, cin)), wlmod.random_s8(rng, (80, cin))
    desc = api.conv_desc(1, rows, 1, 1, cin, 80, 1, 1, 1, 0)
    Ad = torch.empty(rows * cin + skew, dtype=torch.int8, device="cuda")[skew:].view(rows, cin)
    Ad.copy_(dev(A))
    Y = torch.full((rows, 80), 77, dtype=torch.int32, device="cuda")
    ws = torch.full((api.lpdt_qconv_workspace_size(desc, 0),), 85, dtype=torch.uint8, device="cuda")
    api.lpdt_qconv_fwd(desc, Ad, None, dev(Wq), None, Yacc=Y, ws=ws)
    assert rows < 100 or api.lpdt_last_kernel() in ("lpdt::tc::conv_pix_kernel", "lpdt::tc::conv_halo16_kernel")
    assert torch.equal(Y.double(), torch.from_numpy(A).cuda().double() @ torch.from_numpy(Wq).cuda().double().t())


# the table of the weights' sums: blocks of every size (one row of lanes, few and long rows, several goes), both directions
@pytest.mark.parametrize("case", [(2, 40, 1, 1, 2064, 48, 1, 1, 1, 0), (13, 70, 1, 1, 512, 96, 1, 1, 1, 0), (1, 2000, 1, 1, 64, 16, 1, 1, 1, 0),
                                  (2, 6, 9, 9, 32, 16, 3, 3, 1, 1), (1, 3, 12, 12, 48, 32, 2, 2, 1, 0), (1, 2, 10, 10, 16, 16, 1, 3, 2, 1),
                                  (1, 40, 8, 8, 20, 650, 1, 1, 1, 0), (2, 113, 1, 1, 115, 12, 1, 1, 1, 0)])
def test_zero_point_weight_tables(case):
    test_qconv_fwd_affine(case)
    test_qconv_bwd_affine(case)


# forward products on both sides of the line between CUDA cores and tensor cores, with the kernel that each takes: up to 64
# steps a result (4 channels each where rows allow it) and 148 * 16384 steps in all
@pytest.mark.parametrize("case,kernel", [
    ((4, 4, 16, 16, 3, 16, 3, 3, 1, 1), "conv_fwd_generic"),        # 65 K results of 27 steps
    ((4, 4, 16, 16, 3, 32, 3, 3, 1, 1), "conv_halo16_kernel"),      # 131 K: a first layer of 3 channels
    ((2, 16, 16, 16, 3, 24, 3, 3, 1, 1), "conv_pix_kernel"),        # 24 results in a tile of 32
    ((2, 130, 1, 1, 200, 270, 1, 1, 1, 0), "conv_pix_kernel"),      # results in rows of 270: no 16-byte rows
    ((1, 60, 9, 11, 7, 21, 3, 3, 1, 1), "conv_pix_kernel"),
    ((3, 300, 6, 6, 16, 15, 3, 3, 1, 1), "conv_pix_kernel"),        # whole input rows, one result short of a row
    ((40, 32, 1, 1, 64, 10, 1, 1, 1, 0), "conv_fwd_generic"),       # a classifier: 13 K results of 16 steps
    ((8, 32, 1, 1, 512, 10, 1, 1, 1, 0), "conv_pix_kernel")])       # 128 steps
def test_qconv_forward_takes_the_sooner_cores(case, kernel):
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    A, Wq, E, s1, s2 = _conv_inputs(case)
    desc = api.conv_desc(*case)
    Y = torch.full(E.shape, float("nan"), dtype=torch.float32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_fwd(desc, dev(A), dev(s1), dev(Wq), dev(s2), Y=Y, ws=ws_bytes(api.lpdt_qconv_workspace_size(desc, 0)), dev_status=status)
    assert api.lpdt_last_kernel().endswith(kernel)
    assert np.array_equal(Y.cpu().numpy(), oracle.dequant_acc(oracle.qconv_fwd(A, Wq, stride, pad)[0], s1, s2))
    assert int(status.item()) == 0


# long K loops and enough 256-channel tiles for the kernel on pairs of SMs: an odd number of pixel tiles (the last pair is
# half empty), part-zero boxes on the summed side, a part-empty last channel tile; a convolution with a halo; a filter in
# both directions, whose boxes of weights end inside the next node's rows
PAIR_CASES = [(12, 300, 1, 1, 1300, 1284, 1, 1, 1, 0), (2, 33, 12, 12, 128, 512, 3, 3, 1, 1), (3, 23, 8, 16, 368, 488, 3, 3, 1, 1)]


@pytest.mark.parametrize("case", PAIR_CASES)
def test_qconv_pairs_of_sms(case):
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    A, Wq, E, s1, s2 = _conv_inputs(case)
    desc = api.conv_desc(*case)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Y = torch.full(E.shape, float("nan"), dtype=torch.float32, device="cuda")
    bias = np.random.default_rng(1).standard_normal((nodes, Cout)).astype(np.float32)
    ws = ws_bytes(max(api.lpdt_qconv_workspace_size(desc, w) for w in (0, 1)))
    api.lpdt_qconv_fwd(desc, dev(A), dev(s1), dev(Wq), dev(s2), Y=Y, bias=dev(bias), bias_node_stride=Cout, ws=ws, dev_status=status)
    assert api.lpdt_last_kernel().endswith("conv_pair_kernel")
    # the integer sums exactly, from float64 matrix products tap by tap; then the oracle's dequantization
    Af, Wf, Ef = (torch.from_numpy(t).cuda().double() for t in (A, Wq, E))
    acc = torch.zeros(E.shape, dtype=torch.float64, device="cuda")
    dacc = torch.zeros(A.shape, dtype=torch.float64, device="cuda")
    for n in range(nodes):
        for r in range(R):
            for q in range(S):
                oh, ih = slice(max(0, pad - r), min(H, H + pad - r)), slice(max(0, r - pad), min(H, H + r - pad))
                ow, iw = slice(max(0, pad - q), min(W, W + pad - q)), slice(max(0, q - pad), min(W, W + q - pad))
                acc[n, :, oh, ow] += Af[n, :, ih, iw] @ Wf[n, :, r, q].t()
                dacc[n, :, ih, iw] += Ef[n, :, oh, ow] @ Wf[n, :, r, q]
    acc, dacc = acc.cpu().numpy().astype(np.int64).astype(np.int32), dacc.cpu().numpy().astype(np.int64).astype(np.int32)
    assert np.array_equal(Y.cpu().numpy(), oracle.dequant_acc(acc, s1, s2, bias))
    addend = np.random.default_rng(2).standard_normal(A.shape).astype(np.float32)
    dA = torch.full(A.shape, float("nan"), dtype=torch.float32, device="cuda")
    api.lpdt_qconv_bwd_data(desc, dev(E), dev(s1), dev(Wq), dev(s2), dA=dA, ws=ws, dev_status=status, addend=dev(addend))
    if Cin >= 256:
        assert api.lpdt_last_kernel().endswith("conv_pair_kernel")
    assert np.array_equal(dA.cpu().numpy(), oracle.residual_add_bwd(addend, oracle.dequant_acc(dacc, s1, s2)))
    assert int(status.item()) == 0


@pytest.mark.parametrize("case", [RAGGED_CASES[0], RAGGED_CASES[3]])
def test_qconv_ragged_channels_without_room_for_copies(case):
    # the least workspace (no room for padded operand copies) and none at all where none is required: same sums
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    A, Wq, E, _, _ = _conv_inputs(case)
    desc = api.conv_desc(*case)
    wn = nodes * Cout * R * S * Cin
    up = lambda n: (n + 255) // 256 * 256
    Yacc = torch.empty(E.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_fwd(desc, dev(A), None, dev(Wq), None, Yacc=Yacc)
    assert np.array_equal(Yacc.cpu().numpy(), oracle.qconv_fwd(A, Wq, stride, pad)[0])
    dAacc = torch.empty(A.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_bwd_data(desc, dev(E), None, dev(Wq), None, dAacc=dAacc, ws=ws_bytes(up(wn)))
    assert np.array_equal(dAacc.cpu().numpy(), oracle.qconv_bwd_data(E, Wq, H, W, stride, pad)[0])
    dWacc = torch.empty(Wq.shape, dtype=torch.int32, device="cuda")
    least = up(4 * wn) + up(nodes * B * H * W * ((Cin + 15) // 16 * 16))
    api.lpdt_qconv_bwd_weight(desc, dev(E), None, dev(A), None, dWacc=dWacc, ws=ws_bytes(least))
    assert np.array_equal(dWacc.cpu().numpy(), oracle.qconv_bwd_weight(E, A, R, S, stride, pad)[0])


def test_qconv_fwd_affine_matches_quantizer_output():
    # end to end with lpdt_quantize's affine mode: real 0 maps to the zero point, so a zero-padded real
    # convolution of the dequantized tensors equals scale * acc
    nodes, B, H, W, Cin, Cout = 2, 2, 10, 9, 16, 32
    rng = np.random.default_rng(5)
    x = rng.standard_normal((nodes, B, H, W, Cin)).astype(np.float32) + 0.7
    w = rng.standard_normal((nodes, Cout, 3, 3, Cin)).astype(np.float32) * 0.1
    qx, sx, zx = oracle.quantize_affine_u8(x.reshape(nodes, -1))
    qw, sw, zw = oracle.quantize_affine_u8(w.reshape(nodes, -1))
    A, Wq = qx.reshape(x.shape), qw.reshape(w.shape)
    acc_ref, _ = oracle.qconv_fwd_affine(A, zx, Wq, zw, 1, 1)
    desc = api.conv_desc(nodes, B, H, W, Cin, Cout, 3, 3, 1, 1)
    Yacc = torch.empty(acc_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_fwd_affine(desc, dev(A), dev(sx), dev(zx.astype(np.int32)), dev(Wq), dev(sw), dev(zw.astype(np.int32)),
                              Yacc=Yacc, ws=ws_bytes(api.lpdt_qconv_fwd_affine_workspace_size(desc)))
    assert np.array_equal(Yacc.cpu().numpy(), acc_ref)


def test_qconv_fwd_affine_errors():
    desc = api.conv_desc(1, 1, 4, 4, 16, 16)
    A = torch.zeros(1, 1, 4, 4, 16, dtype=torch.uint8, device="cuda")
    Wq = torch.zeros(1, 16, 3, 3, 16, dtype=torch.uint8, device="cuda")
    z = torch.zeros(1, dtype=torch.int32, device="cuda")
    Yacc = torch.zeros(1, 1, 4, 4, 16, dtype=torch.int32, device="cuda")
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_qconv_fwd_affine(desc, A, None, z, Wq, None, z, Yacc=Yacc, ws=ws_bytes(256))
    assert e.value.code == 3                                 # workspace too small
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_qconv_fwd_affine(desc, A, None, None, Wq, None, z, Yacc=Yacc,
                                  ws=ws_bytes(api.lpdt_qconv_fwd_affine_workspace_size(desc)))
    assert e.value.code == 1                                 # zero points missing


@pytest.mark.parametrize("case", CONV_CASES)
def test_qconv_all_three(case):
    nodes, B, H, W, Cin, Cout, R, S, stride, pad = case
    A, Wq, E, s1, s2 = _conv_inputs(case)
    desc = api.conv_desc(*case)
    ws = ws_bytes(max(api.lpdt_qconv_workspace_size(desc, w) for w in (0, 1, 2)))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    Ad, Wd, Ed, s1d, s2d = dev(A), dev(Wq), dev(E), dev(s1), dev(s2)
    # forward, with bias living in a strided parameter vector
    acc_ref, ovf = oracle.qconv_fwd(A, Wq, stride, pad)
    assert ovf == 0
    bias = np.random.default_rng(1).standard_normal((nodes, Cout + 3)).astype(np.float32)
    Y = torch.empty(acc_ref.shape, dtype=torch.float32, device="cuda")
    Yacc = torch.empty(acc_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_fwd(desc, Ad, s1d, Wd, s2d, Y=Y, Yacc=Yacc, bias=dev(bias)[:, 3:], bias_node_stride=Cout + 3,
                       ws=ws, dev_status=status)
    assert np.array_equal(Yacc.cpu().numpy(), acc_ref)
    assert np.array_equal(Y.cpu().numpy(), oracle.dequant_acc(acc_ref, s1, s2, bias[:, 3:]))
    # fp32-only output (the path the training step takes; results may leave through bulk tensor stores):
    # same values, every element written, nothing written outside the tensor
    def guarded(shape):
        n = int(np.prod(shape))
        buf = torch.full((n + 2048,), float("nan"), dtype=torch.float32, device="cuda")
        return buf, buf[1024:1024 + n].view(*shape)
    buf, Y2 = guarded(acc_ref.shape)
    api.lpdt_qconv_fwd(desc, Ad, s1d, Wd, s2d, Y=Y2, bias=dev(bias)[:, 3:], bias_node_stride=Cout + 3, ws=ws,
                       dev_status=status)
    assert torch.equal(Y2, Y) and bool(buf[:1024].isnan().all()) and bool(buf[-1024:].isnan().all())
    # backward data
    dA_ref, _ = oracle.qconv_bwd_data(E, Wq, H, W, stride, pad)
    dA = torch.empty(dA_ref.shape, dtype=torch.float32, device="cuda")
    dAacc = torch.empty(dA_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_bwd_data(desc, Ed, s1d, Wd, s2d, dA=dA, dAacc=dAacc, ws=ws, dev_status=status)
    assert np.array_equal(dAacc.cpu().numpy(), dA_ref)
    assert np.array_equal(dA.cpu().numpy(), oracle.dequant_acc(dA_ref, s1, s2))
    buf, dA2 = guarded(dA_ref.shape)
    api.lpdt_qconv_bwd_data(desc, Ed, s1d, Wd, s2d, dA=dA2, ws=ws, dev_status=status)
    assert torch.equal(dA2, dA) and bool(buf[:1024].isnan().all()) and bool(buf[-1024:].isnan().all())
    # fused shortcut gradient: dA = dequantized sums + addend, one more fp32 addition (= the oracle's residual adjoint)
    addend = np.random.default_rng(2).standard_normal(dA_ref.shape).astype(np.float32)
    buf, dA3 = guarded(dA_ref.shape)
    api.lpdt_qconv_bwd_data(desc, Ed, s1d, Wd, s2d, dA=dA3, ws=ws, dev_status=status, addend=dev(addend))
    want = oracle.residual_add_bwd(addend, oracle.dequant_acc(dA_ref, s1, s2))
    assert np.array_equal(dA3.cpu().numpy(), want) and bool(buf[:1024].isnan().all()) and bool(buf[-1024:].isnan().all())
    dA4 = torch.empty_like(dA); dAacc4 = torch.empty_like(dAacc)
    api.lpdt_qconv_bwd_data(desc, Ed, s1d, Wd, s2d, dA=dA4, dAacc=dAacc4, ws=ws, dev_status=status, addend=dev(addend))
    assert torch.equal(dA4, dA3) and torch.equal(dAacc4, dAacc)
    # backward weight, into a strided gradient vector
    dW_ref, _ = oracle.qconv_bwd_weight(E, A, R, S, stride, pad)
    wn = Cout * R * S * Cin
    dW = torch.zeros(nodes, wn + 5, dtype=torch.float32, device="cuda")
    dWacc = torch.empty(dW_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_bwd_weight(desc, Ed, s1d, Ad, s2d, dW=dW[:, 5:], dw_node_stride=wn + 5, dWacc=dWacc, ws=ws,
                              dev_status=status)
    assert np.array_equal(dWacc.cpu().numpy(), dW_ref)
    assert np.array_equal(dW[:, 5:].cpu().numpy(), oracle.dequant_acc(dW_ref, s1, s2).reshape(nodes, wn))
    assert float(dW[:, :5].abs().max()) == 0.0
    # fp32-only outputs (workspace accumulators) give the same values
    dW2 = torch.zeros(nodes, wn, dtype=torch.float32, device="cuda")
    api.lpdt_qconv_bwd_weight(desc, Ed, s1d, Ad, s2d, dW=dW2, dw_node_stride=wn, ws=ws, dev_status=status)
    assert torch.equal(dW2, dW[:, 5:])
    assert int(status.item()) == 0


def test_qconv_extreme_values_and_errors():
    # all operands at +-127: the largest accumulators the shape can produce
    case = (1, 2, 6, 6, 16, 16, 3, 3, 1, 1)
    A = np.full((1, 2, 6, 6, 16), 127, np.int8); Wq = np.full((1, 16, 3, 3, 16), -127, np.int8)
    desc = api.conv_desc(*case)
    acc_ref, _ = oracle.qconv_fwd(A, Wq, 1, 1)
    Yacc = torch.empty(acc_ref.shape, dtype=torch.int32, device="cuda")
    api.lpdt_qconv_fwd(desc, dev(A), None, dev(Wq), None, Yacc=Yacc, ws=ws_bytes(256))
    assert np.array_equal(Yacc.cpu().numpy(), acc_ref) and acc_ref.min() == -127 * 127 * 144
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_qconv_fwd(desc, dev(A), None, dev(Wq), None, ws=ws_bytes(256))      # no output
    assert e.value.code == 1
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_qconv_bwd_data(desc, dev(A), None, dev(Wq), None, dAacc=Yacc, ws=None)
    assert e.value.code == 3
    bad = api.conv_desc(1, 1, 2, 2, 4, 4, 5, 5, 1, 0)                                 # kernel larger than image
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_qconv_fwd(bad, dev(A), None, dev(Wq), None, Yacc=Yacc, ws=ws_bytes(256))
    assert e.value.code == 1


# ------------------------------------------------------------------ Range-EvoNorm
REN_CASES = [(4, 8, 16, 16, 16, 4), (2, 3, 32, 32, 16, 2), (2, 2, 8, 8, 64, 8), (1, 3, 5, 7, 6, 3),
             (1, 2, 4, 4, 12, 1), (2, 2, 32, 32, 64, 8), (1, 2, 2, 2, 512, 64), (1, 1, 1, 1, 8, 2),
             # samples split over a cluster: ragged pixel counts, odd column counts, large samples
             (1, 3, 7, 9, 24, 3), (1, 2, 15, 15, 32, 4), (2, 1, 9, 9, 16, 2), (1, 2, 31, 33, 64, 16), (1, 1, 40, 40, 64, 8),
             (2, 40, 16, 16, 32, 4)]


def _ren_inputs(case, seed=0, ties=False):
    nodes, B, H, W, C, groups = case
    rng = np.random.default_rng(seed)
    x = (2 * rng.standard_normal((nodes, B, H, W, C))).astype(np.float32)
    if ties:
        x = np.round(x * 2) / 2                # 8-bit-like grid: many tied extrema, hits u = +-3 exactly
    pad = 7
    P = rng.uniform(0.5, 1.5, (nodes, 3 * C + pad)).astype(np.float32)
    P[:, 2 * C:3 * C] -= 1.0
    if ties:
        P[:, :C] = 1.0
    dy = rng.standard_normal(x.shape).astype(np.float32)
    return x, P, dy


@pytest.mark.parametrize("case", REN_CASES)
@pytest.mark.parametrize("ties", [False, True])
def test_range_evonorm_fwd_bwd(case, ties):
    nodes, B, H, W, C, groups = case
    x, P, dy = _ren_inputs(case, ties=ties)
    eps = 1e-5
    v, g, b = P[:, :C], P[:, C:2 * C], P[:, 2 * C:3 * C]
    y32, mn, mx, amn, amx = oracle.range_evonorm_fwd(x, v, g, b, groups, eps, "f32")
    y64 = oracle.range_evonorm_fwd(x, v, g, b, groups, eps, "f64")[0]
    xd, Pd = dev(x), dev(P)
    stride = P.shape[1]
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    i = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")
    y, gmin, gmax, amin_, amax_ = f(*x.shape), f(nodes, B, groups), f(nodes, B, groups), i(nodes, B, groups), i(nodes, B, groups)
    api.lpdt_range_evonorm_fwd(nodes, B, H, W, C, groups, eps, xd, Pd, Pd[:, C:], Pd[:, 2 * C:], stride, y, gmin, gmax,
                               amin_, amax_)
    assert np.array_equal(gmin.cpu().numpy(), mn) and np.array_equal(gmax.cpu().numpy(), mx)
    assert np.array_equal(amin_.cpu().numpy(), amn) and np.array_equal(amax_.cpu().numpy(), amx)
    assert np.array_equal(y.cpu().numpy(), y32)            # same fp32 operation sequence: bit-equal
    close(y, y64)
    dx32, dv32, dg32, db32 = oracle.range_evonorm_bwd(dy, x, v, g, mn, mx, amn, amx, groups, eps, "f32")
    dx64, dv64, dg64, db64 = oracle.range_evonorm_bwd(dy, x, v, g, mn, mx, amn, amx, groups, eps, "f64")
    G = torch.zeros(nodes, stride, dtype=torch.float32, device="cuda")
    dx = f(*x.shape)
    ws = ws_bytes(api.lpdt_range_evonorm_bwd_workspace_size(nodes, B, C))
    api.lpdt_range_evonorm_bwd(nodes, B, H, W, C, groups, eps, dev(dy), xd, Pd, Pd[:, C:], stride, gmin, gmax, amin_, amax_,
                               dx, G, G[:, C:], G[:, 2 * C:], stride, ws)
    close(dx, dx32, 1e-6, 1e-7)
    close(dx, dx64)
    # two-call form: dx first, the parameter-gradient sums later from the partial sums in the workspace
    G2 = torch.zeros_like(G); dx2 = f(*x.shape)
    api.lpdt_range_evonorm_bwd(nodes, B, H, W, C, groups, eps, dev(dy), xd, Pd, Pd[:, C:], stride, gmin, gmax, amin_, amax_,
                               dx2, None, None, None, stride, ws)
    api.lpdt_range_evonorm_bwd_params(nodes, B, C, ws, G2, G2[:, C:], G2[:, 2 * C:], stride)
    assert torch.equal(dx2, dx) and torch.equal(G2, G)
    # parameter-gradient sums at the stated bar (1e-5 relative + 1e-6 absolute, no scaling): the kernel adds
    # the same fp32 terms as the oracle's fp32 instantiation into double accumulators, so it sits within
    # double rounding noise of that one, and within the bar of the all-double evaluation
    Gh = G.cpu().numpy()
    for got, w32, w64 in ((Gh[:, :C], dv32, dv64), (Gh[:, C:2 * C], dg32, dg64), (Gh[:, 2 * C:3 * C], db32, db64)):
        close(got, w32, 1e-6, 1e-7)
        close(got, w64, RTOL, ATOL)
    assert not Gh[:, 3 * C:].any()


@pytest.mark.parametrize("case", REN_CASES)
def test_range_evonorm_fwd_fused_shortcut(case):
    """y = RangeEvoNorm(x) + res in one launch: one more fp32 addition on the bit-equal norm output; the
    per-node max|y| it reports is that of the sum."""
    nodes, B, H, W, C, groups = case
    x, P, _ = _ren_inputs(case, seed=3)
    v, g, b = P[:, :C], P[:, C:2 * C], P[:, 2 * C:3 * C]
    res = np.random.default_rng(11).standard_normal(x.shape).astype(np.float32)
    y32, mn, mx, amn, amx = oracle.range_evonorm_fwd(x, v, g, b, groups, 1e-5, "f32")
    want = oracle.residual_add(res, y32)
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    i = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")
    Pd = dev(P)
    y, gmin, gmax, amin_, amax_ = f(*x.shape), f(nodes, B, groups), f(nodes, B, groups), i(nodes, B, groups), i(nodes, B, groups)
    rng_out = torch.zeros(nodes, device="cuda")
    api.lpdt_range_evonorm_fwd(nodes, B, H, W, C, groups, 1e-5, dev(x), Pd, Pd[:, C:], Pd[:, 2 * C:], P.shape[1], y, gmin,
                               gmax, amin_, amax_, amax_out=rng_out, res=dev(res))
    assert np.array_equal(y.cpu().numpy(), want)
    assert np.array_equal(amin_.cpu().numpy(), amn) and np.array_equal(amax_.cpu().numpy(), amx)
    assert np.array_equal(gmin.cpu().numpy(), mn) and np.array_equal(gmax.cpu().numpy(), mx)
    assert np.array_equal(rng_out.cpu().numpy(), np.abs(want).reshape(nodes, -1).max(1))


def test_fused_ranges_feed_the_quantizer_exactly():
    # the producers' per-node max|x| must equal the range pass bit for bit, so that
    # lpdt_quantize_with_range gives the same codes as lpdt_quantize
    case = (3, 4, 16, 16, 16, 2)
    nodes, B, H, W, C, groups = case
    x, P, dy = _ren_inputs(case, seed=5, ties=True)
    v, g, b = P[:, :C], P[:, C:2 * C], P[:, 2 * C:3 * C]
    y32, mn, mx, amn, amx = oracle.range_evonorm_fwd(x, v, g, b, groups, 1e-5, "f32")
    dx32 = oracle.range_evonorm_bwd(dy, x, v, g, mn, mx, amn, amx, groups, 1e-5, "f32")[0]
    xd, Pd = dev(x), dev(P)
    stride = P.shape[1]
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    i = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")
    ranges = torch.zeros(3, nodes, device="cuda")
    y, gmin, gmax, amin_, amax_ = f(*x.shape), f(nodes, B, groups), f(nodes, B, groups), i(nodes, B, groups), i(nodes, B, groups)
    api.lpdt_range_evonorm_fwd(nodes, B, H, W, C, groups, 1e-5, xd, Pd, Pd[:, C:], Pd[:, 2 * C:], stride, y, gmin, gmax,
                               amin_, amax_, amax_out=ranges[0])
    G = torch.zeros(nodes, stride, device="cuda")
    dx = f(*x.shape)
    ws = ws_bytes(api.lpdt_range_evonorm_bwd_workspace_size(nodes, B, C))
    api.lpdt_range_evonorm_bwd(nodes, B, H, W, C, groups, 1e-5, dev(dy), xd, Pd, Pd[:, C:], stride, gmin, gmax, amin_, amax_,
                               dx, G, G[:, C:], G[:, 2 * C:], stride, ws, amax_out=ranges[1])
    r = f(*x.shape)
    api.lpdt_residual_add(nodes, B, H, W, C, C, 1, 0, y, dx, r, amax_out=ranges[2])
    rh = ranges.cpu().numpy()
    assert np.array_equal(rh[0], np.abs(y32).reshape(nodes, -1).max(1))
    assert np.array_equal(rh[1], np.abs(dx.cpu().numpy()).reshape(nodes, -1).max(1))
    assert np.array_equal(rh[2], np.abs(r.cpu().numpy()).reshape(nodes, -1).max(1))
    n = B * H * W * C
    for t, row, rounding in ((y, 0, 0), (dx, 1, 1), (r, 2, 0)):
        q1 = torch.empty(nodes, n, dtype=torch.int8, device="cuda"); s1 = f(nodes)
        q2 = torch.empty(nodes, n, dtype=torch.int8, device="cuda"); s2 = f(nodes)
        api.lpdt_quantize(t, nodes, n, n, q1, s1, ws_bytes(256), rounding=rounding, seed=5, ctr_offset=1)
        api.lpdt_quantize_with_range(t, nodes, n, n, ranges[row], q2, s2, rounding=rounding, seed=5, ctr_offset=1)
        assert torch.equal(q1, q2) and torch.equal(s1, s2)


# cases whose sample fits one CTA's shared memory: one to 40 samples per node, ragged pixel counts, 2 to 128
# vector columns
REN_Q8_CASES = [(4, 8, 16, 16, 16, 4), (2, 3, 32, 32, 16, 2), (2, 2, 8, 8, 64, 8), (1, 2, 4, 4, 12, 1), (2, 2, 16, 16, 64, 8),
                (1, 2, 2, 2, 512, 64), (1, 1, 1, 1, 8, 2), (1, 3, 7, 9, 24, 3), (1, 2, 15, 17, 64, 16), (2, 40, 16, 16, 32, 4),
                (3, 32, 32, 32, 16, 2), (2, 32, 8, 8, 64, 8), (1, 5, 3, 3, 256, 8)]


def _ren_q8_check(case, ties, with_res, keep_y):
    nodes, B, H, W, C, groups = case
    x, P, dy = _ren_inputs(case, seed=21, ties=ties)
    eps = 1e-5
    v, g, b = P[:, :C], P[:, C:2 * C], P[:, 2 * C:3 * C]
    res = np.random.default_rng(5).standard_normal(x.shape).astype(np.float32) if with_res else None
    y32, mn, mx, amn, amx = oracle.range_evonorm_fwd(x, v, g, b, groups, eps, "f32")
    want_y = oracle.residual_add(res, y32) if with_res else y32
    n = B * H * W * C
    q_ref, s_ref = oracle.quantize_sym_s8(want_y.reshape(nodes, n))
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    i = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")
    xd, Pd, stride = dev(x), dev(P), P.shape[1]
    assert api.lpdt_range_evonorm_fwd_q8_fits(B, H, W, C, groups) == 1
    assert api.lpdt_range_evonorm_bwd_q8_fits(B, H, W, C, groups) == 1
    ctl = torch.zeros(api.lpdt_range_evonorm_q8_ctl_size(nodes), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    y = torch.full(x.shape, float("nan"), dtype=torch.float32, device="cuda") if keep_y else None
    gmin, gmax, amin_, amax_ = f(nodes, B, groups), f(nodes, B, groups), i(nodes, B, groups), i(nodes, B, groups)
    q = torch.full((nodes, n), 99, dtype=torch.int8, device="cuda")
    sc = f(nodes)
    rng_out = torch.full((nodes,), -1.0, device="cuda")
    api.lpdt_range_evonorm_fwd_q8(nodes, B, H, W, C, groups, eps, xd, Pd, Pd[:, C:], Pd[:, 2 * C:], stride, y, gmin, gmax,
                                  amin_, amax_, q, sc, ctl, amax_out=rng_out, res=None if res is None else dev(res),
                                  dev_status=status)
    assert not ctl.any() and int(status.item()) == 0           # the control block is left clean
    assert np.array_equal(gmin.cpu().numpy(), mn) and np.array_equal(gmax.cpu().numpy(), mx)
    assert np.array_equal(amin_.cpu().numpy(), amn) and np.array_equal(amax_.cpu().numpy(), amx)
    if keep_y:
        assert np.array_equal(y.cpu().numpy(), want_y)
    assert np.array_equal(rng_out.cpu().numpy(), np.abs(want_y).reshape(nodes, -1).max(1))
    assert np.array_equal(sc.cpu().numpy(), s_ref)
    assert np.array_equal(q.cpu().numpy(), q_ref)            # the oracle's norm followed by the oracle's quantizer
    # backward: the codes of dx.  dx itself matches the oracle to 1e-6 relative, not bit for bit, so the codes are
    # pinned two ways: they equal the ORACLE's quantizer applied to the dx the plain backward call writes (same
    # arithmetic inside the fused kernel), and dequantized they sit within half a step of the oracle's dx
    dx32 = oracle.range_evonorm_bwd(dy, x, v, g, mn, mx, amn, amx, groups, eps, "f32")[0]
    dx = f(*x.shape)
    ws = ws_bytes(api.lpdt_range_evonorm_bwd_workspace_size(nodes, B, C))
    G = torch.zeros(nodes, stride, device="cuda")
    api.lpdt_range_evonorm_bwd(nodes, B, H, W, C, groups, eps, dev(dy), xd, Pd, Pd[:, C:], stride, gmin, gmax, amin_, amax_,
                               dx, G, G[:, C:], G[:, 2 * C:], stride, ws)
    qe_ref, se_ref = oracle.quantize_sym_s8(dx.cpu().numpy().reshape(nodes, n))
    E = torch.full((nodes, n), 99, dtype=torch.int8, device="cuda")
    sE = f(nodes)
    G2 = torch.zeros_like(G)
    ws2 = ws_bytes(api.lpdt_range_evonorm_bwd_workspace_size(nodes, B, C))
    rng2 = torch.full((nodes,), -1.0, device="cuda")
    api.lpdt_range_evonorm_bwd_q8(nodes, B, H, W, C, groups, eps, dev(dy), xd, Pd, Pd[:, C:], stride, gmin, gmax, amin_,
                                  amax_, E, sE, G2, G2[:, C:], G2[:, 2 * C:], stride, ws2, ctl, amax_out=rng2,
                                  dev_status=status)
    assert not ctl.any() and int(status.item()) == 0
    assert np.array_equal(sE.cpu().numpy(), se_ref)
    assert np.array_equal(E.cpu().numpy(), qe_ref)
    assert torch.equal(G2, G)
    assert np.array_equal(rng2.cpu().numpy(), np.abs(dx.cpu().numpy()).reshape(nodes, -1).max(1))
    deq = E.cpu().numpy().astype(np.float64) * se_ref[:, None].astype(np.float64)
    err = np.abs(deq - dx32.reshape(nodes, n).astype(np.float64))
    bar = 0.5 * se_ref[:, None].astype(np.float64) * (1 + 1e-5) + 1e-6 * np.abs(dx32.reshape(nodes, n)) + 1e-7
    assert (err <= bar).all()
    # deferred parameter sums: same partial sums in the workspace
    G3 = torch.zeros_like(G)
    api.lpdt_range_evonorm_bwd_q8(nodes, B, H, W, C, groups, eps, dev(dy), xd, Pd, Pd[:, C:], stride, gmin, gmax, amin_,
                                  amax_, E, sE, None, None, None, stride, ws2, ctl, dev_status=status)
    api.lpdt_range_evonorm_bwd_params(nodes, B, C, ws2, G3, G3[:, C:], G3[:, 2 * C:], stride)
    assert torch.equal(G3, G) and np.array_equal(E.cpu().numpy(), qe_ref)
    assert not ctl.any() and int(status.item()) == 0


@pytest.mark.parametrize("case", [(2, 3, 8, 8, 16, 2), (1, 2, 2, 2, 64, 8), (2, 2, 4, 6, 12, 3), (1, 5, 32, 32, 64, 8),
                                  (2, 3, 16, 16, 128, 16), (1, 2, 4, 4, 512, 64), (1, 3, 6, 10, 160, 20), (5, 120, 8, 8, 32, 4),
                                  # more samples than fit with 256 threads each: 32, 64, 96 and 128 threads
                                  (3, 120, 2, 2, 16, 2), (3, 120, 4, 4, 64, 8), (2, 160, 2, 6, 96, 12), (2, 160, 2, 2, 512, 64)])
@pytest.mark.parametrize("special", ["", "ties", "infinite", "large", "v", "gamma", "constant"])
def test_range_evonorm_and_max_pooling_in_one_launch(case, special):
    """Equal to the layer and the pooling as two calls: everything to the bit, sums in double up to their order."""
    nodes, B, H, W, C, groups = case
    x, P, dy = _ren_inputs(case, seed=31, ties=special == "ties")
    if special == "infinite":
        x[0, 0, 0, 1, 0] = np.inf
        x[-1, -1, 1, 1, -1] = np.nan
    # products of finite values that are not finite, in the terms of positions that the pooling did not choose
    if special == "large":
        x[0, 0, 0, 1, 0] = x[-1, -1, 1, 0, -1] = -1e30
    if special == "v":
        P[0, 0], P[-1, C - 1] = 3e38, -np.inf
    if special == "gamma":
        P[0, C], P[-1, 2 * C - 1] = np.inf, np.nan
    if special == "constant":
        x[0, 0], x[-1, -1] = 1.5, -1.5
    eps = 0.0 if special == "constant" else 1e-5
    xd, Pd, stride = dev(x), dev(P), P.shape[1]
    f = lambda *s: torch.full(s, 7.0, device="cuda")
    i = lambda *s: torch.full(s, -5, dtype=torch.int32, device="cuda")
    stats = lambda: (f(nodes, B, groups), f(nodes, B, groups), i(nodes, B, groups), i(nodes, B, groups))
    half = (nodes, B, H // 2, W // 2, C)
    same = lambda a, b: np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())          # (NaN equals NaN, 0 equals -0)
    y, st, pooled, idx = f(*x.shape), stats(), f(*half), torch.full(half, 9, dtype=torch.int8, device="cuda")
    api.lpdt_range_evonorm_fwd(nodes, B, H, W, C, groups, eps, xd, Pd, Pd[:, C:], Pd[:, 2 * C:], stride, y, *st)
    api.lpdt_maxpool2x2(nodes, B, H, W, C, y, pooled, idx)
    st2, pooled2, idx2, amax = stats(), f(*half), torch.full(half, 9, dtype=torch.int8, device="cuda"), torch.zeros(nodes, device="cuda")
    api.lpdt_range_evonorm_pool_fwd(nodes, B, H, W, C, groups, eps, xd, Pd, Pd[:, C:], Pd[:, 2 * C:], stride, pooled2, idx2, *st2,
                                    amax_out=amax)
    for a, b in zip((pooled, idx, *st), (pooled2, idx2, *st2)):
        same(a, b)
    same(amax, pooled.abs().reshape(nodes, -1).nan_to_num(0.0, posinf=float("inf")).amax(1))
    g = dev(np.random.default_rng(3).standard_normal(half).astype(np.float32))
    full, dx, dx2, r, r2 = f(*x.shape), f(*x.shape), f(*x.shape), torch.zeros(nodes, device="cuda"), torch.zeros(nodes, device="cuda")
    n = api.lpdt_range_evonorm_bwd_workspace_size(nodes, B, C)
    acc, acc2 = torch.zeros(n, dtype=torch.uint8, device="cuda"), torch.zeros(n, dtype=torch.uint8, device="cuda")
    api.lpdt_maxpool2x2_bwd(nodes, B, H, W, C, g, idx, full)
    api.lpdt_range_evonorm_bwd(nodes, B, H, W, C, groups, eps, full, xd, Pd, Pd[:, C:], stride, *st, dx, None, None, None, stride, acc,
                               amax_out=r)
    api.lpdt_range_evonorm_pool_bwd(nodes, B, H, W, C, groups, eps, g, idx, xd, Pd, Pd[:, C:], stride, *st, dx2, acc2, amax_out=r2)
    # dx at the extrema holds the group sum, whose rounding may go the other way when its terms are added in another order
    np.testing.assert_allclose(dx2.cpu().numpy(), dx.cpu().numpy(), rtol=1.2e-7, atol=0)
    assert int((dx2 != dx).logical_and(~dx.isnan()).sum()) <= 2 * nodes * B * groups
    np.testing.assert_allclose(r2.cpu().numpy(), r.cpu().numpy(), rtol=1.2e-7, atol=0)
    a, b = (t[:nodes * B * 3 * C * 8].view(torch.float64).cpu().numpy() for t in (acc, acc2))
    np.testing.assert_allclose(b, a, rtol=0, atol=1e-15 * H * W * np.nanmax(np.abs(np.where(np.isinf(a), 0, a))))      # H W / 4 terms


def _ren_forms(case, xd, Pd, stride):
    """The forms of the layer that serve a case: name -> (forward, backward).  forward() -> (gmin, gmax, argmin, argmax);
    backward(statistics) -> (gradient of x or its codes and scales, max|gradient|), with every byte around the gradient checked."""
    nodes, B, H, W, C, groups = case
    f = lambda *s: torch.empty(*s, device="cuda")
    args, par = (nodes, B, H, W, C, groups, 1e-5), (Pd, Pd[:, C:])
    ws = ws_bytes(api.lpdt_range_evonorm_bwd_workspace_size(nodes, B, C))
    half = (nodes, B, H // 2, W // 2, C)
    rng = np.random.default_rng(17)
    dy, dyp = dev(rng.standard_normal(xd.shape).astype(np.float32)), dev(rng.standard_normal(half).astype(np.float32))
    idx = torch.empty(half, dtype=torch.int8, device="cuda")

    def stats():
        return (f(nodes, B, groups), f(nodes, B, groups), *(torch.full((nodes, B, groups), -7, dtype=torch.int32, device="cuda") for _ in "12"))

    def guarded(call, dtype=torch.float32, seal=93):
        buf = torch.full((xd.numel() + 8192,), seal, dtype=dtype, device="cuda")
        amax = torch.zeros(nodes, device="cuda")
        call(buf[4096:-4096].view(xd.shape), amax)
        assert bool((buf[:4096] == seal).all()) and bool((buf[-4096:] == seal).all())
        return buf[4096:-4096].view(xd.shape), amax

    def fwd():
        st = stats()
        api.lpdt_range_evonorm_fwd(*args, xd, *par, Pd[:, 2 * C:], stride, f(xd.shape), *st)
        return st

    def bwd(st):
        return guarded(lambda dx, amax: api.lpdt_range_evonorm_bwd(*args, dy, xd, *par, stride, *st, dx, None, None, None, stride, ws,
                                                                   amax_out=amax))
    forms = {"plain": (fwd, bwd)}
    if C // groups % 4 == 0 and H % 2 == 0 and W % 2 == 0:
        def fwd_pool():
            st = stats()
            api.lpdt_range_evonorm_pool_fwd(*args, xd, *par, Pd[:, 2 * C:], stride, f(half), idx, *st)
            return st

        def bwd_pool(st):
            return guarded(lambda dx, amax: api.lpdt_range_evonorm_pool_bwd(*args, dyp, idx, xd, *par, stride, *st, dx, ws, amax_out=amax))
        forms["pool"] = (fwd_pool, bwd_pool)
    if api.lpdt_range_evonorm_fwd_q8_fits(B, H, W, C, groups) and api.lpdt_range_evonorm_bwd_q8_fits(B, H, W, C, groups):
        ctl = torch.zeros(api.lpdt_range_evonorm_q8_ctl_size(nodes), dtype=torch.uint8, device="cuda")

        def fwd_q8():
            st = stats()
            api.lpdt_range_evonorm_fwd_q8(*args, xd, *par, Pd[:, 2 * C:], stride, None, *st,
                                          torch.empty(xd.shape, dtype=torch.int8, device="cuda"), f(nodes), ctl)
            return st

        def bwd_q8(st):
            return guarded(lambda q, amax: api.lpdt_range_evonorm_bwd_q8(*args, dy, xd, *par, stride, *st, q, f(nodes), None, None, None,
                                                                         stride, ws, ctl, amax_out=amax), torch.int8)
        forms["q8"] = (fwd_q8, bwd_q8)
    return forms


# whole samples and samples split over a cluster (forward, backward or both), 2 to 32 channels per group, vector width 1 and 4
REN_POSITION_CASES = [(2, 4, 8, 8, 16, 2), (1, 5, 6, 6, 6, 3), (1, 4, 32, 32, 64, 8), (2, 4, 16, 16, 128, 4), (4, 120, 4, 4, 32, 4),
                      (1, 4, 7, 9, 24, 3)]


@pytest.mark.parametrize("case", REN_POSITION_CASES)
def test_range_evonorm_fwd_positions_of_groups_without_finite_values(case):
    """Every position that the forward pass stores is one of the sample (the oracle's), also where no value beats the infinity
    that a search begins with; the backward pass from these statistics writes inside the gradient and agrees with the oracle."""
    nodes, B, H, W, C, groups = case
    x, P, _ = _ren_inputs(case, seed=41)
    last = x.reshape(nodes * B, H * W, groups, C // groups)
    last[0], last[1], last[2] = np.nan, -np.inf, np.inf
    last[-1, 1:, -1] = np.nan                   # one group of infinities and NaN
    last[-1, 0, -1] = -np.inf
    xd, Pd = dev(x), dev(P)
    _, mn, mx, amn, amx = oracle.range_evonorm_fwd(x, P[:, :C], P[:, C:2 * C], P[:, 2 * C:], groups, 1e-5, "f32")
    dy = np.random.default_rng(17).standard_normal(x.shape).astype(np.float32)
    want = oracle.range_evonorm_bwd(dy, x, P[:, :C], P[:, C:2 * C], mn, mx, amn, amx, groups, 1e-5, "f32")[0]
    for name, (fwd, bwd) in _ren_forms(case, xd, Pd, P.shape[1]).items():
        st = fwd()
        assert np.array_equal(st[2].cpu().numpy(), amn) and np.array_equal(st[3].cpu().numpy(), amx), name
        dx, amax = bwd(st)
        if name == "plain":
            got = dx.cpu().numpy()
            assert np.array_equal(np.isnan(got), np.isnan(want))
            close(got[~np.isnan(want)], want[~np.isnan(want)], 1e-6, 1e-7)


@pytest.mark.parametrize("case", REN_POSITION_CASES)
@pytest.mark.parametrize("low,high", [(-1, -1), (-1, 2 ** 31 - 1), (2 ** 31 - 1, -2 ** 31), ("end", 2 ** 31 - 1), ("end", "end")])
def test_range_evonorm_fwd_then_backward_skips_positions_outside_the_sample(case, low, high):
    """A caller's position outside the sample takes no correction: the gradient is that of equal positions (whose corrections
    cancel), and nothing around it is touched."""
    nodes, B, H, W, C, groups = case
    x, P, _ = _ren_inputs(case, seed=43)
    low, high = (H * W * C if v == "end" else v for v in (low, high))
    for name, (fwd, bwd) in _ren_forms(case, dev(x), dev(P), P.shape[1]).items():
        st = fwd()
        st[2].fill_(0), st[3].fill_(0)
        want, amax_want = bwd(st)
        st[2].fill_(low), st[3].fill_(high)
        dx, amax = bwd(st)
        assert torch.equal(dx, want) and torch.equal(amax, amax_want), name


@pytest.mark.parametrize("case", REN_Q8_CASES)
@pytest.mark.parametrize("ties", [False, True])
def test_range_evonorm_q8(case, ties):
    """Range-EvoNorm with the requantize step inside: codes, scales, statistics and parameter gradients equal
    those of the norm call followed by the quantizer."""
    _ren_q8_check(case, ties, with_res=False, keep_y=False)
    _ren_q8_check(case, ties, with_res=True, keep_y=True)


@pytest.mark.parametrize("env", [{"LPDT_REN_Q8_THREADS": "128"}, {"LPDT_REN_Q8_THREADS": "256", "LPDT_REN_Q8_DEPTH": "4"},
                                 {"LPDT_REN_Q8_THREADS": "384"}])
def test_range_evonorm_q8_on_every_launch_shape(env):
    """The same cases in child processes with the CTA size and ring depth forced."""
    import os, subprocess, sys
    if os.environ.get("LPDT_CHILD") == "1":
        pytest.skip("already inside a child run")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    child_env = dict(os.environ, LPDT_CHILD="1", **env)
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(root, "tests", "test_gpu_ops.py"), "-m", "gpu",
                        "-q", "-x", "-k", "test_range_evonorm_q8 and not launch_shape and not reports"], env=child_env,
                       cwd=root, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and " passed" in r.stdout, r.stdout[-3000:] + r.stderr[-2000:]


def test_range_evonorm_q8_reports_shapes_that_do_not_fit():
    # a sample of 32x32x64 fp32 is 256 KB: beyond one CTA's shared memory
    assert api.lpdt_range_evonorm_fwd_q8_fits(32, 32, 32, 64, 8) == 0
    assert api.lpdt_range_evonorm_bwd_q8_fits(32, 32, 32, 64, 8) == 0
    assert api.lpdt_range_evonorm_fwd_q8_fits(4, 4, 4, 6, 3) == 0          # 2 channels per group: no 4-wide columns
    # more samples per node than half the CTAs the device can hold at once: the meeting could starve
    assert api.lpdt_range_evonorm_bwd_q8_fits(4096, 32, 32, 16, 2) == 0
    t = torch.zeros(2 * 32 * 32 * 64, device="cuda"); ti = torch.zeros(256, dtype=torch.int32, device="cuda")
    q = torch.zeros(2 * 32 * 32 * 64, dtype=torch.int8, device="cuda")
    ctl = torch.zeros(api.lpdt_range_evonorm_q8_ctl_size(1), dtype=torch.uint8, device="cuda")
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_range_evonorm_fwd_q8(1, 2, 32, 32, 64, 8, 1e-5, t, t, t, t, 64, None, t, t, ti, ti, q, t, ctl)
    assert e.value.code == 2
    with pytest.raises(api.LpdtError) as e:      # no control block
        api.lpdt_range_evonorm_fwd_q8(1, 2, 8, 8, 64, 8, 1e-5, t, t, t, t, 64, None, t, t, ti, ti, q, t, None)
    assert e.value.code == 3


def test_range_evonorm_q8_with_a_control_block_that_was_not_cleared():
    """The control block must be zero at launch.  When its ticket counter is not, the tickets name no sample of
    the call: every CTA records LPDT_ERR_INVALID_ARG and returns without touching the tensors (no out-of-range
    access), and the context stays usable."""
    nodes, B, H, W, C, groups = 2, 4, 8, 8, 16, 2
    x, P, dy = _ren_inputs((nodes, B, H, W, C, groups), seed=2)
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    i = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")
    Pd, stride = dev(P), P.shape[1]
    n = B * H * W * C
    ctl = torch.zeros(api.lpdt_range_evonorm_q8_ctl_size(nodes) // 4, dtype=torch.int32, device="cuda")
    ctl[3 * nodes] = nodes * B                         # the ticket counter of a call that never finished
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    q = torch.full((nodes, n), 77, dtype=torch.int8, device="cuda")
    sc = torch.full((nodes,), -1.0, device="cuda")
    gmin, gmax, amin_, amax_ = f(nodes, B, groups), f(nodes, B, groups), i(nodes, B, groups), i(nodes, B, groups)
    api.lpdt_range_evonorm_fwd_q8(nodes, B, H, W, C, groups, 1e-5, dev(x), Pd, Pd[:, C:], Pd[:, 2 * C:], stride, None, gmin,
                                  gmax, amin_, amax_, q, sc, ctl.view(torch.uint8), dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 1                     # LPDT_ERR_INVALID_ARG
    assert (q == 77).all() and (sc == -1.0).all()
    # cleared, the same buffers serve a correct call
    ctl.zero_(); status.zero_()
    api.lpdt_range_evonorm_fwd_q8(nodes, B, H, W, C, groups, 1e-5, dev(x), Pd, Pd[:, C:], Pd[:, 2 * C:], stride, None, gmin,
                                  gmax, amin_, amax_, q, sc, ctl.view(torch.uint8), dev_status=status)
    v, g, b = P[:, :C], P[:, C:2 * C], P[:, 2 * C:3 * C]
    y32 = oracle.range_evonorm_fwd(x, v, g, b, groups, 1e-5, "f32")[0]
    q_ref, s_ref = oracle.quantize_sym_s8(y32.reshape(nodes, n))
    assert int(status.item()) == 0 and not ctl.any()
    assert np.array_equal(q.cpu().numpy(), q_ref) and np.array_equal(sc.cpu().numpy(), s_ref)


def test_range_evonorm_errors():
    t = torch.zeros(64, device="cuda"); ti = torch.zeros(64, dtype=torch.int32, device="cuda")
    with pytest.raises(api.LpdtError) as e:      # one channel per group: the constant is infinite
        api.lpdt_range_evonorm_fwd(1, 1, 2, 2, 4, 4, 1e-5, t, t, t, t, 4, t, t, t, ti, ti)
    assert e.value.code == 1
    with pytest.raises(api.LpdtError) as e:      # groups must divide C
        api.lpdt_range_evonorm_fwd(1, 1, 2, 2, 6, 4, 1e-5, t, t, t, t, 6, t, t, t, ti, ti)
    assert e.value.code == 1


# ------------------------------------------------------------------ gossip
def _gossip_case(nodes, d, seed, heavy=False):
    rng = np.random.default_rng(seed)
    xh = rng.standard_normal((nodes, d)).astype(np.float32)
    resid = rng.standard_normal((nodes, d)) * (np.where(rng.random((nodes, d)) < 0.05, 1.0, 0.01) if heavy else 1.0)
    xhat = (xh - resid).astype(np.float32)
    return xh, xhat


@pytest.mark.parametrize("nodes,d,segs", [
    (4, 2736, None), (16, 10007, None), (8, 50000, [(0, 50000, 500)]), (40, 27041, [(0, 27041, 270)]),
    (5, 3000, [(0, 1000, 10), (1000, 1001, 1), (1001, 3000, 1999)]), (3, 1000, [(0, 1000, 0)]),
    (1, 777, [(0, 777, 5)]), (64, 300, [(0, 300, 3)]),
    # long segments: selection spread over several CTAs (with short and trivial ones beside them)
    (3, 100000, [(0, 100000, 1000)]), (2, 200000, [(0, 40000, 39999), (40000, 41000, 7), (41000, 200000, 1)]),
    (2, 70001, [(0, 33000, 0), (33000, 70001, 37001)]),
    # parameter counts that are even but not multiples of 4 (8-byte accesses), segments starting at odd offsets
    (4, 2738, None), (8, 270410, None), (6, 100002, [(0, 33333, 300), (33333, 100002, 700)]),
])
def test_gossip_mix(nodes, d, segs):
    xh, xhat = _gossip_case(nodes, d, d, heavy=True)
    W = wlmod.ring_matrix(nodes) if nodes >= 3 else np.full((nodes, nodes), 1.0 / nodes, np.float32)
    so = [0, d] if segs is None else [s[0] for s in segs] + [d]
    sk = [d] if segs is None else [s[2] for s in segs]
    gamma = 1.0 if segs is None else 0.3
    x_ref, xhat_ref, q_ref = oracle.gossip_mix(xh, xhat, W, gamma, so, sk)
    xhd, xhatd = dev(xh), dev(xhat)
    xo = torch.empty_like(xhd)
    ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, len(sk)))
    api.lpdt_gossip_mix(nodes, d, xhd, xhatd, xo, dev(W), gamma, so, sk, ws)
    assert np.array_equal(xhatd.cpu().numpy(), xhat_ref)          # selection + update: bit-exact
    close(xo, x_ref)
    # second call on the updated state (error feedback carried over)
    x_ref2, xhat_ref2, _ = oracle.gossip_mix(x_ref, xhat_ref, W, gamma, so, sk)
    xo2 = torch.empty_like(xhd)
    api.lpdt_gossip_mix(nodes, d, dev(x_ref), xhatd, xo2, dev(W), gamma, so, sk, ws)
    assert np.array_equal(xhatd.cpu().numpy(), xhat_ref2)
    close(xo2, x_ref2)


@pytest.mark.parametrize("nodes,d,keep", [(1, 40000, 0.1), (2, 40002, 0.3), (16, 33000, 0.1), (17, 33001, 0.1), (20, 3000, 0.01),
                                          (21, 2002, 0.1), (40, 2003, 0.5), (41, 1000, 0.1), (60, 1001, 0.1), (64, 1002, 0.01)])
def test_gossip_node_counts_and_kept_shares(nodes, d, keep):
    # one to four nodes per warp of the mix, parameter counts of every alignment with a part-empty last tile, two
    # segments that meet inside a tile, kept shares whose candidates are a window of the segment; values on a coarse
    # grid, so that ties decide the cut
    rng = np.random.default_rng(nodes)
    xh = (np.round(rng.standard_normal((nodes, d)) * 64) / 64).astype(np.float32)
    xhat = (np.round(rng.standard_normal((nodes, d)) * 2) / 64).astype(np.float32)
    W = wlmod.ring_matrix(nodes) if nodes >= 3 else np.full((nodes, nodes), 1.0 / nodes, np.float32)
    cut = d - 77
    so, sk = [0, cut, d], [max(1, int(cut * keep)), 7]
    x_ref, xhat_ref, _ = oracle.gossip_mix(xh, xhat, W, 0.3, so, sk)
    xhd, xhatd = dev(xh), dev(xhat)
    xo = torch.empty_like(xhd)
    ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, 2))
    api.lpdt_gossip_mix(nodes, d, xhd, xhatd, xo, dev(W), 0.3, so, sk, ws)
    assert np.array_equal(xhatd.cpu().numpy(), xhat_ref)
    close(xo, x_ref)


# parameter counts of 8-byte rows: the form of the mix for 6 to 24 nodes from the parameters on that give the other form more
# than one tile per CTA, and the nodes and sizes beside it; a pair of parameters that two segments share
@pytest.mark.parametrize("nodes,d", [(5, 220002), (6, 190002), (8, 40002), (8, 160002), (16, 33002), (16, 80002), (17, 2050), (20, 80002), (21, 60002),
                                     (24, 2006), (24, 60002), (25, 60002)])
def test_gossip_with_rows_of_eight_bytes(nodes, d):
    test_gossip_node_counts_and_kept_shares(nodes, d, 0.1)
    if d > 50000:
        return
    segs = [(0, d - 77, d // 50), (d - 77, d, 7)]
    test_gossip_mix_q8(nodes, d, segs)
    for bits in (32, 8):
        test_deepsqueeze_mix(nodes, d, segs, bits)


def test_gossip_topk_with_massive_ties_and_alias():
    # magnitudes from a 4-value set: the tie cut decides almost every pick
    nodes, d, k = 6, 9000, 1234
    rng = np.random.default_rng(5)
    xh = rng.choice(np.array([-2, -1, 1, 2, 0.5, -0.5], np.float32), size=(nodes, d))
    xhat = np.zeros((nodes, d), np.float32)
    W = wlmod.ring_matrix(nodes)
    x_ref, xhat_ref, q_ref = oracle.gossip_mix(xh, xhat, W, 0.5, [0, d], [k])
    assert all(np.count_nonzero(q_ref[i]) == k for i in range(nodes))
    xhd, xhatd = dev(xh), dev(xhat)
    ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, 1))
    api.lpdt_gossip_mix(nodes, d, xhd, xhatd, xhd, dev(W), 0.5, [0, d], [k], ws)   # x_out aliases x_half
    assert np.array_equal(xhatd.cpu().numpy(), xhat_ref)
    close(xhd, x_ref)


def test_gossip_topk_ties_across_chunks():
    # a long segment whose threshold value repeats thousands of times: the tie cut falls inside
    # one of many chunks, in the first one, or in the last one, depending on k
    nodes, d = 3, 90001
    rng = np.random.default_rng(11)
    xh = rng.choice(np.array([-2, -1, 1, 2, 0.5, -0.5], np.float32), size=(nodes, d))
    xh[0, :200] = 1.0; xh[0, 200:] = 0.25            # node 0: every tie of value 1 sits in the first chunk
    xh[2, :-50] = 0.125; xh[2, -50:] = -3.0           # node 2: threshold ties reach into the last chunk
    W = wlmod.ring_matrix(nodes)
    for k in (150, 20000, 60000, 89990):
        xhat = np.zeros((nodes, d), np.float32)
        x_ref, xhat_ref, q_ref = oracle.gossip_mix(xh, xhat, W, 0.5, [0, d], [k])
        assert all(np.count_nonzero(q_ref[i]) == k for i in range(nodes))
        xhd, xhatd = dev(xh), dev(xhat)
        xo = torch.empty_like(xhd)
        ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, 1))
        api.lpdt_gossip_mix(nodes, d, xhd, xhatd, xo, dev(W), 0.5, [0, d], [k], ws)
        assert np.array_equal(xhatd.cpu().numpy(), xhat_ref), k
        close(xo, x_ref)


def test_gossip_topk_candidate_list_with_planted_ties():
    """Long segments of distinct magnitudes (the candidate-list path) with the threshold value planted a few
    hundred times at scattered positions, so that only the ties at the lowest positions are kept; a second
    segment of constant magnitude overflows its list and takes the whole-segment path in the same call."""
    nodes, d1, d2, k1 = 3, 300000, 40000, 3000
    d = d1 + d2
    rng = np.random.default_rng(21)
    xh = rng.standard_normal((nodes, d)).astype(np.float32)
    for i in range(nodes):
        mags = np.sort(np.abs(xh[i, :d1]))[::-1]
        v = mags[k1 - 100]                                    # inside the top k1
        pos = rng.choice(d1, size=400, replace=False)
        xh[i, pos] = v * rng.choice(np.array([-1.0, 1.0], np.float32), size=400)
    xh[:, d1:] = 0.75
    xh[1, d1:] = 0.0                                          # all-zero differences
    xhat = np.zeros((nodes, d), np.float32)
    W = wlmod.ring_matrix(nodes)
    so, sk = [0, d1, d], [k1, 12345]
    x_ref, xhat_ref, q_ref = oracle.gossip_mix(xh, xhat, W, 0.4, so, sk)
    assert all(np.count_nonzero(q_ref[i][:d1]) == k1 for i in range(nodes))
    xhd, xhatd = dev(xh), dev(xhat)
    xo = torch.empty_like(xhd)
    ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, 2))
    api.lpdt_gossip_mix(nodes, d, xhd, xhatd, xo, dev(W), 0.4, so, sk, ws)
    assert np.array_equal(xhatd.cpu().numpy(), xhat_ref)
    close(xo, x_ref)


@pytest.mark.parametrize("nodes,d,segs", [
    (4, 2736, None), (16, 10007, None), (8, 50000, [(0, 50000, 500)]),
    (5, 3000, [(0, 1000, 10), (1000, 1001, 1), (1001, 3000, 1999)]), (3, 1000, [(0, 1000, 0)]),
    (3, 100000, [(0, 100000, 1000)]), (2, 200000, [(0, 40000, 39999), (40000, 41000, 7), (41000, 200000, 1)]),
])
def test_gossip_mix_q8(nodes, d, segs):
    """8-bit messages: public copies (hence the codes sent) bit-exact, mixed parameters within the fp32 bar,
    transmitted steps equal; two steps in a row so that the rounding error is fed back."""
    xh, xhat = _gossip_case(nodes, d, d, heavy=True)
    W = wlmod.ring_matrix(nodes) if nodes >= 3 else np.full((nodes, nodes), 1.0 / nodes, np.float32)
    so = [0, d] if segs is None else [s[0] for s in segs] + [d]
    sk = [d] if segs is None else [s[2] for s in segs]
    gamma = 1.0 if segs is None else 0.3
    xhd, xhatd = dev(xh), dev(xhat)
    ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, len(sk)))
    scale = torch.empty(nodes, len(sk), device="cuda")
    x_in, xhat_ref = xh, xhat
    for _ in range(2):
        x_ref, xhat_ref, q_ref, codes_ref, scale_ref = oracle.gossip_mix_q8(x_in, xhat_ref, W, gamma, so, sk)
        xo = torch.empty_like(xhd)
        api.lpdt_gossip_mix_q8(nodes, d, dev(x_in), xhatd, xo, dev(W), gamma, so, sk, scale, ws)
        assert np.array_equal(scale.cpu().numpy(), scale_ref)
        assert np.array_equal(xhatd.cpu().numpy(), xhat_ref)
        close(xo, x_ref)
        x_in = x_ref


@pytest.mark.parametrize("bits", [32, 8])
@pytest.mark.parametrize("nodes,d,segs", [
    (4, 2736, None), (16, 10007, [(0, 10007, 100)]), (8, 50000, [(0, 50000, 500)]),
    (5, 3000, [(0, 1000, 10), (1000, 1001, 1), (1001, 3000, 1999)]), (3, 1000, [(0, 1000, 0)]),
    (3, 100000, [(0, 100000, 1000)]),
])
def test_deepsqueeze_mix(nodes, d, segs, bits):
    """Deep-Squeeze step: error buffer (hence the messages) bit-exact, mixed parameters within the fp32 bar;
    three steps in a row so that the buffer is carried over."""
    rng = np.random.default_rng(nodes * 1000 + d)
    xh = rng.standard_normal((nodes, d)).astype(np.float32)
    delta_ref = np.zeros((nodes, d), np.float32)
    W = wlmod.ring_matrix(nodes) if nodes >= 3 else np.full((nodes, nodes), 1.0 / nodes, np.float32)
    so = [0, d] if segs is None else [s[0] for s in segs] + [d]
    sk = [d] if segs is None else [s[2] for s in segs]
    eta = 1.0 if segs is None else 0.3
    deltad = dev(delta_ref)
    ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, len(sk)))
    scale = torch.empty(nodes, len(sk), device="cuda")
    x_in = xh
    for step in range(3):
        x_ref, delta_ref, c_ref, scale_ref = oracle.deepsqueeze_mix(x_in, delta_ref, W, eta, so, sk, bits)
        xo = torch.empty(nodes, d, device="cuda")
        api.lpdt_deepsqueeze_mix(nodes, d, dev(x_in), deltad, xo, dev(W), eta, so, sk, ws, message_bits=bits,
                                 msg_scale=scale if bits == 8 else None)
        if bits == 8:
            assert np.array_equal(scale.cpu().numpy(), scale_ref)
        assert np.array_equal(deltad.cpu().numpy(), delta_ref), step
        close(xo, x_ref)
        x_in = (x_ref - 0.05 * rng.standard_normal((nodes, d))).astype(np.float32)      # a stand-in local update


@pytest.mark.parametrize("nodes,d", [(4, 2736), (16, 10007), (8, 270410), (64, 300), (1, 777), (3, 100002)])
def test_sgd_gossip_mix(nodes, d):
    """Fused half-step + dense mix: x_half and x_hat bit-equal to lpdt_sgd_update / the oracle, x within the fp32 bar;
    also bit-equal to the two separate launches."""
    rng = np.random.default_rng(nodes + d)
    x = rng.standard_normal((nodes, d)).astype(np.float32)
    g = rng.standard_normal((nodes, d)).astype(np.float32)
    xhat = (x - 0.1 * rng.standard_normal((nodes, d))).astype(np.float32)
    W = wlmod.ring_matrix(nodes) if nodes >= 3 else np.full((nodes, nodes), 1.0 / nodes, np.float32)
    xh_ref = oracle.sgd_update(x, g, 0.1)
    x_ref, xhat_ref, _ = oracle.gossip_mix(xh_ref, xhat, W, 0.9, [0, d], [d])
    xhd, xhatd, xo = torch.empty(nodes, d, device="cuda"), dev(xhat), torch.empty(nodes, d, device="cuda")
    api.lpdt_sgd_gossip_mix(nodes, d, dev(x), dev(g), 0.1, xhd, xhatd, xo, dev(W), 0.9)
    assert np.array_equal(xhd.cpu().numpy(), xh_ref) and np.array_equal(xhatd.cpu().numpy(), xhat_ref)
    close(xo, x_ref)
    xh2, xhat2, xo2 = torch.empty(nodes, d, device="cuda"), dev(xhat), torch.empty(nodes, d, device="cuda")
    api.lpdt_sgd_update(nodes * d, dev(x), dev(g), 0.1, xh2)
    api.lpdt_gossip_mix(nodes, d, xh2, xhat2, xo2, dev(W), 0.9, [0, d], [d],
                        ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, 1)))
    assert torch.equal(xo, xo2) and torch.equal(xhatd, xhat2)


def directed_ring_matrix(n, rng):
    """Column-stochastic, not row-stochastic: node j keeps a share and pushes the rest to j+1 and j+2."""
    W = np.zeros((n, n), np.float32)
    for j in range(n):
        w = rng.dirichlet(np.ones(3)).astype(np.float32)
        W[j, j] += w[0]; W[(j + 1) % n, j] += w[1]; W[(j + 2) % n, j] += w[2]
    return W


@pytest.mark.parametrize("nodes,d", [(4, 1), (5, 1001), (16, 40000), (64, 4096), (3, 270410)])
def test_pushsum_debias(nodes, d):
    """Sparse-Push over three steps: Deep-Squeeze mix with a column-stochastic matrix, then the bias
    weights and the de-biased model; bias weights and z bit-exact given the same mixed model."""
    rng = np.random.default_rng(nodes * 7 + d)
    W = directed_ring_matrix(nodes, rng)
    x = rng.standard_normal((nodes, d)).astype(np.float32)
    u_ref = np.ones(nodes, np.float32)
    ud = dev(u_ref)
    for step in range(3):
        u_new_ref, z_ref = oracle.pushsum_debias(x, u_ref, W, 0.8)
        un = torch.empty(nodes, device="cuda"); z = torch.empty(nodes, d, device="cuda")
        api.lpdt_pushsum_debias(nodes, d, dev(x), ud, dev(W), 0.8, un, z)
        assert np.array_equal(un.cpu().numpy(), u_new_ref), step
        assert np.array_equal(z.cpu().numpy(), z_ref), step
        u_ref, ud = u_new_ref, un
        x = (x + 0.1 * rng.standard_normal((nodes, d))).astype(np.float32)
    # in place, and the bias weights alone
    xd = dev(x)
    api.lpdt_pushsum_debias(nodes, d, xd, ud, dev(W), 0.8, un2 := torch.empty(nodes, device="cuda"), xd)
    u3, z3 = oracle.pushsum_debias(x, u_ref, W, 0.8)
    assert np.array_equal(xd.cpu().numpy(), z3) and np.array_equal(un2.cpu().numpy(), u3)
    api.lpdt_pushsum_debias(nodes, 0, None, ud, dev(W), 0.8, un3 := torch.empty(nodes, device="cuda"), None)
    assert np.array_equal(un3.cpu().numpy(), u3)


def test_sparse_push_chain():
    """Supplementary Algorithm 4 end to end on a directed graph: Deep-Squeeze mix (top-10 %) then push-sum
    de-biasing, against the same two oracle calls; total mass sum_i x_i / sum_i u_i is what z tracks."""
    rng = np.random.default_rng(44)
    nodes, d = 8, 5000
    W = directed_ring_matrix(nodes, rng)
    x = rng.standard_normal((nodes, d)).astype(np.float32)
    delta_ref = np.zeros((nodes, d), np.float32); u_ref = np.ones(nodes, np.float32)
    deltad, ud = dev(delta_ref), dev(u_ref)
    ws = ws_bytes(api.lpdt_gossip_mix_workspace_size(nodes, d, 1))
    for step in range(3):
        x_ref, delta_ref, _, _ = oracle.deepsqueeze_mix(x, delta_ref, W, 0.5, [0, d], [d // 10], 32)
        u_ref, z_ref = oracle.pushsum_debias(x_ref, u_ref, W, 0.5)
        xo = torch.empty(nodes, d, device="cuda"); un = torch.empty(nodes, device="cuda"); z = torch.empty_like(xo)
        api.lpdt_deepsqueeze_mix(nodes, d, dev(x), deltad, xo, dev(W), 0.5, [0, d], [d // 10], ws)
        api.lpdt_pushsum_debias(nodes, d, xo, ud, dev(W), 0.5, un, z)
        assert np.array_equal(deltad.cpu().numpy(), delta_ref)
        assert np.array_equal(un.cpu().numpy(), u_ref)
        close(z, z_ref)
        ud = un
        x = (z_ref - 0.05 * rng.standard_normal((nodes, d))).astype(np.float32)


def test_gossip_errors():
    t = torch.zeros(4, 8, device="cuda"); W = torch.zeros(4, 4, device="cuda")
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_gossip_mix(4, 8, t, t.clone(), t, W, 1.0, [0, 7], [7], ws_bytes(4096))   # segments don't tile
    assert e.value.code == 1
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_gossip_mix(4, 8, t, t, t, W, 1.0, [0, 8], [8], ws_bytes(4096))           # x_hat aliases x_half
    assert e.value.code == 1
    big = torch.zeros(65, 4, device="cuda")
    with pytest.raises(api.LpdtError) as e:
        api.lpdt_gossip_mix(65, 4, big, big.clone(), big.clone(), torch.zeros(65, 65, device="cuda"), 1.0, [0, 4], [4],
                            ws_bytes(65536))
    assert e.value.code == 2


# ------------------------------------------------------------------ glue
def test_glue_ops():
    rng = np.random.default_rng(8)
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    x = rng.standard_normal(10007).astype(np.float32); g = rng.standard_normal(10007).astype(np.float32)
    out = f(10007)
    api.lpdt_sgd_update(10007, dev(x), dev(g), 0.1, out)
    assert np.array_equal(out.cpu().numpy(), oracle.sgd_update(x, g, 0.1))
    a = rng.standard_normal((2, 3, 8, 8, 16)).astype(np.float32)
    r = rng.standard_normal((2, 3, 8, 8, 16)).astype(np.float32)
    y = f(*r.shape)
    api.lpdt_residual_add(2, 3, 8, 8, 16, 16, 1, 0, dev(r), dev(a), y)
    assert np.array_equal(y.cpu().numpy(), oracle.residual_add(r, a))
    r2 = rng.standard_normal((2, 3, 4, 4, 32)).astype(np.float32)
    y2 = f(*r2.shape)
    api.lpdt_residual_add(2, 3, 8, 8, 16, 32, 2, 8, dev(r2), dev(a), y2)
    assert np.array_equal(y2.cpu().numpy(), oracle.residual_add(r2, a, 2, 8))
    da = f(*a.shape)
    api.lpdt_residual_add_bwd(2, 3, 8, 8, 16, 32, 2, 8, dev(r2), dev(a), da)
    assert np.array_equal(da.cpu().numpy(), oracle.residual_add_bwd(r2, a, 2, 8))
    p = f(2, 3, 16)
    api.lpdt_avgpool(2, 3, 64, 16, dev(a), p)
    assert np.array_equal(p.cpu().numpy(), oracle.avgpool(a))
    dpx = f(*a.shape)
    api.lpdt_avgpool_bwd(2, 3, 64, 16, p, dpx)
    assert np.array_equal(dpx.cpu().numpy(), oracle.avgpool_bwd(oracle.avgpool(a), 8, 8))
    m_ref, i_ref = oracle.maxpool2x2(a)
    m = f(*m_ref.shape); idx = torch.empty(m_ref.shape, dtype=torch.int8, device="cuda")
    api.lpdt_maxpool2x2(2, 3, 8, 8, 16, dev(a), m, idx)
    assert np.array_equal(m.cpu().numpy(), m_ref) and np.array_equal(idx.cpu().numpy(), i_ref)
    dm = f(*a.shape)
    api.lpdt_maxpool2x2_bwd(2, 3, 8, 8, 16, m, idx, dm)
    assert np.array_equal(dm.cpu().numpy(), oracle.maxpool2x2_bwd(m_ref, i_ref, 8, 8))
    z = (3 * rng.standard_normal((3, 32, 10))).astype(np.float32)
    lab = rng.integers(0, 10, (3, 32)).astype(np.int32)
    loss_ref, dz_ref = oracle.softmax_ce(z, lab)
    loss = f(3); dz = f(3, 32, 10)
    api.lpdt_softmax_ce(3, 32, 10, dev(z), dev(lab), loss, dz)
    close(loss, loss_ref); close(dz, dz_ref, 1e-6, 1e-8)
    cs = torch.zeros(3, 14, device="cuda")
    api.lpdt_colsum(3, 32, 10, dev(z), cs[:, 4:], 14)
    close(cs[:, 4:], oracle.colsum(z), 1e-6, 1e-7)


@pytest.mark.parametrize("K", [1, 2, 4, 5, 16, 17, 32, 33])
@pytest.mark.parametrize("B", [1, 31, 33, 300])
def test_softmax_ce_widths(K, B):
    rng = np.random.default_rng(K + B)
    z = (3 * rng.standard_normal((2, B, K))).astype(np.float32)
    lab = rng.integers(0, K, (2, B)).astype(np.int32)
    loss_ref, dz_ref = oracle.softmax_ce(z, lab)
    loss, dz = torch.empty(2, device="cuda"), torch.full((2, B, K), 9.0, device="cuda")
    api.lpdt_softmax_ce(2, B, K, dev(z), dev(lab), loss, dz)
    close(loss, loss_ref); close(dz, dz_ref)


# both sides of the lines between a group of lanes and a thread per sample, groups of every size with ragged last turns
@pytest.mark.parametrize("K,B", [(2, 257), (3, 520), (5, 128), (8, 129), (8, 129 * 4), (9, 65), (16, 128), (16, 129), (16, 305), (20, 96),
                                 (24, 129), (32, 160), (32, 161), (32, 304)])
def test_softmax_ce_on_lanes_and_threads(K, B):
    test_softmax_ce_widths(K, B)


def test_softmax_ce_label_out_of_range_is_guarded():
    """A label outside [0, K) is never used as an index: the sample adds nothing to the loss, its gradient has
    no one-hot term, the status word reports the bad argument, and the other samples are untouched."""
    rng = np.random.default_rng(5)
    z = (2 * rng.standard_normal((2, 8, 10))).astype(np.float32)
    lab = rng.integers(0, 10, (2, 8)).astype(np.int32)
    bad = lab.copy(); bad[0, 3] = 10; bad[1, 0] = -1; bad[1, 7] = 2 ** 30
    loss_ref, dz_ref = oracle.softmax_ce(z, lab)
    f = lambda *sh: torch.empty(*sh, dtype=torch.float32, device="cuda")
    loss, dz = f(2), f(2, 8, 10)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    api.lpdt_softmax_ce(2, 8, 10, dev(z), dev(lab), loss, dz, status)
    assert api.lpdt_check_status(status) == 0
    close(loss, loss_ref); close(dz, dz_ref, 1e-6, 1e-8)
    api.lpdt_softmax_ce(2, 8, 10, dev(z), dev(bad), loss, dz, status)
    assert api.lpdt_check_status(status) == 1                      # LPDT_ERR_INVALID_ARG
    # expected values from the oracle on the valid labels: drop the bad samples' loss terms, undo their one-hot
    ok = (bad >= 0) & (bad < 10)
    per_sample = np.stack([[oracle.softmax_ce(z[n:n + 1, b:b + 1], lab[n:n + 1, b:b + 1])[0][0] for b in range(8)]
                           for n in range(2)])
    close(loss, (per_sample * ok).sum(1) / 8)
    dz_want = dz_ref.copy()
    for n, b in zip(*np.nonzero(~ok)):
        dz_want[n, b, lab[n, b]] += 1.0 / 8
    close(dz, dz_want, 1e-6, 1e-7)


def test_qconv_bwd_weight_empty_batch_writes_zeros():
    """B = 0: the gradient of no samples is zero (written, not left stale), as forward and backward-data
    return LPDT_OK for an empty batch."""
    for case in [(2, 0, 8, 8, 16, 16, 3, 3, 1, 1), (1, 0, 4, 4, 3, 5, 3, 3, 1, 1)]:
        desc = api.conv_desc(*case)
        nodes, _, H, W, Cin, Cout = case[:6]
        wn = Cout * 9 * Cin
        E = torch.empty(nodes, 0, H, W, Cout, dtype=torch.int8, device="cuda")
        A = torch.empty(nodes, 0, H, W, Cin, dtype=torch.int8, device="cuda")
        sc = torch.ones(nodes, device="cuda")
        dW = torch.full((nodes, wn), 7.0, device="cuda")
        dWacc = torch.full((nodes, wn), 7, dtype=torch.int32, device="cuda")
        ws = ws_bytes(api.lpdt_qconv_workspace_size(desc, 2))
        api.lpdt_qconv_bwd_weight(desc, E, sc, A, sc, dW=dW, dw_node_stride=wn, dWacc=dWacc, ws=ws)
        torch.cuda.synchronize()
        assert not dW.any() and not dWacc.any()


def test_bounded_wait_runs_out_and_reports():
    """The barrier wait of the tensor-core kernels with a 1 ms limit on a barrier nothing arrives at: the
    kernel returns, the status word holds LPDT_ERR_TIMEOUT, and the context stays usable."""
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    returned = torch.zeros(1, dtype=torch.int32, device="cuda")
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    api.lpdt_selftest_bounded_wait(1_000_000, status, returned)
    e1.record()
    assert api.lpdt_check_status(status) == 5                      # LPDT_ERR_TIMEOUT
    assert int(returned.item()) == 2
    ms = e0.elapsed_time(e1)
    assert 0.9 <= ms < 50.0, ms
    with pytest.raises(api.LpdtError):
        api.lpdt_selftest_bounded_wait(10 ** 9, status, returned)  # limits beyond 50 ms are refused on the host
    # the device is still healthy: an ordinary call runs and matches the oracle
    x = np.random.default_rng(0).standard_normal((2, 1000)).astype(np.float32)
    q = torch.empty(2, 1000, dtype=torch.int8, device="cuda"); s = torch.empty(2, device="cuda")
    api.lpdt_quantize(dev(x), 2, 1000, 1000, q, s, ws_bytes(api.lpdt_quantize_workspace_size(2)))
    q_ref, s_ref = oracle.quantize_sym_s8(x)
    assert np.array_equal(q.cpu().numpy(), q_ref) and np.array_equal(s.cpu().numpy(), s_ref)


def test_batched_reductions_equal_the_single_calls():
    """lpdt_range_evonorm_bwd_params_batch and lpdt_dequantize_acc_batch: many layers in one launch, bit-identical
    to the per-layer calls (which the tests above compare with the oracle)."""
    rng = np.random.default_rng(12)
    nodes, B = 3, 5
    layers = [(8, 8, 16, 4), (4, 4, 64, 8), (6, 5, 12, 3)]                   # H, W, C, groups
    stride = sum(3 * c for _, _, c, _ in layers) + 11
    G1 = torch.zeros(nodes, stride, device="cuda"); G2 = torch.zeros_like(G1)
    wss, offs, off = [], [], 3
    for H, W, C, groups in layers:
        x, P, dy = _ren_inputs((nodes, B, H, W, C, groups), seed=C)
        Pd, xd = dev(P), dev(x)
        f = lambda *sh: torch.empty(*sh, dtype=torch.float32, device="cuda")
        i = lambda *sh: torch.empty(*sh, dtype=torch.int32, device="cuda")
        y, gmin, gmax, amn, amx = f(*x.shape), f(nodes, B, groups), f(nodes, B, groups), i(nodes, B, groups), i(nodes, B, groups)
        api.lpdt_range_evonorm_fwd(nodes, B, H, W, C, groups, 1e-5, xd, Pd, Pd[:, C:], Pd[:, 2 * C:], P.shape[1], y, gmin,
                                   gmax, amn, amx)
        ws = ws_bytes(api.lpdt_range_evonorm_bwd_workspace_size(nodes, B, C))
        api.lpdt_range_evonorm_bwd(nodes, B, H, W, C, groups, 1e-5, dev(dy), xd, Pd, Pd[:, C:], P.shape[1], gmin, gmax, amn,
                                   amx, f(*x.shape), None, None, None, stride, ws)
        api.lpdt_range_evonorm_bwd_params(nodes, B, C, ws, G1[:, off:], G1[:, off + C:], G1[:, off + 2 * C:], stride)
        wss.append(ws); offs.append(off)
        off += 3 * C
    api.lpdt_range_evonorm_bwd_params_batch(nodes, B, [c for _, _, c, _ in layers], wss, offs, G2, stride)
    assert torch.equal(G1, G2) and G1.abs().sum() > 0
    # int32 sums of three tensors, each a contiguous [nodes][size] block, into one strided fp32 row per node
    sizes, acc_off, out_off = [432, 1000, 7], [0, 64 * 21, 64 * 21 + 64 * 47], [5, 600, 1700]
    acc = torch.from_numpy(rng.integers(-2 ** 31, 2 ** 31 - 1, 64 * 21 + 64 * 47 + 64, dtype=np.int64).astype(np.int32)).cuda()
    s1 = [dev(rng.uniform(0.001, 0.1, nodes).astype(np.float32)) for _ in sizes]
    s2 = [dev(rng.uniform(0.001, 0.1, nodes).astype(np.float32)) for _ in sizes]
    out = torch.zeros(nodes, 1800, device="cuda")
    api.lpdt_dequantize_acc_batch(acc, nodes, acc_off, sizes, out_off, s1, s2, out, 1800)
    want = np.zeros((nodes, 1800), np.float32)
    for t, n in enumerate(sizes):
        a = acc[acc_off[t]:acc_off[t] + nodes * n].cpu().numpy().reshape(nodes, 1, n)
        want[:, out_off[t]:out_off[t] + n] = oracle.dequant_acc(a, s1[t].cpu().numpy(), s2[t].cpu().numpy()).reshape(nodes, n)
    assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("cluster", ["1", "2", "8"])
def test_range_evonorm_cases_on_every_cluster_size(cluster):
    """The forward kernel splits a sample over 1-8 CTAs by a size rule; the cases are re-run in child
    processes with the cluster size forced (capped so that every CTA keeps a thread row)."""
    import os, subprocess, sys
    if os.environ.get("LPDT_CHILD") == "1":
        pytest.skip("already inside a child run")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    child_env = dict(os.environ, LPDT_CHILD="1", LPDT_REN_CLUSTER=cluster)
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(root, "tests", "test_gpu_ops.py"), "-m", "gpu",
                        "-q", "-x", "-k", "test_range_evonorm_fwd or test_fused_ranges"], env=child_env, cwd=root,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]


@pytest.mark.parametrize("cluster", ["2", "4"])
def test_range_evonorm_backward_cases_on_every_cluster_size(cluster):
    """The same for the backward kernel, which splits the samples of small batches over 2 or 4 CTAs."""
    import os, subprocess, sys
    if os.environ.get("LPDT_CHILD") == "1":
        pytest.skip("already inside a child run")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    child_env = dict(os.environ, LPDT_CHILD="1", LPDT_REN_BWD_CLUSTER=cluster)
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(root, "tests", "test_gpu_ops.py"), "-m", "gpu",
                        "-q", "-x", "-k", "test_range_evonorm_fwd or test_fused_ranges"], env=child_env,
                       cwd=root, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]


@pytest.mark.parametrize("env", [{"LPDT_FORCE_HALO": "1"}, {"LPDT_DISABLE_HALO": "1"}, {"LPDT_DISABLE_TC": "1"},
                                 {"LPDT_AFFINE_SEPARATE": "1"}, {"LPDT_PIX_DIRECT_STORE": "1", "LPDT_DISABLE_HALO": "1"},
                                 {"LPDT_PIX_TWO": "0", "LPDT_DISABLE_HALO": "1"}])
def test_qconv_cases_on_every_kernel_family(env):
    """The kernel choice is made once per process from the environment, so the contraction
    cases are re-run in child processes with the halo kernels forced, with the halo kernels
    off (general tensor-core kernels) and with the tensor-core engine off (CUDA-core kernels)."""
    import os, subprocess, sys
    if os.environ.get("LPDT_CHILD") == "1":
        pytest.skip("already inside a child run")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    child_env = dict(os.environ, LPDT_CHILD="1", **env)
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(root, "tests", "test_gpu_ops.py"), "-m", "gpu",
                        "-q", "-x", "-k", "test_qconv_all_three or test_qconv_extreme or test_qconv_fwd_affine or test_qconv_bwd_affine"], env=child_env, cwd=root,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-2000:]
