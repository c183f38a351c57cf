"""Fake quantisation for quantisation-aware training on the GPU (App. B "PTQ
and QAT": Eq. quant with a learnable scale, symmetric or min-max with offset):
forward values and codes bit-exact against the oracle, the straight-through
gradient exact and the scale / offset gradients to fp64 summation order, and
the QAT forward of a linear bit-exact against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2306_04235_gb300 import mnmt, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def host(t):
    torch.cuda.synchronize()
    return t.cpu().numpy()


def _x(seed, n, scale):
    return (synth.Stream(seed, "gfq").normal(n) * scale).astype(np.float32)


@pytest.mark.parametrize("bits,minmax", [(8, False), (4, False), (2, False), (8, True), (4, True)])
@pytest.mark.parametrize("n", [1, 1000, 1 << 20])
def test_fake_quant_forward_and_backward(bits, minmax, n):
    s, r = np.float32(0.03125 * 1.37), np.float32(-0.2)
    x = _x(n + bits, n, 0.6)
    g = _x(n + 7, n, 1.0)
    y = torch.empty(n, dtype=torch.float32, device="cuda")
    q = torch.empty(n, dtype=torch.int32, device="cuda")
    dx, dg = dev(x), dev(g)
    mnmt.mnmt_fake_quant(dx, n, s, r, bits, minmax, y, q)
    ry, rq = O.fake_quant(x, s, bits, r, minmax)
    assert np.array_equal(host(y).view(np.uint32), ry.view(np.uint32))
    assert np.array_equal(host(q), rq)
    gx = torch.empty(n, dtype=torch.float32, device="cuda")
    gs = torch.empty(1, dtype=torch.float64, device="cuda")
    gr = torch.empty(1, dtype=torch.float64, device="cuda")
    mnmt.mnmt_fake_quant_backward(dx, dg, n, s, gx, gs, gr, r, bits, minmax)
    rgx, rgs, rgr = O.fake_quant_backward(x, g, s, bits, r, minmax)
    assert np.array_equal(host(gx).view(np.uint32), rgx.view(np.uint32))
    scale = float(np.sum(np.abs(g.astype(np.float64)))) * (2 ** bits) + 1.0
    assert abs(float(host(gs)[0]) - rgs) <= 1e-13 * scale
    assert abs(float(host(gr)[0]) - rgr) <= 1e-13 * scale


@pytest.mark.parametrize("M,N,K", [(1, 1024, 256), (5, 300, 512), (40, 768, 256), (130, 512, 1024)])
@pytest.mark.parametrize("wbits", [8, 4])
def test_fake_quant_linear_matches_oracle(M, N, K, wbits):
    X = _x(M * 3 + K, M * K, 0.7).reshape(M, K)
    W = synth.weight_draw(synth.Stream(N, "w"), N, K, 0.05).astype(np.float32)
    qmax = 2 ** (wbits - 1) - 1
    s_w = (np.abs(W).max(axis=1) / qmax * 1.1).astype(np.float32)     # learnable scales: any positive values
    s_x = np.float32(3.5 / 127)
    b = synth.uniform_f32(M, "b", (N,), -0.2, 0.2)
    ws = torch.empty(((M * K + 15) // 16) * 16 + N * K, dtype=torch.int8, device="cuda")
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    mnmt.mnmt_fake_quant_linear(dev(X), dev(W), s_x, dev(s_w), dev(b), M, N, K, wbits, ws, y)
    ref = O.fake_quant_linear(X, W, s_x, s_w, b, wbits)
    assert np.array_equal(host(y).view(np.uint32), ref.view(np.uint32))


def test_fake_quant_rejects_bad_scale():
    x = torch.zeros(4, dtype=torch.float32, device="cuda")
    with pytest.raises(mnmt.MnmtError) as ei:
        mnmt.mnmt_fake_quant(x, 4, 0.0, y=x)
    assert ei.value.code == mnmt.EINVAL


@pytest.mark.parametrize("scale_g", [1.0, 1e-30, 1e-42, 1e37])
@pytest.mark.parametrize("off,n", [(0, 4099), (1, 4099), (0, 7), (0, 1 << 16)])
def test_fake_quant_backward_pair_sums(scale_g, off, n):
    """The scale gradient's groups of eight: products inside the range of the
    exact fp32 pairs, below and above it (summed in fp64), all-zero groups,
    remainders and unaligned arrays.  Bound: fp64 addition of n terms."""
    s = np.float32(0.041)
    x, g = _x(n + off, n + off, 0.6), (_x(n + 5, n + off, 1.0) * np.float32(scale_g)).astype(np.float32)
    x[off + 3::97] = 0.0
    x[off + 5::31] = np.float32(9.0)     # clamped
    g[off: off + 40] = 0.0
    dx, dg = dev(x)[off:], dev(g)[off:]
    gx, y = torch.empty(n + off, dtype=torch.float32, device="cuda")[off:], torch.empty(n + off, dtype=torch.float32, device="cuda")[off:]
    gs = torch.empty(1, dtype=torch.float64, device="cuda")
    mnmt.mnmt_fake_quant(dx, n, s, 0.0, 8, False, y)
    mnmt.mnmt_fake_quant_backward(dx, dg, n, s, gx, gs)
    rgx, rgs, _ = O.fake_quant_backward(x[off:], g[off:], s, 8, 0.0, False)
    ry, _ = O.fake_quant(x[off:], s, 8, 0.0, False)
    assert np.array_equal(host(y).view(np.uint32), ry.view(np.uint32))
    assert np.array_equal(host(gx).view(np.uint32), rgx.view(np.uint32))
    terms = np.abs(g[off:].astype(np.float64)) * 127
    assert abs(float(host(gs)[0]) - rgs) <= n * 2.0 ** -53 * float(terms.sum())


def test_fake_quant_backward_non_finite():
    """An infinite or NaN gradient reaches the scale gradient as in fp64."""
    n = 64
    x = _x(1, n, 0.6)
    x[9], x[11] = 0.3, 0.31
    for bad in (np.inf, np.nan):
        g = np.ones(n, np.float32)
        g[9] = bad
        gx = torch.empty(n, dtype=torch.float32, device="cuda")
        gs = torch.empty(1, dtype=torch.float64, device="cuda")
        mnmt.mnmt_fake_quant_backward(dev(x), dev(g), n, 0.041, gx, gs)
        rgx, rgs, _ = O.fake_quant_backward(x, g, np.float32(0.041), 8, 0.0, False)
        assert np.array_equal(host(gx).view(np.uint32), rgx.view(np.uint32))
        assert np.array_equal(np.array([float(host(gs)[0])]), np.array([rgs]), equal_nan=True)


@pytest.mark.parametrize("n", [4095, 4096, 32767, 32769, 262143, 262145])
@pytest.mark.parametrize("minmax", [False, True])
@pytest.mark.parametrize("off", [0, 1])
def test_fake_quant_group_limits(n, minmax, off):
    """Both sides of the sizes from which elements are taken in groups, aligned
    and not.  Bound of the sums: fp64 addition of n terms."""
    s, r = np.float32(0.041), np.float32(-1.7) if minmax else np.float32(0)
    x, g = _x(n, n + off, 0.6), _x(n + 3, n + off, 1.0)
    dx, dg = dev(x)[off:], dev(g)[off:]
    y, gx = (torch.empty(n + off, dtype=torch.float32, device="cuda")[off:] for _ in range(2))
    codes = torch.empty(n + off, dtype=torch.int32, device="cuda")[off:]
    gs, gr = (torch.empty(1, dtype=torch.float64, device="cuda") for _ in range(2))
    mnmt.mnmt_fake_quant(dx, n, s, r, 4, minmax, y, codes)
    mnmt.mnmt_fake_quant_backward(dx, dg, n, s, gx, gs, gr, r, 4, minmax)
    ry, rq = O.fake_quant(x[off:], s, 4, r, minmax)
    rgx, rgs, rgr = O.fake_quant_backward(x[off:], g[off:], s, 4, r, minmax)
    assert np.array_equal(host(y).view(np.uint32), ry.view(np.uint32)) and np.array_equal(host(codes), rq)
    assert np.array_equal(host(gx).view(np.uint32), rgx.view(np.uint32))
    bound = n * 2.0 ** -53 * float(np.abs(g[off:].astype(np.float64)).sum()) * 15
    assert abs(float(host(gs)[0]) - rgs) <= bound and abs(float(host(gr)[0]) - rgr) <= bound
