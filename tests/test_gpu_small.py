"""The few-rows GEMM on both sides of every line its launch rule draws, and of its tiles of 8, 16 and 32 rows: exact sums, bit-equal
outputs, for every storage format and scale granularity, and nothing written outside the rows of the result."""
import numpy as np
import pytest
import torch

import oracle
import paper_2509_21302_b200 as q
import workload
from _util import dev_bf16, host_bits

pytestmark = pytest.mark.gpu


def _check(K, N, M, bits=4, with_bias=True, pad=8):
    rng = np.random.default_rng(K + 7 * N + M)
    spec = workload.LinearSpec("s", K, N, workload.DIST_NORMAL, 90, 0)
    W, b = spec.weight(), spec.bias()
    c = oracle.smooth_factors(spec.x_calib(16), W)
    prep = oracle.prepare_weights(W, c, None, bits)
    dev = (dev_bf16(W), dev_bf16(b) if with_bias else None, torch.from_numpy(c).cuda(), None)
    top = 2 ** (bits - 1) - 1
    xq = rng.integers(-top, top + 1, (M, K)).astype(np.int8)
    xq[0] = top                                        # the largest sums
    X8, G = torch.from_numpy(xq).cuda(), K // 128
    a = (rng.random((M,)) + 0.5).astype(np.float32) * 1e-2
    ag = (rng.random((M, G)) + 0.5).astype(np.float32) * 1e-2
    bias = b if with_bias else None
    acc = oracle.gemm_i32(xq, prep["wq"])
    want = oracle.epilogue(acc, a, prep["w_scale"], bias)

    def run(f):
        Y = torch.full((M + 2, N + pad), 7.0, dtype=torch.bfloat16, device="cuda")
        f(Y[1:M + 1, :N])
        assert torch.all(Y[0] == 7) and torch.all(Y[M + 1] == 7) and torch.all(Y[:, N:] == 7)
        return host_bits(Y[1:M + 1, :N])

    A = torch.from_numpy(a).cuda()
    h = q.prepare_weights(*dev, c8=True, bits=bits)
    assert np.array_equal(run(lambda y: q.w4a4_linear_c8(h, X8, A, y)), want)
    if bits == 4:
        AG, XP = torch.from_numpy(ag).cuda(), torch.from_numpy(oracle.pack_int4(xq)).cuda()
        want_g = oracle.epilogue(oracle.gemm_i32(xq, prep["wq"], 128), ag, prep["w_scale"], bias)
        scratch = torch.empty(N * K, dtype=torch.int8, device="cuda")
        assert np.array_equal(run(lambda y: q.w4a4_linear_c8_packed_weights(h, X8, A, scratch, y)), want)
        assert np.array_equal(run(lambda y: q.w4a4_linear_c8_expanded(h, X8, A, scratch, y)), want)
        assert np.array_equal(run(lambda y: q.w4a4_linear(h, XP, A, 0, y)), want)
        assert np.array_equal(run(lambda y: q.w4a4_linear_c8_grouped(h, X8, AG, y)), want_g)
        assert np.array_equal(run(lambda y: q.w4a4_linear(h, XP, AG, 128, y)), want_g)
    assert h.device_status() == 0
    h.free()


@pytest.mark.parametrize("M", [1, 2, 7, 8, 9, 16, 17, 31, 32, 33, 40, 65])
@pytest.mark.parametrize("K,N", [(1024, 128), (4096, 256)])
def test_row_tiles(K, N, M):
    _check(K, N, M, with_bias=M % 2 == 1)


# M on the last size of the kernel and the first of the other one, for each of the rule's lines
@pytest.mark.parametrize("K,N,lines", [(1024, 1024, (192, 384, 768)), (1024, 3072, (64, 128, 256)), (4096, 1024, (96, 128, 144, 192, 384)),
                                         (4096, 512, (192, 288, 768)), (1024, 1024, (96,)), (1024, 512, (192,)), (4096, 512, (160,)), (4096, 640, (153,))])
def test_both_sides_of_the_rule(K, N, lines):
    for line in lines:
        for M in (line, line + 1):
            _check(K, N, M)


@pytest.mark.parametrize("K,N,M", [(1024, 128, 1), (1024, 384, 33), (4096, 128, 9), (4096, 384, 100)])
def test_eight_bit_codes(K, N, M):
    _check(K, N, M, bits=8)


def test_weights_prepared_just_before():
    """Preparing, quantizing and multiplying back to back, without anything in between, on fresh handles: every launch may start
    while its predecessor drains."""
    K, N, M = 1024, 4096, 5
    g = torch.Generator(device="cuda").manual_seed(1)
    W = [(torch.randn(N, K, generator=g, device="cuda") * 0.02).bfloat16() for _ in range(4)]
    x, c = torch.randn(M, K, generator=g, device="cuda").bfloat16(), torch.rand(K, generator=g, device="cuda") + 0.5

    def run(i, wait):
        h = q.prepare_weights(W[i], None, c, None, c8="only")
        if wait:
            torch.cuda.synchronize()
        xq, a = q.rotate_smooth_quantize_c8(h, x)
        if wait:
            torch.cuda.synchronize()
        return h, q.w4a4_linear_c8(h, xq, a)

    want = [run(i, True)[1].clone() for i in range(4)]
    torch.cuda.synchronize()
    for rep in range(10):
        got = [run(i, False) for i in range(4)]
        for (h, y), w in zip(got, want):
            assert torch.equal(y.view(torch.int16), w.view(torch.int16))
            h.free()


# M on both sides of the few-rows line; an offset of 4 floats is a 16-byte boundary again
@pytest.mark.parametrize("off", [1, 2, 3, 4])
@pytest.mark.parametrize("K,N,M", [(1024, 1024, 384), (1024, 1024, 385), (4096, 1024, 144), (4096, 1024, 145), (4096, 1024, 193)])
def test_group_scales_on_any_float_boundary(K, N, M, off):
    """Scales that are a contiguous view into a larger buffer need only be aligned to 4 bytes, whatever M: quantizing into such a view
    and multiplying from it gives the bits of aligned scales, and nothing beside the view is written."""
    g = torch.Generator(device="cuda").manual_seed(K + M)
    W, x = (torch.randn(N, K, generator=g, device="cuda") * 0.02).bfloat16(), torch.randn(M, K, generator=g, device="cuda").bfloat16()
    h = q.prepare_weights(W, None, torch.rand(K, generator=g, device="cuda") + 0.5, None, c8=True)
    G = K // 128
    buf = torch.full((M * G + 8,), 7.0, device="cuda")
    a = buf[off:off + M * G].view(M, G)
    assert a.is_contiguous() and a.data_ptr() % 16 == 4 * off % 16
    xq, aligned = q.rotate_smooth_quantize_c8_grouped(h, x)
    xq2, a2 = q.rotate_smooth_quantize_c8_grouped(h, x, None, a)
    assert a2 is a and torch.equal(xq, xq2) and torch.equal(a, aligned)
    assert torch.all(buf[:off] == 7) and torch.all(buf[off + M * G:] == 7)
    want = q.w4a4_linear_c8_grouped(h, xq, aligned)
    assert torch.equal(q.w4a4_linear_c8_grouped(h, xq, a).view(torch.int16), want.view(torch.int16))
    packed, _ = q.rotate_smooth_quantize(h, x, 128)
    assert torch.equal(q.w4a4_linear(h, packed, a, 128).view(torch.int16), want.view(torch.int16))
    assert h.device_status() == 0
    h.free()
