"""The extension module's call path against the ctypes one: same results, same objects handed back, same errors."""
import pytest
import torch

import paper_2509_21302_b200 as q
from paper_2509_21302_b200 import binding

pytestmark = pytest.mark.gpu


def _handles(K, N):
    g = torch.Generator(device="cuda").manual_seed(K + N)
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.02).bfloat16()
    b = (torch.randn(N, generator=g, device="cuda") * 0.01).bfloat16()
    c = torch.rand(K, generator=g, device="cuda") + 0.5
    return q.prepare_weights(W, b, c, None, c8=True), q.prepare_weights(W, b, c, None), g


def _calls(h, hp, x, g, K, N, given):
    """Every call of the fast path; `given`: the caller's own output tensors, or none."""
    M = x.shape[0]
    dev = dict(device="cuda")
    gamma, beta = torch.rand(K, generator=g, **dev), torch.rand(K, generator=g, **dev)
    delta, scratch = torch.tensor([0.2], **dev), torch.empty(N * K + 16, dtype=torch.int8, **dev)

    def outs(codes, scales):
        return (torch.empty(M, codes, dtype=torch.uint8 if codes < K else torch.int8, **dev), torch.empty((M, scales) if scales else (M,), **dev)) if given else (None, None)

    y = (lambda: torch.empty(M, N + 8, dtype=torch.bfloat16, **dev)[:, :N]) if given else (lambda: None)
    res = []
    for f, lin, o in (
            (lambda a, b: q.rotate_smooth_quantize(h, x, 0, a, b), lambda c, s: q.w4a4_linear(h, c, s, 0, y()), outs(K // 2, 0)),
            (lambda a, b: q.rotate_smooth_quantize(h, x, 128, a, b), lambda c, s: q.w4a4_linear(h, c, s, 128, y()), outs(K // 2, K // 128)),
            (lambda a, b: q.rotate_smooth_quantize_c8(h, x, a, b), lambda c, s: q.w4a4_linear_c8(h, c, s, y()), outs(K, 0)),
            (lambda a, b: q.rotate_smooth_quantize_c8(hp, x, a, b), lambda c, s: q.w4a4_linear_c8_packed_weights(hp, c, s, scratch, y()), outs(K, 0)),
            (lambda a, b: q.rotate_smooth_quantize_c8_expand(hp, x, scratch, a, b), lambda c, s: q.w4a4_linear_c8_expanded(hp, c, s, scratch, y()), outs(K, 0)),
            (lambda a, b: q.rotate_smooth_quantize_c8_grouped(h, x, a, b), lambda c, s: q.w4a4_linear_c8_grouped(h, c, s, y()), outs(K, K // 128)),
            (lambda a, b: q.rotate_smooth_quantize_static_c8(h, x, delta, a, b), None, outs(K, 0)),
            (lambda a, b: q.layernorm_rotate_smooth_quantize_c8(h, x, gamma, beta, 1e-5, a, b), None, outs(K, 0)),
            (lambda a, b: q.gelu_rotate_smooth_quantize_c8(h, x, a, b), None, outs(K, 0)),
            (lambda a, b: q.rotate_smooth_quantize_tc(h, x, True, a, b), None, outs(K, 0)),
            (lambda a, b: q.rotate_smooth_quantize_tc(h, x, False, a, b), None, outs(K // 2, 0))):
        c, s = f(*o)
        if given:
            assert c is o[0] and s is o[1]
        res += [c, s]
        if lin is not None:
            res.append(lin(c, s))
    return res


@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("K,N,M,pad", [(1024, 256, 1, 0), (1024, 256, 131, 64), (4096, 128, 3, 8), (1024, 128, 0, 0)])
def test_same_results_as_through_ctypes(K, N, M, pad, given, monkeypatch):
    h, hp, g = _handles(K, N)
    x = torch.randn(M, K + pad, generator=g, device="cuda").bfloat16()[:, :K]
    st = g.get_state()
    fast = _calls(h, hp, x, g, K, N, given)
    g.set_state(st)
    monkeypatch.setattr(binding, "_fast", None)
    slow = _calls(h, hp, x, g, K, N, given)
    monkeypatch.undo()
    assert len(fast) == len(slow)
    for a, b in zip(fast, slow):
        assert a.shape == b.shape and a.dtype == b.dtype and a.stride() == b.stride() and a.device == b.device and torch.equal(a, b)


def test_same_errors_as_through_ctypes():
    K, N, M = 1024, 128, 5
    h, hp, g = _handles(K, N)
    x = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    xq, a = q.rotate_smooth_quantize_c8(h, x)
    for bad in (lambda: q.rotate_smooth_quantize_c8(h, x.float()), lambda: q.rotate_smooth_quantize_c8(h, x.cpu()), lambda: q.rotate_smooth_quantize_c8(h, x[:, :512]),
                lambda: q.rotate_smooth_quantize_c8(h, x, xq.view(torch.uint8), a), lambda: q.w4a4_linear_c8(h, xq[:, ::2], a),
                lambda: q.w4a4_linear_c8(h, xq, a.double()), lambda: q.w4a4_linear_c8(h, xq, a, torch.empty(M, N + 1, device="cuda").bfloat16())):
        with pytest.raises(AssertionError):
            bad()
    with pytest.raises(q.QvggtError) as e:        # no one-code-per-byte copy in this handle
        q.w4a4_linear_c8(hp, xq, a)
    assert e.value.status == -4
    with pytest.raises(q.QvggtError) as e:        # row stride not a multiple of 8
        q.rotate_smooth_quantize_c8(h, torch.empty(M, K + 4, device="cuda").bfloat16()[:, :K])
    assert e.value.status == -3
    h.free()
    with pytest.raises(RuntimeError):
        q.rotate_smooth_quantize_c8(h, x)


def test_preparation_calls_give_the_same_and_refuse_the_same(monkeypatch):
    K, N = 1024, 256
    g = torch.Generator(device="cuda").manual_seed(5)
    W = (torch.randn(N, K, generator=g, device="cuda") * 0.02).bfloat16()
    b, X = torch.randn(N, generator=g, device="cuda").bfloat16(), torch.randn(37, K, generator=g, device="cuda").bfloat16()
    v = (torch.randint(0, 2, (K,), generator=g, device="cuda") * 2 - 1).to(torch.int8)

    def run():
        c = q.calibrate_smooth(X, W, 0.5, 0.02, 50.0)
        out = [c]
        for bias, sign, c8, bits in ((b, None, True, 4), (None, v, "only", 4), (b, v, False, 4), (b, None, False, 8)):
            h = q.prepare_weights(W, bias, c, sign, c8=c8, bits=bits)
            view = h.view()
            out += [view["wq"], view["w_scale"], view["amul"], view["bias"], h.view_c8()]
            assert h.bits == bits
            h.free()
        return out

    fast = run()
    lib = binding._fast

    class OnlyViews:                      # the other calls through ctypes
        weights_view, weights_view_c8 = staticmethod(lib.weights_view), staticmethod(lib.weights_view_c8)
        calibrate_smooth = prepare_weights = staticmethod(lambda *a: None)

    monkeypatch.setattr(binding, "_fast", OnlyViews)
    slow = run()
    monkeypatch.undo()
    for a, s in zip(fast, slow):
        assert (a is None) == (s is None) and (a is None or (a.dtype == s.dtype and torch.equal(a, s)))
    for bad in (lambda: q.calibrate_smooth(X, W.float()), lambda: q.calibrate_smooth(X[:, ::2], W), lambda: q.prepare_weights(W.float(), None, fast[0]),
                lambda: q.prepare_weights(W, b[:5], fast[0]), lambda: q.prepare_weights(W, None, fast[0][:5]), lambda: q.prepare_weights(W, None, fast[0], v.float())):
        with pytest.raises(AssertionError):
            bad()
    with pytest.raises(q.QvggtError) as e:
        q.prepare_weights(W[:100], None, fast[0])
    assert e.value.status == -2


def test_group_scales_of_another_shape_are_refused():
    """[M, K/128] and nothing else that holds as many values: transposed scales or those of a larger batch give no result."""
    K, N, M = 1024, 128, 5
    h, hp, g = _handles(K, N)
    x = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    xq, a = q.rotate_smooth_quantize_c8_grouped(h, x)
    for bad in (a.t().contiguous(), a.reshape(-1), a.reshape(1, M, K // 128), torch.cat([a, a]), torch.cat([a, a], 1)):
        with pytest.raises(AssertionError):
            q.w4a4_linear_c8_grouped(h, xq, bad)
    for keep in (a, a.clone()):
        q.w4a4_linear_c8_grouped(h, xq, keep)


def test_a_view_that_cannot_be_copied_says_why():
    """Out of memory is out of memory, not a status of the library."""
    h, hp, g = _handles(1024, 4096)
    torch.cuda.empty_cache()
    total, used = torch.cuda.get_device_properties(0).total_memory, torch.cuda.memory_reserved()
    torch.cuda.set_per_process_memory_fraction(used / total)
    try:
        for view in (h.view, h.view_c8):
            with pytest.raises(torch.cuda.OutOfMemoryError):
                view()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert h.view()["wq"].shape == (4096, 512) and h.view_c8().shape == (4096, 1024)


@pytest.mark.skipif(torch.cuda.device_count() < 2, reason="needs two devices")
def test_a_handle_of_another_device_can_be_viewed():
    h, hp, g = _handles(1024, 128)
    want, codes = h.view(), h.view_c8()
    torch.cuda.synchronize()
    with torch.cuda.device(1):
        got, other = h.view(), h.view_c8()
        for k, v in got.items():
            assert v.device.index == 1 and torch.equal(v.cpu(), want[k].cpu())
        assert other.device.index == 1 and torch.equal(other.cpu(), codes.cpu())


def test_a_tensor_without_memory_of_its_own_is_refused():
    """A tensor whose address cannot be asked for (one inside vmap) among real ones, in every place: an exception, and no harm to the
    interpreter."""
    K, N, M = 1024, 128, 3
    h, hp, g = _handles(K, N)
    x = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    gamma, beta = torch.rand(K, generator=g, device="cuda"), torch.rand(K, generator=g, device="cuda")
    xq, a = q.rotate_smooth_quantize_c8(h, x)
    scratch, delta = torch.empty(N * K, dtype=torch.int8, device="cuda"), torch.tensor([0.2], device="cuda")
    for f, t in ((lambda v: q.rotate_smooth_quantize_c8(h, v), x), (lambda v: q.layernorm_rotate_smooth_quantize_c8(h, x, v, beta), gamma),
                 (lambda v: q.layernorm_rotate_smooth_quantize_c8(h, x, gamma, v), beta), (lambda v: q.rotate_smooth_quantize_static_c8(h, x, v), delta),
                 (lambda v: q.rotate_smooth_quantize_c8_expand(hp, x, v), scratch), (lambda v: q.w4a4_linear_c8(h, v, a), xq),
                 (lambda v: q.w4a4_linear_c8(h, xq, v), a), (lambda v: q.w4a4_linear_c8_packed_weights(hp, xq, a, v), scratch),
                 (lambda v: q.w4a4_linear_c8_expanded(hp, xq, a, v), scratch), (lambda v: q.calibrate_smooth(x, v), x),
                 (lambda v: q.prepare_weights(x.repeat(128, 1)[:128], None, v), gamma)):
        with pytest.raises(Exception):
            torch.func.vmap(f)(torch.stack([t, t]))
    want = q.w4a4_linear_c8(h, xq, a)
    assert torch.equal(want, q.w4a4_linear_c8(h, xq, a)) and h.device_status() == 0
