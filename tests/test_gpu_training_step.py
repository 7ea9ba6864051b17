"""The three GEMMs of a training step in use: a dense layer whose forward, backward-data and
backward-weight products run through the library (weights in wide storage, updated in place), checked
product by product against the oracle, and a small classifier on synthetic data trained with it beside
the same model in FP32 (the paper's claim, Sec. 6: HBFP follows the FP32 training curve)."""
import numpy as np
import pytest

import oracle
from tests.helpers import dgrad_filters_view, ofmt

pytestmark = pytest.mark.gpu

TOL = 1e-6


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_1804_01526_b200 import autograd as hbfp_nn, binding
    binding.lib()
    return torch, hbfp_nn, binding


def fmt_dict(f):
    return dict(mant_bits=f.mant_bits, block=f.block, tile=f.tile, rounding=f.rounding, seed=f.seed, stream_id=f.stream_id)


def test_layer_products_match_the_oracle(env):
    torch, hbfp_nn, hb = env
    torch.manual_seed(0)
    batch, fin, fout, t = 96, 200, 136, 24
    layer = hbfp_nn.HbfpLinear(fin, fout, mant_bits=8, tile=t, rounding=1, seed=5, stream_id=10, batch_block=32)
    x = torch.randn(batch, fin, device="cuda").relu().requires_grad_(True)
    y = layer(x)
    dy = torch.randn(batch, fout, device="cuda") * 1e-3
    y.backward(dy)
    assert hb.device_status() == 0
    # the narrow copy the layer multiplied by, from its wide storage
    q16, g16 = layer.wide.mant.cpu().numpy(), layer.wide.exps.cpu().numpy()
    s16 = np.repeat(g16, t, axis=0)[:fin, :]
    qm, sm = oracle.wide_narrow(q16, s16, 8)
    grid = sm[::t, :]
    X, dY = x.detach().cpu().numpy(), dy.cpu().numpy()
    # forward
    qx, sx = oracle.quantize(X, 1, ofmt(fmt_dict(layer.fmt_act(0))))
    ref = oracle.gemm(qx, sx, np.ascontiguousarray(qm.T), np.ascontiguousarray(np.repeat(grid.T, t, axis=0)[:fout, :]), t)
    Y = (y - layer.bias).detach().cpu().numpy()
    assert (np.abs(Y.astype(np.float64) - ref["c_ref"]) <= TOL * ref["a_mag"] + 1e-12).all()
    # backward-data
    qd, sd = oracle.quantize(dY, 1, ofmt(fmt_dict(layer.fmt_act(2))))
    ref = oracle.gemm(qd, sd, qm, sm, t)
    assert (np.abs(x.grad.cpu().numpy().astype(np.float64) - ref["c_ref"]) <= TOL * ref["a_mag"]).all()
    # backward-weight: X^T dY with blocks along the batch axis
    ref = oracle.hbfp_gemm(1, 0, X, dY, ofmt(fmt_dict(layer.fmt_act(0, batch_axis=True))),
                           ofmt(fmt_dict(layer.fmt_act(2, batch_axis=True))))
    assert (np.abs(layer.weight.grad.cpu().numpy().astype(np.float64) - ref["c_ref"]) <= TOL * ref["a_mag"]).all()
    # and the update lands in wide storage as the oracle computes it
    delta = (-0.1 * layer.weight.grad).contiguous()
    layer.apply_update(delta)
    q2, s2 = oracle.wide_update(q16, s16, delta.cpu().numpy(), ofmt(fmt_dict(layer.fmt_weight())))
    assert np.array_equal(layer.wide.mant.cpu().numpy(), q2)
    assert np.array_equal(layer.wide.exps.cpu().numpy(), s2[::t, :])


def test_small_classifier_trains_like_fp32(env):
    torch, hbfp_nn, hb = env
    torch.manual_seed(1)
    n_cls, fin, hid, batch, steps, lr = 10, 64, 128, 128, 80, 0.2
    centers = torch.randn(n_cls, fin, device="cuda") * 1.5
    gen = torch.Generator(device="cuda").manual_seed(2)

    def draw():
        labels = torch.randint(0, n_cls, (batch,), device="cuda", generator=gen)
        return centers[labels] + torch.randn(batch, fin, device="cuda", generator=gen), labels

    l1 = hbfp_nn.HbfpLinear(fin, hid, mant_bits=8, tile=24, rounding=1, seed=3, stream_id=0)
    l2 = hbfp_nn.HbfpLinear(hid, n_cls, mant_bits=8, tile=24, rounding=1, seed=3, stream_id=10)
    # the FP32 twin starts from the same (wide-representable) weights
    w1 = l1.weight.detach().clone().requires_grad_(True)
    w2 = l2.weight.detach().clone().requires_grad_(True)
    b1 = torch.zeros(hid, device="cuda", requires_grad=True)
    b2 = torch.zeros(n_cls, device="cuda", requires_grad=True)
    loss_fn = torch.nn.CrossEntropyLoss()
    hist_h, hist_f = [], []
    for _ in range(steps):
        x, labels = draw()
        loss_h = loss_fn(l2(torch.relu(l1(x))), labels)
        for p in (l1.weight, l1.bias, l2.weight, l2.bias):
            p.grad = None
        loss_h.backward()
        with torch.no_grad():
            for layer in (l1, l2):
                layer.apply_update(-lr * layer.weight.grad)          # FP32 optimiser arithmetic, BFP weight storage
                layer.bias -= lr * layer.bias.grad
        loss_f = loss_fn(torch.relu(x @ w1 + b1) @ w2 + b2, labels)
        for p in (w1, b1, w2, b2):
            p.grad = None
        loss_f.backward()
        with torch.no_grad():
            for p in (w1, b1, w2, b2):
                p -= lr * p.grad
        hist_h.append(float(loss_h.detach()))
        hist_f.append(float(loss_f.detach()))
    assert hb.device_status() == 0
    first, last_h, last_f = np.mean(hist_h[:5]), np.mean(hist_h[-10:]), np.mean(hist_f[-10:])
    assert last_h < 0.5 * first, (first, last_h)                     # it learns
    assert abs(last_h - last_f) <= 0.15 * max(last_f, 0.05), (last_h, last_f)   # and follows the FP32 curve


def test_convolution_layer_products_match_the_oracle_and_fp32(env):
    torch, hbfp_nn, hb = env
    torch.manual_seed(2)
    n, hw, c, f = 2, 16, 64, 64
    layer = hbfp_nn.HbfpConv3x3(c, f, mant_bits=8, pixel_block=64)
    x = torch.randn(n, hw, hw, c, device="cuda").relu().requires_grad_(True)
    y = layer(x)
    dy = torch.randn(n, hw, hw, f, device="cuda") * 1e-2
    y.backward(dy)
    assert hb.device_status() == 0
    t = c
    q16, g16 = layer.wide.mant.cpu().numpy(), layer.wide.exps.cpu().numpy()
    s16 = np.repeat(g16, t, axis=0)[: 9 * c, :]
    qm, sm = oracle.wide_narrow(q16, s16, 8)
    grid = sm[::t, :]
    X, dY = x.detach().cpu().numpy(), dy.cpu().numpy().reshape(n * hw * hw, f)
    cols = oracle.im2col(X, 3, 3, 1)
    fa = dict(mant_bits=8, block=c, rounding=0, seed=0)
    # forward
    qx, sx = oracle.quantize(cols, 1, ofmt(fa))
    ref = oracle.gemm(qx, sx, np.ascontiguousarray(qm.T), np.ascontiguousarray(np.repeat(grid.T, t, axis=0)[:f, :]), t)
    Y = y.detach().cpu().numpy().reshape(n * hw * hw, f)
    assert (np.abs(Y.astype(np.float64) - ref["c_ref"]) <= TOL * ref["a_mag"] + 1e-12).all()
    # backward-weight
    fb = dict(mant_bits=8, block=64, rounding=0, seed=0)
    ref = oracle.hbfp_gemm(1, 0, cols, dY, ofmt(fb), ofmt(fb))
    assert (np.abs(layer.weight.grad.cpu().numpy().astype(np.float64) - ref["c_ref"]) <= TOL * ref["a_mag"]).all()
    # backward-data: the GEMM against the oracle, the scatter against torch's own convolution gradient
    qd, sd = oracle.quantize(dY, 1, ofmt(fa))
    ref = oracle.gemm(qd, sd, qm, sm, t)                         # gradient of the im2col matrix [pixels][9 c]
    dcols = ref["c_ref"].reshape(n, hw, hw, 3, 3, c)
    dxp = np.zeros((n, hw + 2, hw + 2, c))
    for i in range(3):
        for j in range(3):
            dxp[:, i:i + hw, j:j + hw, :] += dcols[:, :, :, i, j, :]
    dx_ref = dxp[:, 1:hw + 1, 1:hw + 1, :]
    assert np.allclose(x.grad.cpu().numpy(), dx_ref, rtol=1e-4, atol=1e-6)
    # ... computed as the convolution of the packed gradient with the regrouped forward weights: bit for bit the
    # oracle's GEMM on the gathered quantised gradient, taps in that operand's order
    qa = oracle.im2col(qd.reshape(n, hw, hw, f), 3, 3, 1)
    sa = oracle.im2col(sd.reshape(n, hw, hw, 1), 3, 3, 1)
    qb, sb = dgrad_filters_view(qm, sm, 9, c)
    ref = oracle.gemm(qa, sa, qb, sb, t)
    assert np.array_equal(x.grad.cpu().numpy().reshape(n * hw * hw, c), ref["c_seq"])
    # and the whole layer stays close to the FP32 convolution it stands for
    w4 = layer.weight.detach().view(3, 3, c, f).permute(3, 2, 0, 1).contiguous()          # [f][c][3][3]
    y32 = torch.nn.functional.conv2d(x.detach().permute(0, 3, 1, 2), w4, padding=1).permute(0, 2, 3, 1)
    rel = (y.detach() - y32).norm() / y32.norm()
    assert float(rel) < 2e-2


@pytest.mark.parametrize("c,f", [(24, 40), (64, 40), (32, 96)])
def test_convolution_layer_on_shapes_without_an_implicit_route(env, c, f):
    """Feature-map counts that the implicit GEMM or the regrouped filters do not cover take the gathered operand and the scatter:
    the same products as the library's calls one by one (the scatter's FP32 sums to rounding: nine terms, 9 * 2^-24)."""
    torch, hbfp_nn, hb = env
    torch.manual_seed(4)
    n, hw = 2, 8
    px = n * hw * hw
    layer = hbfp_nn.HbfpConv3x3(c, f)
    x = torch.randn(n, hw, hw, c, device="cuda").requires_grad_(True)
    dy = torch.randn(n, hw, hw, f, device="cuda")
    y = layer(x)
    y.backward(dy)
    q = hb.quantize(x.detach().view(px, c), 1, layer.fmt_pixels(0))
    want = hb.gemm_q(px, f, 9 * c, hb.im2col_packed(q, n, hw, hw, c, 3, 3, 1), layer.views[0])
    assert torch.allclose(y.detach().view(px, f), want, rtol=1e-6, atol=1e-6 * float(want.abs().max()))
    dcols = hb.gemm_q(px, 9 * c, f, dy.view(px, f), layer.views[1], fmtA=layer.fmt_pixels(2)).view(n, hw, hw, 3, 3, c)
    dxp = torch.zeros((n, hw + 2, hw + 2, c), device="cuda")
    for i in range(3):
        for j in range(3):
            dxp[:, i:i + hw, j:j + hw, :] += dcols[:, :, :, i, j, :]
    want = dxp[:, 1:hw + 1, 1:hw + 1, :]
    assert torch.allclose(x.grad, want, rtol=1e-5, atol=9 * 2.0 ** -24 * float(dcols.abs().max()) * 9)
    assert layer.weight.grad.shape == (9 * c, f) and hb.device_status() == 0


def test_layer_nodes_follow_autograd(env):
    """Gradients only for what asks for one, none recorded under no_grad, the library's error out of a backward pass."""
    torch, hbfp_nn, hb = env
    layer = hbfp_nn.HbfpLinear(48, 24)
    x = torch.randn(32, 48, device="cuda")
    layer(x).sum().backward()
    assert x.grad is None and layer.weight.grad.shape == (48, 24) and layer.bias.grad.shape == (24,)
    with torch.no_grad():
        assert layer(x).grad_fn is None
    layer.requires_grad_(False)
    assert not layer(x).requires_grad
    xg = x.clone().requires_grad_(True)
    layer(xg).sum().backward()
    assert xg.grad.shape == x.shape
    wide = hbfp_nn.HbfpLinear(48, 24, mant_bits=12, batch_block=600)      # block sums of 600 products of 12 bits exceed int32
    y = wide(x)
    with pytest.raises(hb.HbfpError) as e:
        y.sum().backward()
    assert e.value.code == hb.ERR_UNSUPPORTED
    with pytest.raises(ValueError):
        layer(x.half())


@pytest.mark.parametrize("batch,fin,fout,m,t", [(16, 300, 130, 8, 64), (128, 784, 1024, 8, 24), (300, 256, 128, 8, 128), (256, 40, 33, 8, 32), (2304, 1024, 2048, 12, 64),
                                                (640, 2048, 1280, 8, 32), (2048, 2048, 2560, 8, 128), (300, 4096, 100, 8, 64), (130, 500, 131, 12, 24)])
def test_bias_added_by_the_product_and_its_gradient(env, batch, fin, fout, m, t):
    """Whichever kernel the product takes, adding the bias in its store gives the bits of adding it afterwards; the column sums
    of dY against binary64 (a chain of at most batch / 64 + 22 additions of like magnitude)."""
    torch, hbfp_nn, hb = env
    torch.manual_seed(6)
    layer = hbfp_nn.HbfpLinear(fin, fout, mant_bits=m, tile=t, seed=2)
    x, bias = torch.randn(batch, fin, device="cuda"), torch.randn(fout, device="cuda")
    with torch.no_grad():
        plain = layer(x)                     # the bias starts as zeros
        layer.bias.copy_(bias)
        assert torch.equal(layer(x), plain + bias)
    dy = torch.randn(batch, fout, device="cuda")
    layer.weight.requires_grad_(False)
    layer(x).backward(dy)
    d = dy.double()
    bound = (batch / 64 + 22) * 2.0 ** -24 * d.abs().sum(0)
    assert bool(((layer.bias.grad.double() - d.sum(0)).abs() <= bound).all()) and hb.device_status() == 0


def test_out_of_memory_keeps_its_type(env):
    """A caller that catches torch.OutOfMemoryError to shrink a batch finds it out of the calls and the layers (the allocator's limit
    for this process is lowered; the GPU has room). Results of gigabytes from operands of megabytes, so that nothing the allocator
    still holds from elsewhere could serve them."""
    torch, hbfp_nn, hb = env
    A, fmt = torch.randn(40000, 8, device="cuda"), hb.Format(8, 64)
    layer, x = hbfp_nn.HbfpLinear(64, 6000, rounding=0), torch.randn(200000, 64, device="cuda")
    conv, xc = hbfp_nn.HbfpConv3x3(64, 8192), torch.randn(64, 32, 32, 64, device="cuda")
    long = torch.randn(10000000, 1, device="cuda")
    px = hb.quantize(xc.view(-1, 64), 1, conv.fmt_pixels(0))
    total = torch.cuda.get_device_properties(0).total_memory
    torch.cuda.empty_cache()
    torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (8 << 20)) / total)
    try:
        for call in (lambda: hb.gemm(0, 1, A, A, fmt, fmt), lambda: hb.quantize(long, 1, hb.Format(12, 64)), lambda: layer(x), lambda: conv(xc),
                     lambda: hb.conv_forward(px, conv.views[0], 64, 32, 32, 64, 3, 3, 1)):
            with pytest.raises(torch.OutOfMemoryError):
                call()
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert layer(x[:60000]).shape == (60000, 6000)


def test_inputs_of_the_wrong_width_do_not_train(env):
    """More columns than the weights have rows: no gradient of the right shape from the first columns alone. Fewer: refused at once."""
    torch, hbfp_nn, hb = env
    layer = hbfp_nn.HbfpLinear(96, 48, rounding=0)
    for requires_grad in (False, True):
        y = layer(torch.randn(64, 100, device="cuda", requires_grad=requires_grad))
        with pytest.raises(RuntimeError, match="invalid gradient"):
            y.sum().backward()
    assert layer.weight.grad is None
    with pytest.raises(hb.HbfpError):
        layer(torch.randn(64, 90, device="cuda"))


@pytest.mark.parametrize("kind", ["linear", "conv"])
def test_layers_under_a_trace_forward_mode_and_function_transforms(env, kind):
    """A trace records the layer (and replays it on other inputs, with gradients), what has no derivative of that kind says so."""
    torch, hbfp_nn, hb = env
    import torch.autograd.forward_ad as fwad
    torch.manual_seed(9)
    layer, shape = (hbfp_nn.HbfpLinear(96, 48, rounding=0), (64, 96)) if kind == "linear" else (hbfp_nn.HbfpConv3x3(64, 64), (2, 16, 16, 64))
    x, x2 = torch.randn(shape, device="cuda"), torch.randn(shape, device="cuda").requires_grad_(True)
    traced = torch.jit.trace(layer, (x,), check_trace=False)
    want, got = layer(x2), traced(x2)
    assert torch.equal(want, got)
    dy = torch.randn_like(want)
    assert torch.equal(*(torch.autograd.grad(y, x2, dy)[0] for y in (want, got)))
    with fwad.dual_level(), pytest.raises(NotImplementedError):
        layer(fwad.make_dual(x, torch.ones_like(x)))
    for transform in (lambda: torch.func.jvp(layer, (x,), (x,)), lambda: torch.func.grad(lambda v: layer(v).sum())(x), lambda: torch.func.vmap(layer)(x[None])):
        with pytest.raises(RuntimeError, match="functorch transforms"):
            transform()
    assert torch.equal(layer(x2), want)


@pytest.mark.parametrize("shape,dtype,device", [((48,), "float16", "cuda"), ((48,), "bfloat16", "cuda"), ((1,), "float32", "cuda"), ((), "float32", "cuda"), ((), "float32", "cpu"),
                                                ((48,), "float64", "cuda")])
def test_bias_of_another_type_or_shape(env, shape, dtype, device):
    """Whatever torch adds to a float32 matrix: the sum's type and values, and a gradient like the bias."""
    torch, hbfp_nn, hb = env
    torch.manual_seed(3)
    layer, x, dy = hbfp_nn.HbfpLinear(96, 48, rounding=0), torch.randn(64, 96, device="cuda"), torch.randn(64, 48, device="cuda")
    with torch.no_grad():
        plain = layer(x)
    layer.bias = torch.nn.Parameter(torch.randn(shape, device=device).to(getattr(torch, dtype)))
    y = layer(x)
    want = plain + layer.bias
    assert y.dtype == want.dtype and torch.equal(y, want)
    if dtype != "float64":                      # the products take float32 gradients
        y.backward(dy)
        assert layer.bias.grad.dtype == layer.bias.dtype and layer.bias.grad.shape == layer.bias.shape
        sums = dy.sum(0) if shape else dy.sum(0).sum()
        assert torch.allclose(layer.bias.grad.float(), (sums.sum(0, keepdim=True) if shape == (1,) else sums).to(device), rtol=1e-2, atol=1e-2)


def test_a_layer_cast_to_half_precision_computes_as_before(env):
    torch, hbfp_nn, hb = env
    layer, x = hbfp_nn.HbfpLinear(96, 48, rounding=0).half(), torch.randn(64, 96, device="cuda")
    layer(x).sum().backward()
    assert layer(x).dtype == torch.float32 and layer.weight.grad.dtype == layer.bias.grad.dtype == torch.float16


def test_layers_that_override_their_formats(env):
    """The format methods are what a subclass (or one layer) changes the conversions by: both passes use what they return."""
    import dataclasses
    torch, hbfp_nn, hb = env

    class Literal(hbfp_nn.HbfpLinear):
        def fmt_act(self, which, batch_axis=False):
            return dataclasses.replace(super().fmt_act(which, batch_axis), exp_mode=1)

    # powers of two, where the two exponent rules differ (the block's largest value saturates under the literal one)
    x = torch.exp2(torch.randint(-6, 3, (64, 96), device="cuda").float())
    dy = torch.exp2(torch.randint(-6, 3, (64, 48), device="cuda").float())
    torch.manual_seed(1)
    own = Literal(96, 48, rounding=0)
    own(x).backward(dy)
    f = own.fmt_act(0)
    assert torch.equal(own(x).detach(), hb.gemm_q(64, 48, 96, x, own.views[0], fmtA=f) + own.bias.detach())
    assert torch.equal(own.weight.grad, hb.gemm(1, 0, x, dy, own.fmt_act(0, True), own.fmt_act(2, True)))
    assert not torch.equal(own(x), hb.gemm_q(64, 48, 96, x, own.views[0], fmtA=dataclasses.replace(f, exp_mode=0)) + own.bias)
    conv, xc = hbfp_nn.HbfpConv3x3(64, 64), torch.randn(2, 16, 16, 64, device="cuda")
    plain = conv(xc)
    conv.fmt_pixels = lambda which: hb.Format(mant_bits=4, block=64, stream_id=which)
    px = hb.quantize(xc.view(-1, 64), 1, conv.fmt_pixels(0))
    assert torch.equal(conv(xc).view(-1, 64), hb.conv_forward(px, conv.views[0], 2, 16, 16, 64, 3, 3, 1)) and not torch.equal(conv(xc), plain)


def test_bias_gradient_can_be_differentiated(env):
    torch, hbfp_nn, hb = env
    layer, x = hbfp_nn.HbfpLinear(96, 48, rounding=0), torch.randn(64, 96, device="cuda")
    dy, v = torch.randn(64, 48, device="cuda", requires_grad=True), torch.randn(48, device="cuda")
    (db,) = torch.autograd.grad(layer(x), layer.bias, dy, create_graph=True)
    (g,) = torch.autograd.grad(db, dy, v)
    assert torch.equal(g, v.expand(64, 48))
    plain = torch.autograd.grad(layer(x), layer.bias, dy.detach())[0]
    assert torch.allclose(db, plain, rtol=1e-5, atol=1e-5)


def test_a_gradient_that_never_came_counts_as_zeros(env):
    torch, hbfp_nn, hb = env

    class Drop(torch.autograd.Function):
        @staticmethod
        def forward(ctx, x):
            return x.clone()

        @staticmethod
        def backward(ctx, g):
            return None

    layer, conv = hbfp_nn.HbfpLinear(96, 48, rounding=0), hbfp_nn.HbfpConv3x3(64, 64)
    for mod, x in ((layer, torch.randn(64, 96, device="cuda", requires_grad=True)), (conv, torch.randn(2, 16, 16, 64, device="cuda", requires_grad=True))):
        Drop.apply(mod(x)).sum().backward()
        for t in (x, *mod.parameters()):
            assert t.grad.shape == t.shape and not t.grad.any()


def test_other_threads_run_while_a_call_is_in_the_library(env):
    """The interpreter lock is let go around the library: with entry points that only sleep (libc's usleep, whose argument is the
    product's first extent) in place of the product's, another thread counts on meanwhile."""
    import ctypes
    import threading
    torch, hbfp_nn, hb = env
    native, L = hb.host(), hb.lib()
    sleep = ctypes.cast(ctypes.CDLL(None).usleep, ctypes.c_void_p).value
    entry = {n: ctypes.cast(getattr(L, n), ctypes.c_void_p).value for n in hb._HOST_ENTRY_POINTS}
    p = hb.quantize(torch.randn(32, 32, device="cuda"), 1, hb.Format(8, 32))
    out, count, stop = torch.empty(32, 32, device="cuda"), [0], threading.Event()

    def counter():
        while not stop.wait(0.01):
            count[0] += 1

    native.bind(hb.HbfpError, *({**entry, "hbfp_gemm_q_workspace": sleep, "hbfp_gemm_q_bias": sleep}[n] for n in hb._HOST_ENTRY_POINTS))
    thread = threading.Thread(target=counter)
    try:
        thread.start()
        before = count[0]
        native.gemm_q(300000, 32, 32, p, p, 0, 0, None, None, out, None, 0)      # 0.6 s asleep in the library
        during = count[0] - before
    finally:
        native.bind(hb.HbfpError, *(entry[n] for n in hb._HOST_ENTRY_POINTS))
        stop.set()
        thread.join()
    assert during >= 10
    assert torch.equal(hb.gemm_q(32, 32, 32, p, p), hb.gemm_q(32, 32, 32, p, p, flags=hb.GEMM_FORCE_SIMT))


@pytest.mark.parametrize("rows,cols", [(1, 2097121), (130, 2097153), (3, 8388484)])
def test_column_sums_of_more_columns_than_a_grid_has(env, rows, cols):
    """A layer's bias gradient for any number of outputs (one and four columns per lane; rows + 1 additions at most)."""
    import ctypes
    torch, hbfp_nn, hb = env
    x, out = torch.randn(rows, cols, device="cuda"), torch.full((cols + 1,), 7.0, device="cuda")
    assert hb.lib().hbfp_column_sums(ctypes.c_void_p(x.data_ptr()), ctypes.c_int64(rows), ctypes.c_int64(cols), ctypes.c_int64(cols), ctypes.c_void_p(out.data_ptr()),
                                     ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    d = x.double()
    assert bool(((out[:-1].double() - d.sum(0)).abs() <= (rows + 1) * 2.0 ** -24 * d.abs().sum(0)).all()) and float(out[-1]) == 7.0


@pytest.mark.parametrize("batch,fin,fout,tile", [(300, 296, 92, 32), (520, 64, 33, 24), (936, 1287, 200, 24), (130, 4000, 70, 64), (700, 640, 640, 64), (16, 256, 130, 32)])
def test_bias_added_by_whichever_kernel_ends_the_product(env, batch, fin, fout, tile):
    """The smallest products, sums of split-K parts, unsplit tiles and a few rows: the value of adding it afterwards, bit for bit."""
    torch, hbfp_nn, hb = env
    layer = hbfp_nn.HbfpLinear(fin, fout, tile=tile, rounding=0)
    x = torch.randn(batch, fin, device="cuda")
    with torch.no_grad():
        plain = layer(x)
        layer.bias.normal_()
        assert torch.equal(layer(x), plain + layer.bias)
    assert hb.device_status() == 0


@pytest.mark.parametrize("kind", ["linear", "linear12", "conv"])
def test_layer_step_captured_in_a_cuda_graph(env, kind):
    """Forward, both gradients and the update of the weights in one graph: replays train on as the same steps outside one do."""
    torch, hbfp_nn, hb = env

    def make():
        torch.manual_seed(5)
        if kind == "conv":
            return hbfp_nn.HbfpConv3x3(64, 64)
        return hbfp_nn.HbfpLinear(600, 712, mant_bits=12 if kind == "linear12" else 8, tile=64 if kind == "linear12" else 24, rounding=0)

    x = torch.randn((8, 16, 16, 64) if kind == "conv" else (2100, 600), device="cuda", requires_grad=True)
    dy = torch.randn((8, 16, 16, 64) if kind == "conv" else (2100, 712), device="cuda")

    def step(layer, grads):
        got = torch.autograd.grad(layer(x), [x, layer.weight], dy)
        for out, g in zip(grads, got):
            out.copy_(g)
        layer.apply_update(got[1] * -1e-2)

    eager, captured = make(), make()
    want, got = ([torch.empty_like(x), torch.empty_like(eager.weight)] for _ in range(2))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step(make(), got)                                 # sets the kernels' attributes
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step(captured, got)
    for _ in range(4):
        step(eager, want)
        graph.replay()
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        assert torch.equal(captured.wide.mant, eager.wide.mant) and torch.equal(captured.wide.exps, eager.wide.exps)
        assert torch.equal(captured.weight.data, eager.weight.data)
    assert hb.device_status() == 0
