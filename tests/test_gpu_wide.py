"""GPU parity of wide weight storage through the C ABI: 16-bit mantissas and tile exponents bit-exact
(nearest-even and stochastic rounding), the narrow views equal to the top bits of the wide mantissas,
the in-place FP32 update equal to the oracle's, and GEMMs on the derived views equal to the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1804_01526_b200 import workloads as wl
from tests.helpers import decode_packed, gfmt, ofmt, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hb():
    from paper_1804_01526_b200 import binding
    binding.lib()
    return binding


def F(m, t, rounding=0, seed=0, stream_id=0):
    return dict(mant_bits=m, block=t, tile=t, rounding=rounding, seed=seed, stream_id=stream_id)


def check_views(hb, views, qm, sm, t):
    """views (c0, c1) against the canonical narrow arrays qm [d0][d1], sm [d0][ceil(d1/t)]."""
    c0, c1 = views
    q1, s1 = decode_packed(c1, hb.packed_layout(c1.rows, c1.k, c1.fmt))
    assert np.array_equal(q1, qm) and np.array_equal(s1, sm)
    q0, s0 = decode_packed(c0, hb.packed_layout(c0.rows, c0.k, c0.fmt))
    grid = sm[::t, :]                                            # [tiles along d0][tiles along d1]
    assert np.array_equal(q0, qm.T)
    assert np.array_equal(s0, np.repeat(grid.T, t, axis=0)[: qm.shape[1], :])


CASES = [
    ((784, 1024), "he_weight", F(8, 24, 1, seed=1, stream_id=1)),      # MLP layer, the paper's sweet spot: tile 24
    ((1024, 10), "he_weight", F(8, 24)),
    ((1000, 4096 // 4), "he_weight", F(12, 64, 1, seed=7, stream_id=11)),
    ((130, 257), "lognormal", F(4, 128)),
    ((61, 100), "lognormal", F(12, 24, 1, seed=5)),
    ((7, 5), "normal", F(8, 16)),
]


@pytest.mark.parametrize("shape,law,fd", CASES)
def test_wide_quantise_and_narrow_views_match_the_oracle(hb, shape, law, fd):
    kw = {"fan_in": shape[0]} if law == "he_weight" else {}
    w = wl.draw(law, shape, seed=21, **kw)
    t, m = fd["tile"], fd["mant_bits"]
    wide, views = hb.wide_quantize(to_dev(w), gfmt(fd))
    assert hb.device_status() == 0
    q16, s16 = oracle.wide_quantize(w, ofmt(fd))
    assert np.array_equal(wide.mant.cpu().numpy(), q16)
    assert np.array_equal(wide.exps.cpu().numpy(), s16[::t, :])
    qm, sm = oracle.wide_narrow(q16, s16, m)
    check_views(hb, views, qm, sm, t)
    # the read-only entry point writes the same views
    again = hb.wide_narrow(wide, gfmt(fd))
    check_views(hb, again, qm, sm, t)
    # the FP32 value of the wide copy is Eq. 1 written out: mantissa times 2^(tile exponent), exact
    val = hb.wide_dequantize(wide).cpu().numpy()
    assert np.array_equal(val, np.ldexp(q16.astype(np.float64), np.repeat(s16, t, axis=1)[:, : shape[1]].astype(np.int64)).astype(np.float32))
    for a, b in zip(again, views):                               # and the same bytes in every documented position
        lay = hb.packed_layout(a.rows, a.k, a.fmt)
        for pl in range(lay["planes"]):
            lo, hi = pl * lay["plane_stride"], pl * lay["plane_stride"] + a.rows * lay["kst"]
            assert np.array_equal(a.mant[lo:hi].cpu().numpy(), b.mant[lo:hi].cpu().numpy())
    # wide storage alone
    wide2, none = hb.wide_quantize(to_dev(w), gfmt(fd), want_views=False)
    assert none is None and np.array_equal(wide2.mant.cpu().numpy(), q16)


@pytest.mark.parametrize("shape,fd", [((784, 1024), F(8, 24, 1, seed=3, stream_id=4)), ((333, 200), F(12, 64)),
                                      ((130, 257), F(8, 128, 1, seed=9))])
def test_wide_update_matches_the_oracle_over_several_steps(hb, shape, fd):
    w = wl.draw("he_weight", shape, seed=22, fan_in=shape[0])
    t, m = fd["tile"], fd["mant_bits"]
    wide, _ = hb.wide_quantize(to_dev(w), gfmt(fd), want_views=False)
    q, s = oracle.wide_quantize(w, ofmt(fd))
    for step in range(3):
        delta = (wl.draw("grad", shape, seed=30 + step) * (10.0 if step == 1 else 1.0)).astype(np.float32)
        if step == 2:
            delta[:, : shape[1] // 2] = 0                        # part of the matrix does not move
        fstep = dict(fd, seed=fd["seed"] + 100 * step)             # fresh draws every step
        views = hb.wide_update(wide, to_dev(delta), gfmt(fstep))
        assert hb.device_status() == 0
        q, s = oracle.wide_update(q, s, delta, ofmt(fstep))
        assert np.array_equal(wide.mant.cpu().numpy(), q)
        assert np.array_equal(wide.exps.cpu().numpy(), s[::t, :])
        qm, sm = oracle.wide_narrow(q, s, m)
        check_views(hb, views, qm, sm, t)


def test_forward_and_backward_data_on_views_derived_from_wide_storage(hb):
    # Y = X W and dX = dY W^T read the same narrow copy (top 8 bits, which can hold -128)
    batch, fin, fout, t = 128, 784, 1024, 24
    fw = F(8, t, 1, seed=1, stream_id=1)
    fx = dict(mant_bits=8, block=t, rounding=1, seed=1, stream_id=0)
    W = wl.draw("he_weight", (fin, fout), seed=23, fan_in=fin)
    X = wl.draw("half_normal", (batch, fin), seed=24)
    dY = wl.draw("grad", (batch, fout), seed=25)
    wide, (c0, c1) = hb.wide_quantize(to_dev(W), gfmt(fw))
    q16, s16 = oracle.wide_quantize(W, ofmt(fw))
    qm, sm = oracle.wide_narrow(q16, s16, 8)
    assert int(qm.min()) >= -128
    grid = sm[::t, :]
    # forward: contraction over fin; B operand canonical [fout][fin]
    qx, sx = oracle.quantize(X, 1, ofmt(fx))
    sB_rows = np.repeat(grid.T, t, axis=0)[:fout, :]
    ref = oracle.gemm(qx, sx, np.ascontiguousarray(qm.T), np.ascontiguousarray(sB_rows), t)
    Y = hb.gemm_q(batch, fout, fin, to_dev(X), c0, fmtA=gfmt(fx)).cpu().numpy()
    err = np.abs(Y.astype(np.float64) - ref["c_ref"].astype(np.float64))
    assert (err <= 1e-6 * ref["a_mag"]).all()
    # backward-data: contraction over fout; B operand canonical [fin][fout] = the stored orientation
    fdy = dict(fx, stream_id=2)
    qd, sd = oracle.quantize(dY, 1, ofmt(fdy))
    ref = oracle.gemm(qd, sd, qm, sm, t)
    dX = hb.gemm_q(batch, fin, fout, to_dev(dY), c1, fmtA=gfmt(fdy)).cpu().numpy()
    err = np.abs(dX.astype(np.float64) - ref["c_ref"].astype(np.float64))
    assert (err <= 1e-6 * ref["a_mag"]).all()
    assert hb.device_status() == 0


def test_wide_argument_errors(hb):
    import torch
    w = to_dev(wl.draw("normal", (64, 64), seed=1))
    with pytest.raises(hb.HbfpError) as e:                          # tile != block
        hb.wide_quantize(w, hb.Format(mant_bits=8, block=32, tile=16))
    assert e.value.code == hb.ERR_INVALID_ARG
    with pytest.raises(hb.HbfpError) as e:                          # tiles above 128 are not supported here
        hb.wide_quantize(w, hb.Format(mant_bits=8, block=256, tile=256))
    assert e.value.code == hb.ERR_UNSUPPORTED
    wide, _ = hb.wide_quantize(w, hb.Format(mant_bits=8, block=16, tile=16), want_views=False)
    with pytest.raises(ValueError):
        hb.wide_update(wide, torch.zeros((32, 64), device="cuda"), hb.Format(mant_bits=8, block=16, tile=16))


def test_wide_storage_of_an_empty_matrix(hb):
    import torch
    f = hb.Format(mant_bits=8, block=16, tile=16)
    wide, views = hb.wide_quantize(torch.empty((0, 32), device="cuda"), f)
    assert wide.mant.numel() == 0 and hb.device_status() == 0
    hb.wide_update(wide, torch.empty((0, 32), device="cuda"), f, views=views)
    hb.wide_narrow(wide, f, views=views)
    assert hb.device_status() == 0


@pytest.mark.parametrize("shape,t,rounding", [
    ((1, 4), 4, 0), ((3, 1028), 4, 1),                  # four weights per access: one row, a part of a group of rows
    ((130, 2056), 24, 1), ((128, 256), 64, 0),          # several column blocks; whole tiles
    ((9, 1030), 24, 1), ((70, 36), 6, 0),               # one weight per access: ragged rows; a tile that is no multiple of 4
])
def test_update_also_writes_the_fp32_value(hb, shape, t, rounding):
    fd = F(8, t, rounding, seed=3)
    w, delta = wl.draw("normal", shape, seed=5), wl.draw("normal", shape, seed=6) * np.float32(0.01)
    wide, views = hb.wide_quantize(to_dev(w), gfmt(fd))
    value = hb.wide_update_value(wide, to_dev(delta), gfmt(fd), views).cpu().numpy()
    q16, e = wide.mant.cpu().numpy(), wide.exps.cpu().numpy().astype(np.int64)
    s16 = np.repeat(np.repeat(e, t, axis=0)[: shape[0]], t, axis=1)[:, : shape[1]]
    exact = np.ldexp(q16.astype(np.float64), s16).astype(np.float32)      # 16-bit mantissas: exact in binary32
    assert np.array_equal(value, exact)
    assert np.array_equal(hb.wide_dequantize(wide).cpu().numpy(), exact)


# Tile geometries that are not whole tiles of 32, 64 or 128 (and these in widths cut from the words early): strips of one to eight tile rows, ragged last tiles and strips in both
# directions, odd row lengths, every view from FP32 weights, from wide words and after an update.
@pytest.mark.parametrize("d0,d1,t,m,rounding", [
    (1, 1, 1, 8, 1), (70, 13, 1, 8, 0), (83, 91, 5, 12, 1), (64, 40, 8, 4, 0), (75, 163, 9, 8, 1), (129, 257, 16, 12, 0), (145, 301, 17, 8, 1), (48, 120, 24, 8, 1),
    (95, 241, 24, 12, 0), (65, 129, 32, 8, 1), (64, 127, 32, 4, 1), (131, 259, 33, 8, 0), (97, 193, 48, 12, 1), (65, 257, 64, 8, 1), (128, 256, 64, 4, 0),
    (101, 203, 100, 8, 1), (129, 255, 128, 12, 1), (256, 128, 128, 4, 1), (41, 104, 32, 8, 1), (129, 200, 64, 12, 0), (63, 72, 64, 4, 1), (150, 328, 128, 9, 1)])
def test_weight_tiles_of_any_geometry(hb, d0, d1, t, m, rounding):
    fd = F(m, t, rounding, seed=11, stream_id=2)
    w = wl.draw("lognormal", (d0, d1), seed=77)
    w[0, 0] = 0.0
    w[:, d1 // 2] = np.float32(2.0) ** np.arange(d0, dtype=np.float32).clip(0, 20)      # tile maxima at powers of two
    q16, s16 = oracle.wide_quantize(w, ofmt(fd))
    wide, views = hb.wide_quantize(to_dev(w), gfmt(fd))
    assert np.array_equal(wide.mant.cpu().numpy(), q16) and np.array_equal(wide.exps.cpu().numpy(), s16[::t, :])
    check_views(hb, views, *oracle.wide_narrow(q16, s16, m), t)
    check_views(hb, hb.wide_narrow(wide, gfmt(fd)), *oracle.wide_narrow(q16, s16, m), t)
    # a pitch longer than the rows; the update with and without the FP32 value
    delta = (wl.draw("grad", (d0, d1 + 3), seed=78) * 3).astype(np.float32)
    q16, s16 = oracle.wide_update(q16, s16, np.ascontiguousarray(delta[:, :d1]), ofmt(fd))
    other = hb.Wide(wide.mant.clone(), wide.exps.clone(), t)
    value = hb.wide_update_value(other, to_dev(delta)[:, :d1], gfmt(fd), views)
    check_views(hb, views, *oracle.wide_narrow(q16, s16, m), t)
    check_views(hb, hb.wide_update(wide, to_dev(delta)[:, :d1], gfmt(fd)), *oracle.wide_narrow(q16, s16, m), t)
    for x in (wide, other):
        assert np.array_equal(x.mant.cpu().numpy(), q16) and np.array_equal(x.exps.cpu().numpy(), s16[::t, :])
    assert np.array_equal(value.cpu().numpy(), hb.wide_dequantize(wide).cpu().numpy())
    # straight to m bits
    c0, c1, grid = hb.quantize_tiles(to_dev(w), gfmt(fd))
    qn, sn = oracle.quantize(w, 1, ofmt(fd))
    check_views(hb, (c0, c1), qn, sn, t)
    assert np.array_equal(grid.cpu().numpy(), sn[::t, :])
    assert hb.device_status() == 0


# The same on both sides of every line between a CTA per tile and strips, with strips cut down and whole, and a view by itself: small and
# middling tiles, aligned and not, with and without draws.
@pytest.mark.parametrize("d0,d1,t,m,rounding", [
    (58, 111, 2, 8, 1), (101, 101, 4, 12, 0), (130, 262, 5, 8, 1), (192, 400, 8, 8, 1), (201, 411, 8, 4, 0), (300, 290, 12, 12, 1), (272, 1120, 16, 8, 0),
    (480, 928, 16, 8, 1), (500, 501, 20, 8, 1), (601, 597, 24, 8, 0), (600, 1160, 24, 12, 1), (864, 1224, 24, 8, 1), (1008, 1032, 24, 4, 0), (420, 1100, 28, 8, 0),
    (780, 797, 32, 8, 1), (400, 520, 40, 8, 1), (1648, 1728, 48, 8, 0), (1632, 1736, 48, 8, 1), (800, 993, 65, 8, 0), (1600, 1699, 65, 8, 1), (216, 360, 72, 12, 1),
    (1000, 1003, 88, 8, 0), (1250, 1251, 96, 8, 0), (224, 560, 112, 8, 1), (1344, 1512, 112, 8, 0)])
def test_weight_tiles_on_both_sides_of_the_kernels_rule(hb, d0, d1, t, m, rounding):
    test_weight_tiles_of_any_geometry(hb, d0, d1, t, m, rounding)
    # a view by itself
    fd = F(m, t, rounding, seed=11, stream_id=2)
    w = wl.draw("lognormal", (d0, d1), seed=78)
    for axis in (0, 1):
        p = hb.quantize(to_dev(w), axis, gfmt(fd))
        q, s = decode_packed(p, hb.packed_layout(p.rows, p.k, p.fmt))
        q_ref, s_ref = oracle.quantize(w, axis, ofmt(fd))
        assert np.array_equal(q, q_ref) and np.array_equal(s, s_ref)


@pytest.mark.parametrize("d0,d1,t,rounding,per_tile", [
    (64, 64, 8, 0, True), (100, 100, 5, 1, True), (256, 300, 24, 0, True), (1000, 1000, 24, 1, True), (2048, 2048, 40, 0, True), (1000, 1000, 72, 1, True),
    (4096, 4096, 80, 0, True), (2048, 2048, 120, 1, True), (1001, 1003, 72, 0, True), (2000, 3001, 72, 1, True), (256, 300, 8, 0, False), (784, 1024, 8, 1, False),
    (1111, 5001, 24, 0, False), (1000, 1500, 32, 1, False), (2000, 3001, 100, 1, False)])
def test_launches_of_weight_updates(hb, d0, d1, t, rounding, per_tile):
    """A CTA per tile, or strips of which there are enough for every SM where the tiles are."""
    import ctypes
    import torch

    class Params(ctypes.Structure):                       # CUDA_KERNEL_NODE_PARAMS_v2
        _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3), ("block", ctypes.c_uint * 3), ("shared", ctypes.c_uint), ("rest", ctypes.c_void_p * 4)]

    f = hb.Format(mant_bits=8, block=t, tile=t, rounding=rounding)
    wide, views = hb.wide_quantize(torch.randn(d0, d1, device="cuda"), f)
    delta = torch.zeros(d0, d1, device="cuda")
    hb.wide_update(wide, delta, f, views=views)           # sets the kernels' attributes
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        hb.wide_update(wide, delta, f, views=views)
    driver, node, n, p = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_size_t(1), Params()
    assert driver.cuGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.byref(node), ctypes.byref(n)) == 0 and n.value == 1
    assert driver.cuGraphKernelNodeGetParams_v2(node, ctypes.byref(p)) == 0
    nu, nv = -(-d0 // t), -(-d1 // t)
    ctas = p.grid[0] * p.grid[1]
    assert (tuple(p.grid) == (nv, nu, 1) and p.block[0] == 256) == per_tile
    assert min(148, nu * nv) <= ctas <= nu * nv


def test_tiles_of_different_lengths_from_two_threads(hb):
    """One kernel serves several tile lengths, each with its own need of shared memory: a thread that launches the one must not take
    from another what it launches the other with."""
    import threading
    import torch
    failed = []

    def work(t):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            f = hb.Format(mant_bits=8, block=t, tile=t, rounding=1, seed=2)
            w = torch.randn(1000, 1000, device="cuda")
            wide, views = hb.wide_quantize(w, f)
            try:
                for _ in range(4000):
                    hb.wide_update(wide, w, f, views=views)
            except hb.HbfpError as e:
                failed.append((t, str(e)))
            stream.synchronize()

    threads = [threading.Thread(target=work, args=(t,)) for t in (8, 16)]
    for x in threads: x.start()
    for x in threads: x.join()
    assert not failed and hb.device_status() == 0
