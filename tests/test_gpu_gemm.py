"""GPU parity of the BFP GEMMs through the C ABI: per-block integer sums bit-exact, outputs within
1e-6 of the FP32 accumulator magnitude of the oracle's order-free reference, and bit-equal to the
oracle's sequential accumulation where the kernel accumulates blocks in ascending order."""
import numpy as np
import pytest

import oracle
from paper_1804_01526_b200 import workloads as wl
from tests.helpers import gfmt, ofmt, to_dev

pytestmark = pytest.mark.gpu

TOL = 1e-6      # of the accumulator magnitude sum_kb |T|, as the target states


@pytest.fixture(scope="module")
def hb():
    from paper_1804_01526_b200 import binding
    binding.lib()
    return binding


def run_spec(hb, sp, tensors, flags, expect_seq=True):
    A, B = tensors[sp.a_key], tensors[sp.b_key]
    ref = oracle.hbfp_gemm(sp.transA, sp.transB, A, B, ofmt(sp.fmt_a), ofmt(sp.fmt_b))
    C = hb.gemm(sp.transA, sp.transB, to_dev(A), to_dev(B), gfmt(sp.fmt_a), gfmt(sp.fmt_b), flags=flags)
    C = C.cpu().numpy()
    assert hb.device_status() == 0
    err = np.abs(C.astype(np.float64) - ref["c_ref"].astype(np.float64))
    assert (err <= TOL * ref["a_mag"]).all(), (sp.name, float((err / np.maximum(ref["a_mag"], 1e-300)).max()))
    if expect_seq:
        assert np.array_equal(C, ref["c_seq"]), sp.name
    return C, ref


def impls(hb):
    return [hb.GEMM_FORCE_SIMT, hb.GEMM_AUTO]


@pytest.mark.parametrize("flag", ["simt", "auto"])
def test_single_256_cube(hb, flag):
    specs = wl.config_single_256()
    t = wl.materialize(specs, seed=0)
    run_spec(hb, specs[0], t, hb.GEMM_FORCE_SIMT if flag == "simt" else hb.GEMM_AUTO)


@pytest.mark.parametrize("flag", ["simt", "auto"])
def test_mlp_training_step_gemms(hb, flag):
    specs = wl.config_mlp()
    t = wl.materialize(specs, seed=1)
    for sp in specs:
        run_spec(hb, sp, t, hb.GEMM_FORCE_SIMT if flag == "simt" else hb.GEMM_AUTO,
                 expect_seq=(flag == "simt"))


@pytest.mark.parametrize("flag", ["simt", "auto"])
def test_resnet_im2col_gemms_reduced_batch(hb, flag):
    # batch 2 instead of 128 (M = 2048 / 512 rows): same K, N, formats and value laws
    specs = wl.config_resnet_im2col(batch=2)
    t = wl.materialize(specs, seed=2)
    for sp in specs:
        run_spec(hb, sp, t, hb.GEMM_FORCE_SIMT if flag == "simt" else hb.GEMM_AUTO,
                 expect_seq=(flag == "simt"))


@pytest.mark.parametrize("flag", ["simt", "auto"])
def test_transformer_gemms_reduced(hb, flag):
    # tokens 192, hidden 256: 12-bit hi/lo mantissas, 64 x 64 shared weight tiles, stochastic rounding
    specs = wl.config_transformer(tokens=192, hidden=256)
    t = wl.materialize(specs, seed=7)
    for sp in specs:
        run_spec(hb, sp, t, hb.GEMM_FORCE_SIMT if flag == "simt" else hb.GEMM_AUTO,
                 expect_seq=(flag == "simt"))


SMALL_CASES = [
    # transA, transB, M, N, K, mantissa bits, block, tile of B, rounding
    (0, 0, 128, 1024, 784, 8, 24, 24, 1),       # forward GEMM of the MLP configuration
    (0, 1, 128, 784, 1024, 8, 24, 24, 1),       # its backward-data GEMM (shared tiles read the other way)
    (1, 0, 784, 1024, 128, 8, 24, 0, 1),        # its backward-weight GEMM
    (0, 0, 1, 1, 1, 8, 32, 0, 0),
    (0, 0, 33, 95, 100, 6, 64, 0, 0),           # ragged in every dimension, two 32-byte steps per block
    (0, 0, 70, 50, 520, 8, 128, 0, 0),
    (1, 1, 40, 72, 900, 8, 200, 0, 1),          # blocks that span two 128-byte slices
    (0, 0, 64, 48, 300, 8, 0, 0, 0),            # one exponent per row / column
    (0, 0, 256, 256, 256, 4, 32, 32, 0),
]


@pytest.mark.parametrize("tA,tB,M,N,K,m,b,t,rounding", SMALL_CASES)
def test_small_problem_kernel_equals_the_sequential_definition(hb, tA, tB, M, N, K, m, b, t, rounding):
    """The tiled kernel for the smallest problems never splits K and adds blocks in ascending order: bit-equal to the oracle's c_seq."""
    A = wl.draw("lognormal", (K, M) if tA else (M, K), seed=31)
    B = wl.draw("he_weight", (N, K) if tB else (K, N), seed=32, fan_in=K)
    fa = dict(mant_bits=m, block=b, rounding=rounding, seed=4, stream_id=0)
    fb = dict(mant_bits=m, block=b, tile=t, rounding=rounding, seed=4, stream_id=1)
    ref = oracle.hbfp_gemm(tA, tB, A, B, ofmt(fa), ofmt(fb))
    C = hb.gemm(tA, tB, to_dev(A), to_dev(B), gfmt(fa), gfmt(fb), flags=hb.GEMM_FORCE_SMALL).cpu().numpy()
    assert hb.device_status() == 0 and hb.last_gemm_kernel() == "gemm_small_kernel"
    assert np.array_equal(C, ref["c_seq"])
    err = np.abs(C.astype(np.float64) - ref["c_ref"].astype(np.float64))
    assert (err <= TOL * ref["a_mag"]).all()


def test_small_problem_kernel_is_what_small_problems_get_and_large_ones_do_not(hb):
    fd = dict(mant_bits=8, block=64)
    A, B = wl.draw("normal", (256, 512), seed=33), wl.draw("normal", (512, 256), seed=34)
    hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd, stream_id=1))
    assert hb.last_gemm_kernel() == "gemm_small_kernel"
    A, B = wl.draw("normal", (1024, 2048), seed=35), wl.draw("normal", (2048, 1024), seed=36)
    hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd, stream_id=1))
    assert hb.last_gemm_kernel() == "gemm_tc_kernel"
    f12 = dict(mant_bits=12, block=64)
    with pytest.raises(hb.HbfpError) as e:
        hb.gemm(0, 0, to_dev(A[:64, :128].copy()), to_dev(B[:128, :64].copy()), gfmt(f12), gfmt(f12, stream_id=1), flags=hb.GEMM_FORCE_SMALL)
    assert e.value.code == hb.ERR_UNSUPPORTED


@pytest.mark.parametrize("impl", ["simt", "tensor"])
@pytest.mark.parametrize("m,b,M,N,K", [(8, 32, 200, 136, 288), (8, 128, 130, 260, 1024), (12, 64, 96, 72, 320),
                                       (8, 24, 50, 40, 100), (8, 0, 64, 64, 700), (8, 64, 128, 256, 512)])
def test_block_partials_are_bit_exact(hb, impl, m, b, M, N, K):
    A = wl.draw("lognormal", (M, K), seed=21)
    B = wl.draw("lognormal", (K, N), seed=22)
    fd = dict(mant_bits=m, block=b, rounding=1, seed=4)
    qA, sA = oracle.quantize(A, 1, ofmt(fd))
    qB, sB = oracle.quantize(B, 0, ofmt(fd, stream_id=1))
    ref = oracle.gemm(qA, sA, qB, sB, b, want_partials=True)
    pa = hb.quantize(to_dev(A), 1, gfmt(fd))
    pb = hb.quantize(to_dev(B), 0, gfmt(fd, stream_id=1))
    flag = hb.GEMM_FORCE_SIMT if impl == "simt" else hb.GEMM_FORCE_TENSOR
    try:
        P = hb.gemm_block_partials(pa, pb, flag)
    except hb.HbfpError as e:
        if impl == "tensor" and e.code == hb.ERR_UNSUPPORTED:
            pytest.skip("no tensor-core kernel for this case")
        raise
    assert np.array_equal(P.cpu().numpy(), ref["P"])
    assert hb.device_status() == 0


def test_backward_data_uses_packed_forward_weights(hb):
    """W is quantised ONCE into shared tiles; forward uses view c0 and backward-data view c1."""
    t, batch, fin, fout = 24, 64, 200, 136
    X = wl.draw("half_normal", (batch, fin), seed=31)
    W = wl.draw("he_weight", (fin, fout), seed=32, fan_in=fin)
    dY = wl.draw("grad", (batch, fout), seed=33)
    fw = dict(mant_bits=8, block=t, tile=t, rounding=1, seed=1, stream_id=1)
    fx = dict(mant_bits=8, block=t, rounding=1, seed=1, stream_id=0)
    fg = dict(mant_bits=8, block=t, rounding=1, seed=1, stream_id=2)
    c0, c1, _ = hb.quantize_tiles(to_dev(W), gfmt(fw))
    Y = hb.gemm_q(batch, fout, fin, to_dev(X), c0, transA=0, fmtA=gfmt(fx), flags=hb.GEMM_FORCE_SIMT).cpu().numpy()
    dX = hb.gemm_q(batch, fin, fout, to_dev(dY), c1, transA=0, fmtA=gfmt(fg), flags=hb.GEMM_FORCE_SIMT).cpu().numpy()
    assert np.array_equal(Y, oracle.hbfp_gemm(0, 0, X, W, ofmt(fx), ofmt(fw))["c_seq"])
    assert np.array_equal(dX, oracle.hbfp_gemm(0, 1, dY, W, ofmt(fg), ofmt(fw))["c_seq"])


def test_argument_errors_are_reported_not_thrown_by_cuda(hb):
    import torch
    A = torch.zeros((64, 64), device="cuda")
    f = hb.Format(8, 32)
    with pytest.raises(hb.HbfpError) as e:
        hb.gemm(0, 0, A, A, f, f, workspace=torch.empty(1024, dtype=torch.int8, device="cuda"))
    assert e.value.code == hb.ERR_WORKSPACE
    with pytest.raises(hb.HbfpError) as e:
        hb.gemm(0, 0, A, A, f, hb.Format(8, 64))
    assert e.value.code == hb.ERR_INVALID_ARG
    with pytest.raises(hb.HbfpError) as e:
        hb.quantize(A, 1, hb.Format(8, 32, rounding=5))
    assert e.value.code == hb.ERR_INVALID_ARG
    assert hb.device_status() == 0
    C = hb.gemm(0, 0, A[:0], A, f, f)          # empty M
    assert C.shape == (0, 64)


# The paired-SM kernel (two CTAs per 256 x 256 tile) needs at least 74 such tiles; these shapes span
# several tiles per SM pair, ragged edges in M, N and K, a second CTA whose half tile lies entirely
# outside the matrix (M % 256 <= 128, N % 256 <= 128), and all three blocks-per-stage variants.
PAIR_CASES = [
    # m, block, M, N, K
    (8, 128, 2560, 2048, 640),
    (8, 128, 2400, 2100, 1000),
    (8, 64, 2660, 2304, 448),
    (6, 64, 2304, 2188, 200),
    (8, 32, 2560, 2048, 288),
    (8, 100, 2688, 2176, 1000),
    (4, 16, 2330, 2332, 176),
]


@pytest.mark.parametrize("m,b,M,N,K", PAIR_CASES)
def test_paired_sm_kernel_matches_oracle_bit_for_bit(hb, m, b, M, N, K):
    A = wl.draw("lognormal", (M, K), seed=31)
    B = wl.draw("lognormal", (K, N), seed=32)
    fd = dict(mant_bits=m, block=b, rounding=0, seed=0)
    ref = oracle.hbfp_gemm(0, 0, A, B, ofmt(fd), ofmt(fd))
    C2 = hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd), flags=hb.GEMM_FORCE_TENSOR_2SM).cpu().numpy()
    assert hb.device_status() == 0
    err = np.abs(C2.astype(np.float64) - ref["c_ref"].astype(np.float64))
    assert (err <= TOL * ref["a_mag"]).all()
    assert np.array_equal(C2, ref["c_seq"])      # blocks accumulated in ascending order, no split-K
    C1 = hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd), flags=hb.GEMM_FORCE_TENSOR_1SM).cpu().numpy()
    assert np.array_equal(C1, C2)
    Ca = hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd), flags=hb.GEMM_AUTO).cpu().numpy()
    assert np.array_equal(Ca, C2)


def test_paired_sm_kernel_transposed_operands_and_stochastic_rounding(hb):
    # wgrad-shaped call: both operands are contracted along their row axis (column quantiser)
    M, N, K = 2304, 2304, 384
    X = wl.draw("half_normal", (K, M), seed=41)
    dY = wl.draw("grad", (K, N), seed=42)
    fa = dict(mant_bits=8, block=128, rounding=1, seed=9)
    ref = oracle.hbfp_gemm(1, 0, X, dY, ofmt(fa), ofmt(fa, stream_id=1))
    C = hb.gemm(1, 0, to_dev(X), to_dev(dY), gfmt(fa), gfmt(fa, stream_id=1), flags=hb.GEMM_FORCE_TENSOR_2SM).cpu().numpy()
    assert hb.device_status() == 0
    assert np.array_equal(C, ref["c_seq"])


def test_paired_sm_kernel_refuses_what_it_cannot_run(hb):
    A = to_dev(wl.draw("normal", (256, 256), seed=1))
    f8 = dict(mant_bits=8, block=128, rounding=0, seed=0)
    with pytest.raises(hb.HbfpError) as e:           # too few tiles to occupy the SM pairs
        hb.gemm(0, 0, A, A, gfmt(f8), gfmt(f8), flags=hb.GEMM_FORCE_TENSOR_2SM)
    assert e.value.code == hb.ERR_UNSUPPORTED
    big = to_dev(wl.draw("normal", (2560, 2048), seed=2))
    f12 = dict(mant_bits=12, block=64, rounding=0, seed=0)
    with pytest.raises(hb.HbfpError) as e:           # two mantissa planes
        hb.gemm(0, 1, big, big, gfmt(f12), gfmt(f12), flags=hb.GEMM_FORCE_TENSOR_2SM)
    assert e.value.code == hb.ERR_UNSUPPORTED


def test_mlp_step_captured_in_a_cuda_graph_replays_on_new_data(hb):
    """The calls are stream-ordered and allocate nothing when given their buffers, so a whole
    training step's GEMMs (stochastic rounding included: the draws depend on seed, stream id and
    element index only) can be captured once and replayed on new contents of the same tensors."""
    import torch
    specs = wl.config_mlp()
    t = wl.materialize(specs, seed=1)
    dev = {k: to_dev(v) for k, v in t.items()}
    outs = [torch.empty((sp.M, sp.N), dtype=torch.float32, device="cuda") for sp in specs]
    wss = [torch.empty(max(hb.gemm_workspace(sp.transA, sp.transB, sp.M, sp.N, sp.K, gfmt(sp.fmt_a), gfmt(sp.fmt_b)), 1),
                       dtype=torch.int8, device="cuda") for sp in specs]

    def step():
        for sp, C, ws in zip(specs, outs, wss):
            hb.gemm(sp.transA, sp.transB, dev[sp.a_key], dev[sp.b_key], gfmt(sp.fmt_a), gfmt(sp.fmt_b),
                    out=C, workspace=ws)

    step()                                   # eager: also sets the kernels' attributes once
    torch.cuda.synchronize()
    eager = [C.clone() for C in outs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    for C in outs:
        C.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert hb.device_status() == 0
    for sp, C, E in zip(specs, outs, eager):
        assert torch.equal(C, E), sp.name
    # new contents, same buffers: the replay must compute on them
    t2 = wl.materialize(specs, seed=5)
    for k, v in t2.items():
        dev[k].copy_(to_dev(v))
    graph.replay()
    torch.cuda.synchronize()
    assert hb.device_status() == 0
    for sp, C in zip(specs, outs):
        ref = oracle.hbfp_gemm(sp.transA, sp.transB, t2[sp.a_key], t2[sp.b_key], ofmt(sp.fmt_a), ofmt(sp.fmt_b))
        err = np.abs(C.cpu().numpy().astype(np.float64) - ref["c_ref"].astype(np.float64))
        assert (err <= TOL * ref["a_mag"]).all(), sp.name


@pytest.mark.parametrize("m,M,N,K", [(8, 128, 1024, 784), (8, 384, 512, 1024), (4, 200, 136, 1000), (12, 256, 256, 320)])
def test_one_exponent_per_row_no_blocks_no_tiles(hb, m, M, N, K):
    # "HBFP without tiles": block = 0, the whole contraction axis shares one exponent (one K-block per GEMM)
    A = wl.draw("half_normal", (M, K), seed=51)
    B = wl.draw("he_weight", (K, N), seed=52, fan_in=K)
    fd = dict(mant_bits=m, block=0, rounding=0, seed=0)
    ref = oracle.hbfp_gemm(0, 0, A, B, ofmt(fd), ofmt(fd))
    for flags in (hb.GEMM_FORCE_SIMT, hb.GEMM_AUTO):
        C = hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd), flags=flags).cpu().numpy()
        assert hb.device_status() == 0
        err = np.abs(C.astype(np.float64) - ref["c_ref"].astype(np.float64))
        assert (err <= TOL * ref["a_mag"]).all()
        assert np.array_equal(C, ref["c_seq"])          # a single block: one product, one rounding


@pytest.mark.parametrize("M,N,K", [(128, 10, 1024), (1024, 10, 128), (200, 137, 256), (300, 66, 96)])
def test_tensor_core_kernel_writes_outputs_of_any_width(hb, M, N, K):
    # an output whose row pitch is not a multiple of four floats (the MLP's ten-class layer) cannot take
    # 16-byte stores; the tensor-core kernel then stores element by element
    A = wl.draw("half_normal", (M, K), seed=61)
    B = wl.draw("he_weight", (K, N), seed=62, fan_in=K)
    fd = dict(mant_bits=8, block=32, rounding=0, seed=0)
    ref = oracle.hbfp_gemm(0, 0, A, B, ofmt(fd), ofmt(fd))
    C = hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd), flags=hb.GEMM_FORCE_TENSOR).cpu().numpy()
    assert hb.device_status() == 0
    err = np.abs(C.astype(np.float64) - ref["c_ref"].astype(np.float64))
    assert (err <= TOL * ref["a_mag"]).all()
    # a view into a wider buffer with an odd pitch and an odd column offset
    import torch
    buf = torch.full((M, N + 7), -1.0, device="cuda")
    hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd), out=buf[:, 3:3 + N], flags=hb.GEMM_FORCE_TENSOR)
    out = buf.cpu().numpy()
    assert np.array_equal(out[:, 3:3 + N], C) and (out[:, :3] == -1).all() and (out[:, 3 + N:] == -1).all()


def _range_case(hb, A, B, flag):
    """GEMM of two FP32 matrices (8-bit mantissas, blocks of 128) on the kernel `flag` selects: returns
    (status return code, result, oracle reference)."""
    fd = dict(mant_bits=8, block=128)
    ref = oracle.hbfp_gemm(0, 0, A, B, ofmt(fd), ofmt(fd, stream_id=1))
    C = hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd, stream_id=1), flags=flag).cpu().numpy()
    rc, code = hb.device_status_rc()
    return rc, code, C, ref


@pytest.mark.parametrize("kernel", ["1sm", "2sm"])
def test_large_magnitudes_are_computed_or_reported_never_silently_wrong(hb, kernel):
    """Operands far from 1: the tensor-core kernels factor the block scale 2^(sA + sB); outside the
    range in which that is exact they must say so through the device status word."""
    flag = hb.GEMM_FORCE_TENSOR_1SM if kernel == "1sm" else hb.GEMM_FORCE_TENSOR_2SM
    M, N, K = 2304, 2304, 256            # 81 pair tiles: enough for the paired kernel
    rng = np.random.default_rng(77)
    B = wl.draw("normal", (K, N), seed=78)
    # (1) |A| ~ 2^60, |B| ~ 1: inside binary32, outside a fixed split of the scale
    A = (wl.draw("normal", (M, K), seed=79) * np.float32(2.0 ** 60)).astype(np.float32)
    rc, code, C, ref = _range_case(hb, A, B, flag)
    assert rc == hb.OK and code == 0
    assert np.array_equal(C, ref["c_seq"])
    # (2) |A| ~ 2^115: products are still finite with |B| ~ 2^-40
    A2 = (wl.draw("normal", (M, K), seed=80) * np.float32(2.0 ** 115)).astype(np.float32)
    B2 = (B * np.float32(2.0 ** -40)).astype(np.float32)
    rc, code, C, ref = _range_case(hb, A2, B2, flag)
    if rc == hb.OK:
        assert np.array_equal(C, ref["c_seq"])
    else:
        assert rc == hb.ERR_EXPONENT_RANGE and 900 <= code < 1000
    # (3) rows of one tile 140 binades apart: no split of the scale serves both
    A3 = wl.draw("normal", (M, K), seed=81)
    A3[0::2] *= np.float32(2.0 ** 70)
    A3[1::2] *= np.float32(2.0 ** -70)
    rc, code, C, ref = _range_case(hb, A3.astype(np.float32), B, flag)
    if rc == hb.OK:
        err = np.abs(C.astype(np.float64) - ref["c_ref"].astype(np.float64))
        assert (err <= TOL * ref["a_mag"]).all()
    else:
        assert rc == hb.ERR_EXPONENT_RANGE and 900 <= code < 1000
    # the library is healthy afterwards
    rc, code, C, ref = _range_case(hb, wl.draw("normal", (M, K), seed=82), B, flag)
    assert rc == hb.OK and np.array_equal(C, ref["c_seq"])


def test_large_magnitudes_with_two_plane_mantissas_are_computed_or_reported(hb):
    """12-bit mantissas take the biased path of the single-SM kernel with a narrower exponent range
    (the bias is scaled by 256 * 2^sA): inside it the result is the oracle's, outside the status says so."""
    M, N, K = 384, 320, 256
    fd = dict(mant_bits=12, block=64)
    B = wl.draw("normal", (K, N), seed=178)
    for scale_a, scale_b in ((2.0 ** 60, 1.0), (2.0 ** 100, 2.0 ** -40), (2.0 ** 112, 2.0 ** -60), (1.0, 1.0)):
        A = (wl.draw("normal", (M, K), seed=179) * np.float32(scale_a)).astype(np.float32)
        Bs = (B * np.float32(scale_b)).astype(np.float32)
        ref = oracle.hbfp_gemm(0, 0, A, Bs, ofmt(fd), ofmt(fd, stream_id=1))
        C = hb.gemm(0, 0, to_dev(A), to_dev(Bs), gfmt(fd), gfmt(fd, stream_id=1), flags=hb.GEMM_FORCE_TENSOR_1SM).cpu().numpy()
        rc, code = hb.device_status_rc()
        if rc == hb.OK:
            assert np.array_equal(C, ref["c_seq"]), (scale_a, scale_b)
        else:
            assert scale_a > 2.0 ** 80 and rc == hb.ERR_EXPONENT_RANGE and 900 <= code < 1000
    assert rc == hb.OK            # the last, ordinary case ran clean


def test_a_bounded_wait_that_runs_out_is_reported_and_leaves_the_library_usable(hb):
    """The wait routine of the GEMM kernels, on a barrier nobody arrives on, with a budget of a few
    thousand cycles: the status word carries the code, the next read is clean, the next GEMM is right."""
    assert hb.device_status() == 0
    assert hb.selftest_bounded_wait(limit_cycles=5000, code=777) == 2      # abandoned, abort flag raised
    assert hb.device_status_rc() == (hb.ERR_TIMEOUT, 777)
    assert hb.device_status_rc() == (hb.OK, 0)
    specs = wl.config_single_256()
    run_spec(hb, specs[0], wl.materialize(specs, seed=0), hb.GEMM_AUTO)


def test_last_gemm_cycles_reports_the_paired_kernel_length(hb):
    """hbfp_last_gemm_cycles: the paired-SM kernel's length in SM cycles (longest CTA), a plausible number of them."""
    import torch
    n = 4096
    f = hb.Format(8, 128)
    A = to_dev(wl.draw("lognormal", (n, n), seed=71))
    pa, pb = hb.quantize(A, 1, f), hb.quantize(A, 0, f)
    ws = torch.empty(max(hb.gemm_q_workspace(n, n, n, pa, pb), 1), dtype=torch.int8, device="cuda")
    out = torch.empty((n, n), dtype=torch.float32, device="cuda")
    s, e = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    hb.gemm_q(n, n, n, pa, pb, out=out, workspace=ws, flags=hb.GEMM_FORCE_TENSOR_2SM)
    s.record()
    hb.gemm_q(n, n, n, pa, pb, out=out, workspace=ws, flags=hb.GEMM_FORCE_TENSOR_2SM)
    e.record()
    torch.cuda.synchronize()
    assert hb.last_gemm_kernel() == "gemm_tc2_kernel"
    cycles = hb.last_gemm_cycles()
    mhz = cycles / s.elapsed_time(e) / 1e3
    # 32 K-blocks x 4 tiles per cluster at several hundred cycles each; a clock between 0.5 and 2.2 GHz
    assert 32 * 4 * 300 < cycles < 32 * 4 * 20000
    assert 500 < mhz < 2200
    assert hb.device_status() == 0


def test_last_gemm_cycles_counts_from_the_kernels_start(hb):
    """A launch of one K-block and one tile per cluster: 5900 cycles, 2600 of them before the work begins (barriers, tensor memory, both
    SMs of each pair ready); without those it would be 3300."""
    import torch
    f = hb.Format(8, 128)
    a, b = hb.quantize(torch.randn(9472, 128, device="cuda"), 1, f), hb.quantize(torch.randn(512, 128, device="cuda"), 1, f)
    cycles = []
    for _ in range(9):
        hb.gemm_q(9472, 512, 128, a, b, flags=hb.GEMM_FORCE_TENSOR_2SM)
        cycles.append(hb.last_gemm_cycles())
    assert 4600 < sorted(cycles)[4] < 12000


# The floating-point operand forms (gemm_fp.cu): short blocks of 8-bit mantissas, 9 to 12 bits; one SM or a pair per tile.
# Edges of tiles in M and N, a last K stage with a single block, padded blocks, an output pitch that TMA cannot store.
FP_FORM_CASES = [
    # m, block, M, N, K, law, kernel
    (8, 32, 2304, 2176, 1760, "lognormal", "gemm_fp_kernel"),
    (8, 24, 2305, 2051, 1751, "lognormal", "gemm_fp_kernel"),
    (8, 64, 2304, 2310, 1664, "normal", "gemm_fp_kernel"),
    (8, 64, 2433, 3071, 1602, "lognormal", "gemm_fp_kernel/pair"),
    (6, 48, 2433, 2177, 1700, "lognormal", "gemm_fp_kernel"),
    (12, 32, 2176, 2050, 1888, "outliers", "gemm_fp_kernel"),
    (12, 64, 2433, 2303, 1600, "lognormal", "gemm_fp_kernel/pair"),
    (10, 40, 2177, 2052, 1990, "normal", "gemm_fp_kernel"),
]


@pytest.mark.parametrize("m,b,M,N,K,law,kernel", FP_FORM_CASES)
def test_floating_point_operand_forms_are_bit_equal_to_the_sequential_definition(hb, m, b, M, N, K, law, kernel):
    """Block sums are exact in every form and blocks are added in ascending order with one rounding each, so without
    split-K the result is the reference kernel's (gemm_simt, itself bit-equal to the oracle's c_seq) bit for bit;
    the largest mantissas everywhere give the largest block sums."""
    import torch
    fa, fb = hb.Format(m, b, rounding=1, seed=3), hb.Format(m, b, rounding=1, seed=3, stream_id=1)
    A, B = to_dev(wl.draw(law, (M, K), seed=91)), to_dev(wl.draw(law, (K, N), seed=92))
    for X, Y in ((A, B), (torch.full_like(A, 1.999), torch.full_like(B, -1.999))):
        pa, pb = hb.quantize(X, 1, fa), hb.quantize(Y, 0, fb)
        want = hb.gemm_q(M, N, K, pa, pb, flags=hb.GEMM_FORCE_SIMT)
        buf = torch.full((M, N + 3), 7.0, device="cuda")
        for out in (None, buf[:, 1:1 + N]):
            got = hb.gemm(0, 0, X, Y, fa, fb, out=out)
            assert hb.last_gemm_launch() == kernel and hb.device_status() == 0
            assert torch.equal(got, want)
            assert torch.equal(hb.gemm_q(M, N, K, pa, pb, out=out), want) and hb.last_gemm_launch() == kernel
        assert bool((buf[:, 0] == 7).all()) and bool((buf[:, N + 1:] == 7).all())


@pytest.mark.parametrize("m,b,M,N,K,rounding", [(8, 24, 1, 1, 100, 1), (8, 32, 130, 70, 1024, 0), (8, 64, 16, 4096, 4096, 1), (12, 64, 129, 65, 2048, 1),
                                                (12, 24, 257, 10, 700, 0), (8, 32, 640, 500, 33, 1), (5, 40, 1000, 260, 900, 0)])
@pytest.mark.parametrize("tA,tB", [(0, 0), (1, 1)])
def test_small_products_of_fp32_operands_converted_straight_to_the_form(hb, m, b, M, N, K, rounding, tA, tB):
    """FP32 operands of both storage orders, few tiles, K split over the CTAs of a cluster: within 1e-6 of the accumulator
    magnitude of the product of the packed operands."""
    import torch
    A = to_dev(wl.draw("outliers", (K, M) if tA else (M, K), seed=95))
    B = to_dev(wl.draw("normal", (N, K) if tB else (K, N), seed=96))
    fa, fb = hb.Format(m, b, rounding=rounding, seed=6), hb.Format(m, b, rounding=rounding, seed=6, stream_id=1)
    C = hb.gemm(tA, tB, A, B, fa, fb, flags=hb.GEMM_FORCE_TENSOR)
    assert hb.last_gemm_launch() == ("gemm_fp_kernel" if K < 256 else "gemm_fp_kernel/split")
    pa, pb = hb.quantize(A, 0 if tA else 1, fa), hb.quantize(B, 1 if tB else 0, fb)
    da, db = hb.dequantize(pa).double(), hb.dequantize(pb).double()
    assert hb.device_status() == 0
    assert bool(((C.double() - da @ db.t()).abs() <= TOL * (da.abs() @ db.abs().t()) + 1e-30).all())


@pytest.mark.parametrize("m,b,M,N,K", [(8, 24, 600, 520, 1700), (8, 24, 1111, 777, 3001), (8, 32, 640, 1280, 2048), (8, 64, 900, 500, 1300), (12, 24, 600, 520, 1700),
                                       (12, 24, 1000, 600, 1000), (8, 32, 650, 330, 900), (8, 32, 640, 500, 2600), (8, 64, 511, 385, 3300)])
def test_contraction_split_over_clusters_of_any_size(hb, m, b, M, N, K):
    """K split over clusters of 2 to 7 CTAs, last parts shorter than the others: within 1e-6 of the accumulator magnitude."""
    A, B = to_dev(wl.draw("outliers", (M, K), seed=97)), to_dev(wl.draw("lognormal", (K, N), seed=98))
    fa, fb = hb.Format(m, b), hb.Format(m, b, stream_id=1)
    C = hb.gemm(0, 0, A, B, fa, fb)
    da, db = (hb.dequantize(hb.quantize(x, ax, f)).double() for x, ax, f in ((A, 1, fa), (B, 0, fb)))
    assert hb.device_status() == 0 and hb.last_gemm_launch() == "gemm_fp_kernel/split"
    assert bool(((C.double() - da @ db.t()).abs() <= TOL * (da.abs() @ db.abs().t()) + 1e-30).all())


@pytest.mark.parametrize("M,N,K,m,t,rounding", [(1, 1, 1, 8, 32, 0), (16, 4096, 4096, 8, 64, 0), (17, 129, 128, 8, 128, 1), (5, 1000, 777, 8, 24, 1), (32, 127, 3001, 8, 48, 1),
                                                (33, 640, 513, 4, 32, 0), (64, 300, 8192, 8, 128, 1), (128, 10, 1024, 8, 24, 1), (100, 900, 1000, 6, 40, 0), (16, 256, 11000, 8, 32, 0)])
def test_few_rows_against_packed_weights_in_one_launch(hb, M, N, K, m, t, rounding):
    """Conversion, product and sum over K in one kernel: edges of the 128 weight rows and of the 16, 32 and 64 activation rows,
    blocks with padding, odd row lengths, more blocks than tensor memory holds, an output that starts at an odd column. Within
    1e-6 of the accumulator magnitude of the product of what hbfp_quantize makes of the same operand."""
    import torch
    X, W = to_dev(wl.draw("outliers", (M, K), seed=71)), to_dev(wl.draw("he_weight", (K, N), seed=72, fan_in=K))
    fx = hb.Format(mant_bits=m, block=t, rounding=rounding, seed=3)
    c0 = hb.quantize_tiles(W, hb.Format(mant_bits=m, block=t, tile=t, rounding=rounding, seed=3, stream_id=1), want_grid=False)[0]
    dx, dw = hb.dequantize(hb.quantize(X, 1, fx)).double(), hb.dequantize(c0).double()
    want, mag = dx @ dw.t(), dx.abs() @ dw.abs().t()
    buf = torch.full((M, N + 3), 7.0, device="cuda")
    for out in (None, buf[:, 1:1 + N]):
        got = hb.gemm_q(M, N, K, X, c0, fmtA=fx, out=out)
        assert hb.last_gemm_launch() == "gemm_skinny_kernel" and hb.device_status() == 0
        assert bool(((got.double() - want).abs() <= TOL * mag + 1e-30).all())
    assert bool((buf[:, 0] == 7).all()) and bool((buf[:, N + 1:] == 7).all())


def test_few_rows_kernel_reports_weights_beyond_its_exact_range(hb):
    """P * 2^sB leaves binary32 above sB = 104: the oracle's values or the status, nothing else."""
    M, N, K, t = 4, 160, 1024, 64
    X, W = wl.draw("normal", (M, K), seed=73), wl.draw("normal", (K, N), seed=74)
    fx, fw = hb.Format(8, t), hb.Format(8, t, tile=t, stream_id=1)
    for scale_x, scale_w in ((2.0 ** -60, 2.0 ** 100), (2.0 ** 100, 2.0 ** -60), (2.0 ** -100, 2.0 ** 118)):
        x, w = to_dev(X * np.float32(scale_x)), to_dev(W * np.float32(scale_w))
        c0 = hb.quantize_tiles(w, fw, want_grid=False)[0]
        got = hb.gemm_q(M, N, K, x, c0, fmtA=fx)
        assert hb.last_gemm_kernel() == "gemm_skinny_kernel"
        want = hb.dequantize(hb.quantize(x, 1, fx)).double() @ hb.dequantize(c0).double().t()
        if hb.device_status() == 0:
            assert bool(((got.double() - want).abs() <= 1e-5 * want.abs().max()).all())
        else:
            assert scale_w > 2.0 ** 110


@pytest.mark.parametrize("M,N,K,m,b,rounding", [(256, 256, 256, 8, 32, 0), (1, 1, 1, 8, 32, 1), (33, 65, 100, 8, 24, 0), (40, 72, 130, 4, 48, 1), (64, 96, 512, 8, 128, 1),
                                                (31, 200, 384, 8, 24, 1), (100, 36, 511, 6, 64, 0), (256, 512, 200, 8, 100, 1)])
@pytest.mark.parametrize("tA,tB", [(0, 0), (1, 0), (0, 1), (1, 1)])
def test_small_products_of_fp32_operands_in_one_launch(hb, M, N, K, m, b, rounding, tA, tB):
    """Both operands converted inside the product, in every storage order, at unaligned rows and ragged blocks: bit for bit the
    reference kernel on what hbfp_quantize makes of them."""
    import torch
    A = to_dev(wl.draw("outliers", (K, M) if tA else (M, K), seed=51))
    B = to_dev(wl.draw("lognormal", (N, K) if tB else (K, N), seed=52))
    fa, fb = hb.Format(m, b, rounding=rounding, seed=9), hb.Format(m, b, rounding=rounding, seed=9, stream_id=1)
    want = hb.gemm_q(M, N, K, hb.quantize(A, 0 if tA else 1, fa), hb.quantize(B, 1 if tB else 0, fb), flags=hb.GEMM_FORCE_SIMT)
    for X in (A, torch.cat([A, A], 1)[:, 1:1 + A.shape[1]] if A.shape[1] > 1 else A):
        fresh = X is A
        if not fresh:
            want = hb.gemm_q(M, N, K, hb.quantize(X.contiguous(), 0 if tA else 1, fa), hb.quantize(B, 1 if tB else 0, fb), flags=hb.GEMM_FORCE_SIMT)
        got = hb.gemm(tA, tB, X, B, fa, fb)
        # draws down columns need whole groups of eight lines
        fused = rounding == 0 or not ((tA and M % 8) or (not tB and N % 8))
        assert hb.last_gemm_launch() == ("gemm_small_fused_kernel" if fused else "gemm_small_kernel") and hb.device_status() == 0
        assert torch.equal(got, want)


@pytest.mark.parametrize("first,second", [((32, 4096, 4096, 64), (16, 4096, 1024, 64)), ((64, 2048, 2048, 64), (64, 4096, 1024, 64)), ((1, 2048, 4096, 24), (1, 512, 512, 24))])
def test_few_rows_kernels_of_different_plans_run_on_two_streams(hb, first, second):
    """Two launches whose CTAs fit an SM by shared memory but not by tensor memory (512 and 32, 256 and 128, 512 and 64 columns), on
    two streams at once: a CTA gives its columns back before it waits for its cluster, so both finish, with the bits of a run alone."""
    import torch
    work = []
    for k, (M, N, K, t) in enumerate((first, second)):
        X, W = to_dev(wl.draw("normal", (M, K), seed=110 + k)), to_dev(wl.draw("he_weight", (K, N), seed=120 + k, fan_in=K))
        fx = hb.Format(8, t)
        c0 = hb.quantize_tiles(W, hb.Format(8, t, tile=t, stream_id=1), want_grid=False)[0]
        alone = hb.gemm_q(M, N, K, X, c0, fmtA=fx)
        assert hb.last_gemm_kernel() == "gemm_skinny_kernel"
        ws = torch.empty(max(hb.gemm_q_workspace(M, N, K, X, c0, fmtA=fx), 1), dtype=torch.int8, device="cuda")
        work.append((torch.cuda.Stream(), alone, [torch.empty_like(alone) for _ in range(64)], lambda o, a=(M, N, K, X, c0), f=fx, w=ws: hb.gemm_q(*a, fmtA=f, out=o, workspace=w)))
    torch.cuda.synchronize()
    for i in range(64):
        for stream, _, outs, call in work:
            with torch.cuda.stream(stream):
                call(outs[i])
    torch.cuda.synchronize()
    assert hb.device_status() == 0
    for _, alone, outs, _ in work:
        assert all(torch.equal(o, alone) for o in outs)


# Calls of several launches each, placed early behind one another, on two streams at once: both conversions beside each other, forms
# (split, in pairs), integer kernels with and without split-K, the smallest products.
@pytest.mark.parametrize("first,second", [
    ((1111, 777, 3001, 8, 24), (512, 512, 4096, 8, 32)), ((2048, 2304, 512, 12, 64), (2304, 2304, 1024, 8, 128)), ((300, 200, 4000, 8, 128), (2048, 2304, 512, 8, 64)),
    ((64, 96, 128, 8, 32), (1024, 1024, 1024, 8, 32))])
def test_products_of_fp32_operands_on_two_streams(hb, first, second):
    import torch
    work = []
    for k, (M, N, K, m, b) in enumerate((first, second)):
        A, B = to_dev(wl.draw("normal", (M, K), seed=130 + k)), to_dev(wl.draw("outliers", (K, N), seed=140 + k))
        fa, fb = hb.Format(m, b, rounding=1, seed=4), hb.Format(m, b, rounding=1, seed=4, stream_id=1)
        alone = hb.gemm(0, 0, A, B, fa, fb)
        ws = torch.empty(max(hb.gemm_workspace(0, 0, M, N, K, fa, fb), 1), dtype=torch.int8, device="cuda")
        work.append((torch.cuda.Stream(), alone, [torch.empty_like(alone) for _ in range(48)], lambda o, a=(0, 0, A, B, fa, fb), w=ws: hb.gemm(*a, out=o, workspace=w)))
    torch.cuda.synchronize()
    for i in range(48):
        for stream, _, outs, call in work:
            with torch.cuda.stream(stream):
                call(outs[i])
    torch.cuda.synchronize()
    assert hb.device_status() == 0
    for _, alone, outs, _ in work:
        assert all(torch.equal(o, alone) for o in outs)


@pytest.mark.parametrize("M,N,K", [(128, 128, 256), (600, 520, 1700), (2304, 2176, 1760)])
def test_scaled_operand_form_reports_products_beyond_binary32(hb, M, N, K):
    """Products of 2^129 that cancel to 2^122 within a block, in one of its MMA steps or across two: the sum is representable, and the
    kernel leaves it or records the status, on the way from FP32 operands and from packed ones."""
    import torch
    fa, fb = hb.Format(8, 32), hb.Format(8, 32, stream_id=1)
    a, b = torch.zeros(M, K, device="cuda"), torch.zeros(K, N, device="cuda")
    a[:, :32] = 127.0 * 2.0 ** 57
    for k in (1, 16):
        b.zero_()
        b[0], b[k] = 127.0 * 2.0 ** 58, -126.0 * 2.0 ** 58
        pa, pb = hb.quantize(a, 1, fa), hb.quantize(b, 0, fb)
        want = hb.gemm_q(M, N, K, pa, pb, flags=hb.GEMM_FORCE_SIMT)
        assert bool((want == 127.0 * 2.0 ** 115).all())
        for call in (lambda: hb.gemm(0, 0, a, b, fa, fb, flags=hb.GEMM_FORCE_TENSOR), lambda: hb.gemm_q(M, N, K, pa, pb, flags=hb.GEMM_FORCE_TENSOR)):
            got, rc = call(), hb.device_status_rc()[0]
            assert rc == hb.ERR_EXPONENT_RANGE or (rc == hb.OK and torch.equal(got, want))
    for scale in (2.0 ** 50, 2.0 ** -60):          # far inside the range nothing is recorded
        hb.gemm(0, 0, torch.randn_like(a) * scale, torch.randn_like(b), fa, fb, flags=hb.GEMM_FORCE_TENSOR)
        assert hb.device_status() == 0


@pytest.mark.parametrize("M,N,K", [(128, 10, 1024), (1024, 10, 128), (200, 137, 256), (300, 66, 96)])
@pytest.mark.parametrize("b", [32, 128])
def test_integer_tensor_core_kernel_writes_outputs_of_any_width(hb, M, N, K, b):
    """The single-SM integer kernel at pitches that cannot take 16-byte stores (GEMM_FORCE_TENSOR goes to the operand forms where
    blocks are short, this flag does not)."""
    import torch
    A, B = wl.draw("half_normal", (M, K), seed=61), wl.draw("he_weight", (K, N), seed=62, fan_in=K)
    fd = dict(mant_bits=8, block=b, rounding=0, seed=0)
    ref = oracle.hbfp_gemm(0, 0, A, B, ofmt(fd), ofmt(fd))
    buf = torch.full((M, N + 7), -1.0, device="cuda")
    for out in (None, buf[:, 3:3 + N]):
        C = hb.gemm(0, 0, to_dev(A), to_dev(B), gfmt(fd), gfmt(fd), out=out, flags=hb.GEMM_FORCE_TENSOR_1SM).cpu().numpy()
        assert hb.last_gemm_launch() == "gemm_tc_kernel" and hb.device_status() == 0
        assert (np.abs(C.astype(np.float64) - ref["c_ref"].astype(np.float64)) <= TOL * ref["a_mag"]).all()
    assert bool((buf[:, :3] == -1).all()) and bool((buf[:, 3 + N:] == -1).all())


@pytest.mark.parametrize("M,N,K,m,b", [(128, 200, 10865, 8, 64), (64, 56, 12416, 12, 32), (208, 384, 52072, 8, 64)])
def test_few_tiles_with_a_long_contraction_take_the_integer_kernel(hb, M, N, K, m, b):
    """More parts of K than a cluster has CTAs: split over the whole chip, and faster by a fifth to a third than the operand forms."""
    A, B = to_dev(wl.draw("normal", (M, K), seed=131)), to_dev(wl.draw("normal", (K, N), seed=132))
    fa, fb = hb.Format(m, b), hb.Format(m, b, stream_id=1)
    C = hb.gemm(0, 0, A, B, fa, fb)
    assert hb.last_gemm_launch() == "gemm_tc_kernel" and hb.device_status() == 0
    da, db = hb.dequantize(hb.quantize(A, 1, fa)).double(), hb.dequantize(hb.quantize(B, 0, fb)).double()
    assert bool(((C.double() - da @ db.t()).abs() <= TOL * (da.abs() @ db.abs().t()) + 1e-30).all())


@pytest.mark.parametrize("M,N,K,tA,rounding,fused", [(512, 512, 256, 0, 1, False), (512, 512, 256, 0, 0, True), (512, 512, 128, 0, 1, True), (256, 448, 448, 1, 1, False), (256, 448, 448, 0, 1, True),
                                                     (256, 256, 448, 1, 1, True), (256, 256, 256, 1, 1, True)])
def test_small_products_with_draws_in_one_launch_or_three(hb, M, N, K, tA, rounding, fused):
    """Where tiles repeat the draws too often the operands are converted on their own: the same bits either way."""
    import torch
    A, B = to_dev(wl.draw("normal", (K, M) if tA else (M, K), seed=141)), to_dev(wl.draw("normal", (K, N), seed=142))
    fa, fb = hb.Format(8, 32, rounding=rounding, seed=4), hb.Format(8, 32, rounding=rounding, seed=4, stream_id=1)
    got = hb.gemm(tA, 0, A, B, fa, fb)
    assert hb.last_gemm_launch() == ("gemm_small_fused_kernel" if fused else "gemm_small_kernel") and hb.device_status() == 0
    assert torch.equal(got, hb.gemm_q(M, N, K, hb.quantize(A, 0 if tA else 1, fa), hb.quantize(B, 0, fb), flags=hb.GEMM_FORCE_SIMT))


@pytest.mark.parametrize("m,b,tiles", [(8, 32, (0, 0)), (8, 64, (0, 1)), (12, 64, (1, 0)), (8, 32, (1, 1)), (12, 32, (1, 1))])
def test_operand_forms_stay_inside_the_workspace_they_ask_for(hb, m, b, tiles):
    """Operands converted straight to their form and, with weight tiles, by way of packed copies that share one place: the reference
    kernel's bits, and the bytes behind the workspace untouched."""
    import torch
    M, N, K = 2433, 2177, 1700
    A, B = to_dev(wl.draw("lognormal", (M, K), seed=151)), to_dev(wl.draw("normal", (K, N), seed=152))
    fa, fb = (hb.Format(m, b, tile=b * t, rounding=1, seed=2, stream_id=k) for k, t in enumerate(tiles))
    need = hb.gemm_workspace(0, 0, M, N, K, fa, fb)
    ws = torch.full((need + 4096,), 55, dtype=torch.int8, device="cuda")
    got = hb.gemm(0, 0, A, B, fa, fb, workspace=ws[:need])
    assert hb.last_gemm_launch().startswith("gemm_fp_kernel") and hb.device_status() == 0
    assert bool((ws[need:] == 55).all())
    assert torch.equal(got, hb.gemm_q(M, N, K, hb.quantize(A, 1, fa), hb.quantize(B, 0, fb), flags=hb.GEMM_FORCE_SIMT))


# Kernels of a stream are placed before their predecessors have ended, and the second operand is converted beside the first: calls
# that follow one another without a pause, over buffers that are rewritten between them, give what each gives alone. Routes: small
# fused, forms (row and column conversions, split over clusters, pairs), integer kernels with and without split-K, few rows against
# weights updated just before, whole-axis blocks.
@pytest.mark.parametrize("M,N,K,m,b,rounding,tA,packed", [
    (64, 96, 128, 8, 32, 1, 0, False), (1111, 777, 301, 8, 24, 1, 0, False), (512, 512, 4096, 8, 32, 0, 1, False), (2048, 2560, 256, 12, 64, 1, 0, False),
    (300, 200, 4000, 8, 128, 0, 1, False), (2304, 2304, 1024, 8, 128, 0, 0, False), (130, 70, 1000, 8, 0, 0, 1, False), (512, 300, 24, 8, 24, 1, 0, False),
    (16, 512, 768, 8, 64, 0, 0, True), (700, 512, 768, 12, 64, 1, 0, True), (700, 512, 768, 8, 128, 0, 0, True)])
def test_calls_in_a_row_give_what_each_gives_alone(hb, M, N, K, m, b, rounding, tA, packed):
    import torch
    fa, fb = hb.Format(mant_bits=m, block=b, rounding=rounding, seed=3), hb.Format(mant_bits=m, block=b, rounding=rounding, seed=3, stream_id=1)
    fw = hb.Format(mant_bits=m, block=b, tile=b, rounding=rounding, seed=3, stream_id=1)
    gen = torch.Generator(device="cuda").manual_seed(7)
    new = lambda *shape: torch.randn(*shape, device="cuda", generator=gen)
    As = [new(K, M) if tA else new(M, K) for _ in range(4)]
    Bs = [new(K, N) * 0.1 for _ in range(4)]

    def run(pause):
        A, B = torch.empty_like(As[0]), torch.empty_like(Bs[0])
        wide, views = hb.wide_quantize(Bs[0], fw) if packed else (None, None)
        out = []
        for i in range(12):
            A.copy_(As[i % 4])
            B.copy_(Bs[(i + i // 4) % 4])
            if pause: torch.cuda.synchronize()
            if packed: hb.wide_update(wide, B, fw, views=views)
            if pause: torch.cuda.synchronize()
            for _ in range(2):
                out.append(hb.gemm_q(M, N, K, A, views[0], fmtA=fa) if packed else hb.gemm(tA, 0, A, B, fa, fb))
                if pause: torch.cuda.synchronize()
        return out

    want = run(True)
    for _ in range(4):
        assert all(torch.equal(x, y) for x, y in zip(run(False), want))
    assert hb.device_status() == 0


def edges_in_order(graph) -> list:
    """The kinds of the edges of a captured chain of nodes, from its first node on: 0 the whole of the node before, 1 programmatic."""
    import ctypes
    driver, raw, n = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t()
    assert driver.cuGraphGetEdges_v2(raw, None, None, None, ctypes.byref(n)) == 0
    source, target, data = (ctypes.c_uint64 * n.value)(), (ctypes.c_uint64 * n.value)(), (ctypes.c_uint8 * 8 * n.value)()
    assert driver.cuGraphGetEdges_v2(raw, source, target, data, ctypes.byref(n)) == 0
    step = {a: (b, d[2]) for a, b, d in zip(source, target, data)}         # third byte of CUgraphEdgeData: the type
    assert len(step) == n.value                                 # one way through
    (at,) = set(step) - {b for b, _ in step.values()}
    kinds = []
    while at in step:
        at, kind = step[at]
        kinds.append(kind)
    return kinds


# The second conversion runs beside the first, the product is placed early, but for long launches of the 12-bit form.
@pytest.mark.parametrize("n,m,b,chained", [(2048, 8, 32, 1), (4096, 8, 32, 1), (4096, 8, 24, 1), (4096, 8, 64, 1), (2048, 12, 64, 1), (4096, 12, 64, 0), (4096, 12, 24, 0)])
def test_products_of_operand_forms_are_placed_early(hb, n, m, b, chained):
    import torch
    f = hb.Format(mant_bits=m, block=b)
    A, C, ws = torch.randn(n, n, device="cuda"), torch.empty(n, n, device="cuda"), torch.empty(1 << 28, dtype=torch.int8, device="cuda")
    hb.gemm(0, 0, A, A, f, f, C, ws)
    assert hb.last_gemm_launch().startswith("gemm_fp_kernel")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        hb.gemm(0, 0, A, A, f, f, C, ws)
    assert edges_in_order(graph) == [1, chained]


# Kernels that load much through L1 are not placed behind a product, which leaves them little of it, nor are a few long CTAs; others are,
# and those behind others.
@pytest.mark.parametrize("rows,op,chained", [(1024, "rows", 1), (8192, "rows", 0), (1024, "columns", 1), (8192, "columns", 0), (1024, "update", 1), (4096, "update", 0), (512, "long update", 0), (8192, "value", 0)])
def test_long_kernels_and_long_ctas_are_not_placed_behind_a_product(hb, rows, op, chained):
    import torch
    t = 128 if op == "long update" else 64
    f, fw = hb.Format(block=24 if op == "columns" else 64), hb.Format(block=t, tile=t)
    pa, pb = hb.quantize(torch.randn(512, 256, device="cuda"), 1, f), hb.quantize(torch.randn(512, 256, device="cuda"), 1, f)
    x, C, ws = torch.randn(rows, 4096, device="cuda"), torch.empty(512, 512, device="cuda"), torch.empty(1 << 24, dtype=torch.int8, device="cuda")
    out = hb.quantize(x, 0 if op == "columns" else 1, f)
    wide, views = hb.wide_quantize(x, fw)
    other = torch.empty_like(x)

    def kernel():
        if op == "rows": hb.quantize(x, 1, f, out)
        elif op == "columns": hb.quantize(x, 0, f, out)
        elif op.endswith("update"): hb.wide_update(wide, x, fw, views=views)
        else: hb.wide_dequantize(wide, other)

    def steps():
        hb.gemm_q(512, 512, 256, pa, pb, out=C, workspace=ws)
        kernel()
        kernel()

    steps()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        steps()
    assert edges_in_order(graph)[-2:] == [chained, 1]


# Routes in which the second operand is converted beside the first, on an operand that the kernel before has just written: packed
# weights of an update in place, the FP32 value of wide weights.
# Replayed too: the word through which the first conversion passes on what it has waited for starts every replay anew.
@pytest.mark.parametrize("m,b,N", [(8, 32, 2304), (8, 64, 2304), (12, 64, 2304), (12, 32, 2304), (8, 24, 2307), (12, 24, 2307)])
@pytest.mark.parametrize("kind", ["packed weights", "both packed", "fp32"])
def test_products_of_operands_that_the_kernel_before_has_written(hb, m, b, N, kind):
    import torch
    M, K = 2048, 2048
    fa, fb = hb.Format(mant_bits=m, block=b), hb.Format(mant_bits=m, block=b, stream_id=1)
    fw = hb.Format(mant_bits=m, block=b, tile=b, stream_id=1)
    gen = torch.Generator(device="cuda").manual_seed(9)
    A = torch.randn(M, K, device="cuda", generator=gen)
    w0 = torch.randn(K, N, device="cuda", generator=gen) * 0.05
    deltas = [torch.randn(K, N, device="cuda", generator=gen) * 0.05 for _ in range(3)]
    pa = hb.quantize(A, 1, fa) if kind == "both packed" else A

    def run(pause):
        wide, views = hb.wide_quantize(w0, fw)
        W = torch.empty(K, N, device="cuda")
        out = []
        for i in range(12):
            if kind == "fp32":
                hb.wide_update(wide, deltas[i % 3], fw, want_views=False)
                hb.wide_dequantize(wide, W)
            else:
                hb.wide_update(wide, deltas[i % 3], fw, views=views)
            if pause: torch.cuda.synchronize()
            out.append(hb.gemm(0, 0, A, W, fa, fb) if kind == "fp32" else hb.gemm_q(M, N, K, pa, views[0], fmtA=fa))
            if pause: torch.cuda.synchronize()
        return out

    want = run(True)
    assert hb.last_gemm_launch().startswith("gemm_fp_kernel")
    for _ in range(4):
        assert all(torch.equal(x, y) for x, y in zip(run(False), want))
    wide, views = hb.wide_quantize(w0, fw)
    W, C, ws, delta = torch.empty(K, N, device="cuda"), torch.empty(M, N, device="cuda"), torch.empty(1 << 27, dtype=torch.int8, device="cuda"), deltas[0].clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        if kind == "fp32":
            hb.wide_update(wide, delta, fw, want_views=False)
            hb.wide_dequantize(wide, W)
            hb.gemm(0, 0, A, W, fa, fb, C, ws)
        else:
            hb.wide_update(wide, delta, fw, views=views)
            hb.gemm_q(M, N, K, pa, views[0], fmtA=fa, out=C, workspace=ws)
    got = []
    for i in range(12):
        delta.copy_(deltas[i % 3])
        graph.replay()
        got.append(C.clone())
    assert all(torch.equal(x, y) for x, y in zip(got, want))
    assert hb.device_status() == 0
