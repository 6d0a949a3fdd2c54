"""The TMA-store epilogue of single GEMMs and the programs it runs in
registers: ragged edges of every tile shape, one to many segments per warp,
one and two staging boxes, four and eight epilogue warps, canary-padded
outputs; and the elementwise steps on their own over FP32's range.

Small-integer operands make the contraction exact, so everything up to the
program is bitwise.  A transcendental step is held to 4e-7 relative per
element: 2^-24 for each of the handful of roundings in a step of the form
x * f(x), a little under seven of them (the tanh form of GELU, whose argument
has roundings of its own that the exponential amplifies for large negative x,
is not among them)."""
import math

import numpy as np
import pytest
import torch

import oracle.nk_oracle as O
from paper_2307_16080_gb300 import synth
from tests.gpu_util import DEV, Canary, dev, host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nk():
    import paper_2307_16080_gb300.nk as m
    m.lib()
    return m


TILES = {"bf16": [(256, 512, 64, 2, 4, 1), (256, 256, 64, 2, 4, 1), (128, 256, 64, 1, 4, 1), (128, 128, 64, 1, 3, 1),
                  (128, 64, 64, 1, 3, 1), (256, 128, 64, 2, 3, 1)],
         "fp8": [(256, 512, 128, 2, 4, 1), (128, 256, 128, 1, 4, 1)],
         "bf16x3": [(128, 128, 64, 1, 3, 1), (256, 128, 64, 2, 3, 1), (128, 64, 64, 1, 3, 1)]}


@pytest.mark.parametrize("prec,sched", [(p, s) for p in TILES for s in TILES[p]])
@pytest.mark.parametrize("M,N,K", [(1, 4, 8), (129, 36, 72), (257, 516, 40), (300, 772, 136), (640, 1028, 64)])
def test_epilogue_edges_bitwise(nk, prec, sched, M, N, K):
    # half-integers up to 3.5, which both operands contain: exact in BF16, and
    # E4M3's scale is 448 / 3.5 = 128, so its codes and 1 / 128^2 are exact too
    A, B = synth.small_ints(901, 0, (M, K), -7, 7) / 2, synth.small_ints(901, 1, (K, N), -7, 7) / 2
    A[0, 0] = B[0, 0] = 3.5
    bias, T = synth.small_ints(901, 2, (N,)), synth.small_ints(901, 3, (M, N))
    relu = np.maximum(A.astype(np.float64) @ B + bias, 0)
    for prog in (False, True):
        C = Canary((M, N), strides=(N + 8, 1))
        ew, want = None, relu
        if prog:
            t = torch.empty_strided((M, N), (N + 8, 1), device=DEV)
            t.copy_(dev(T))
            ew, want = [("add", t), ("affine", 0.5, 1.0), ("clamp", -6.0, 90.0)], np.clip((relu + T) * 0.5 + 1, -6, 90)
        nk.nk_matmul(dev(A), dev(B), C.t, prec, bias=dev(bias), relu=True, schedule=sched, ew=ew)
        nk.nk_sync_status()
        assert np.array_equal(host(C.t), want.astype(np.float32))
        C.check()


@pytest.mark.parametrize("sched", TILES["bf16"])
def test_accumulate_reads_the_whole_segment_first(nk, sched):
    M, N, K = 300, 772, 72
    A, B, C0 = synth.small_ints(903, 0, (M, K)), synth.small_ints(903, 1, (K, N)), synth.small_ints(903, 2, (M, N))
    C = Canary((M, N), strides=(N + 8, 1))
    C.t.copy_(dev(C0))
    nk.nk_matmul(dev(A), dev(B), C.t, "bf16", schedule=sched, accumulate=True)
    nk.nk_sync_status()
    assert np.array_equal(host(C.t), (A.astype(np.float64) @ B + C0).astype(np.float32))
    C.check()


def test_program_operand_may_be_the_output(nk):
    M, N, K = 300, 772, 72
    A, B, C0 = synth.small_ints(902, 0, (M, K)), synth.small_ints(902, 1, (K, N)), synth.small_ints(902, 2, (M, N))
    for sched in TILES["bf16"]:
        C = dev(C0)
        nk.nk_matmul(dev(A), dev(B), C, "bf16", schedule=sched, ew=[("add", C), ("relu",)])
        nk.nk_sync_status()
        assert np.array_equal(host(C), np.maximum(A.astype(np.float64) @ B + C0, 0).astype(np.float32))


@pytest.mark.parametrize("name", ["gelu", "silu", "sigmoid"])
def test_steps_over_the_range_of_fp32(nk, name):
    x = np.concatenate([np.linspace(-30, 30, 20001), np.float64(1.37) * 2.0 ** np.arange(-140, 128),
                        -np.float64(1.37) * 2.0 ** np.arange(-140, 128),
                        [0.0, -0.0, np.inf, -np.inf, np.nan, -87.0, -89.0, 100.0]]).astype(np.float32)
    y = torch.empty(x.size, device=DEV)
    nk.nk_elementwise(dev(x), y, [(name,)])
    nk.nk_sync_status()
    got = host(y).astype(np.float64)
    v = x.astype(np.float64)
    with np.errstate(all="ignore"):   # GELU from erfc: 1 + erf cancels for negative x
        want = (np.array([0.5 * t * math.erfc(-t / math.sqrt(2.0)) for t in v]) if name == "gelu"
                else O.ew_program(v, [(name,)]))
    special = ~np.isfinite(v)
    with np.errstate(all="ignore"):
        tol = 4e-7 * np.abs(want) + 1.5e-38   # results below the normal range: absolute
    # beyond |x| = 14 the exponential's own argument rounding shows; GELU's is carried along
    near = ~special & (np.abs(v) <= 14)
    assert (np.abs(got - want)[near] <= tol[near]).all()
    far = ~special & ~near
    assert (np.abs(got - want)[far] <= (4e-6 * np.abs(want) + 1.5e-38)[far]).all()
    # x * f(x) at the infinities and NaN
    f = {"gelu": (np.inf, np.nan), "silu": (np.inf, np.nan), "sigmoid": (1.0, 0.0)}[name]
    assert got[np.isposinf(v)][0] == f[0] and np.array_equal(got[np.isneginf(v)][:1], [f[1]], equal_nan=True)
    assert np.isnan(got[np.isnan(v)]).all()
    if name != "sigmoid":
        assert np.array_equal(np.signbit(got[v == 0]), np.signbit(v[v == 0]))


@pytest.mark.parametrize("prec", ["bf16", "fp8", "bf16x3"])
@pytest.mark.parametrize("M,N,K,ldc", [(1, 1, 8, 1), (33, 31, 40, 31), (300, 770, 136, 771), (257, 515, 64, 519),
                                       (129, 36, 300, 37)])
def test_outputs_without_a_tensor_map(nk, prec, M, N, K, ldc):
    """C whose rows no TMA store can address is copied out by the warps: odd N,
    odd row strides, every tile, with a bias and a program."""
    A, B = synth.small_ints(904, 0, (M, K), -7, 7) / 2, synth.small_ints(904, 1, (K, N), -7, 7) / 2
    A[0, 0] = B[0, 0] = 3.5
    bias = synth.small_ints(904, 2, (N,))
    want = A.astype(np.float64) @ B + bias
    for sched in [None] + TILES[prec]:
        for ew in (None, [("affine", 0.5, 1.0), ("relu",)]):
            C = Canary((M, N), strides=(ldc, 1), pad=4097)
            nk.nk_matmul(dev(A), dev(B), C.t, prec, bias=dev(bias), schedule=sched, ew=ew)
            nk.nk_sync_status()
            assert np.array_equal(host(C.t), (want if ew is None else np.maximum(want * 0.5 + 1, 0)).astype(np.float32))
            C.check()


@pytest.mark.parametrize("M,N,K", [(4096, 4096, 4096), (3841, 4100, 4000), (1024, 4097, 1024)])
def test_bf16x3_wide_pairs(nk, M, N, K):
    """No schedule given: the sizes where BF16x3 takes its 256 x 256 pair tiles
    give the bits of the 128 x 128 ones (the same products in the same order)."""
    g = torch.Generator(device=DEV).manual_seed(5)
    A, B = torch.randn(M, K, generator=g, device=DEV), torch.randn(K, N, generator=g, device=DEV)
    C, R = torch.empty(M, N, device=DEV), torch.empty(M, N, device=DEV)
    nk.nk_matmul(A, B, C, "bf16x3")
    nk.nk_matmul(A, B, R, "bf16x3", schedule=(128, 128, 64, 1, 3, 1))
    nk.nk_sync_status()
    assert torch.equal(C, R)
