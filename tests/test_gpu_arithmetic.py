"""Arithmetic of the GEMMs against 64 bits: the sigmoids of their epilogues over every float, and the
FP32 product from three bf16 slices per operand, on rows of like and of unlike magnitudes."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    """tests/arith_shim.cu as a library, linked against the repository's own."""
    from paper_2502_06073_gb300 import _build
    _build.build()
    so = str(tmp_path_factory.mktemp("shim") / "libshim.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-I", _build.CSRC,
                    os.path.join(HERE, "arith_shim.cu"), _build.LIB, "-o", so,
                    "-Xlinker", "-rpath=" + os.path.dirname(_build.LIB)], check=True)
    assert torch.cuda.is_available()
    return ctypes.CDLL(so)


@pytest.mark.parametrize("which", ["sigm_fast", "sigm_ftz", "sigm_nr"])
def test_sigmoid_of_every_float_within_its_bound(shim, which):
    """The bounds are those stated at the functions, from the documented errors of the hardware
    exponential, power, reciprocal and division and of expf, one rounding per operation."""
    worst = torch.zeros(2, dtype=torch.int32, device="cuda")
    k = ["sigm_fast", "sigm_ftz", "sigm_nr"].index(which)
    assert shim.shim_check_sigmoid(k, ctypes.c_void_p(worst.data_ptr())) == 0
    ratio, bad = worst.cpu().numpy()[:1].view(np.float32)[0], int(worst[1])
    print(f"{which}: largest error {ratio:.3f} of the bound")
    assert bad == 0 and ratio <= 1.0


def _chunk_max(x, K1):
    """|x| with every element replaced by the largest of its row's 32-element chunk (the second
    part of a concatenated K starts a chunk of its own)."""
    x = x.abs()
    out = torch.empty_like(x)
    for a, b in ((0, K1), (K1, x.shape[1])):
        for k in range(a, b, 32):
            e = min(k + 32, b)
            out[:, k:e] = x[:, k:e].amax(1, keepdim=True)
    return out


def _operands(M, N, K, span, seed):
    """Normal rows; with a span, A's columns scaled by powers of two over 2^span inside every
    chunk and B's rows by their inverses, so that every term of the products counts alike."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    A = torch.randn(M, K, generator=g, device="cuda")
    Bt = torch.randn(N, K, generator=g, device="cuda")
    if span:
        s = torch.exp2(torch.randint(0, span + 1, (K,), generator=g, device="cuda") - span / 2.0)
        A, Bt = A * s, Bt / s
    return A, Bt


@pytest.mark.parametrize("span", [0, 10])
@pytest.mark.parametrize("M,N,K1,K2", [(1, 16, 16, 0), (129, 144, 48, 0), (300, 256, 352, 0),
                                       (257, 272, 80, 112), (5000, 256, 256, 96)])
def test_fp32_gemm_error_within_its_bound(shim, M, N, K1, K2, span):
    """|error| <= (2^-23 + (K / 16 + 3) 2^-22) sum_k amax_k bmax_k, amax and bmax the largest
    magnitudes of an element's chunk.  The first term: the dropped products a2 b3 and a3 b2 and the
    rounding of a3 and b3, 2^-25 of the units' product each.  The second: an accumulation that
    truncates, at most 2^-23 of the running sum of each accumulator per 16 elements, the last sum,
    and FP32's own rounding of the result.  Rows of like magnitude must also be no further off
    than a plain FP32 product (2-norm over the whole output, a quarter for the spread of samples)."""
    A, Bt = _operands(M, N, K1 + K2, span, 1000 + K1)
    A1, A2 = A[:, :K1].contiguous(), A[:, K1:].contiguous()
    W1, W2 = Bt[:, :K1].contiguous(), Bt[:, K1:].contiguous()
    ld = shim.shim_split_ld(K1, K2)
    slices = torch.empty(3 * N * ld, dtype=torch.bfloat16, device="cuda")
    out = torch.empty(M, N, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    p = lambda t: ctypes.c_void_p(t.data_ptr() if t.numel() else 0)  # noqa: E731
    assert shim.shim_gemm_f32(p(A1), p(A2), p(W1), p(W2), M, N, K1, K2, p(slices), p(out),
                              p(err)) == 0 and int(err[0]) == 0
    exact = A.double() @ Bt.double().T
    e = (out.double() - exact).abs()
    scale = _chunk_max(A, K1).double() @ _chunk_max(Bt, K1).double().T
    c = 2.0 ** -23 + ((K1 + K2) / 16 + 3) * 2.0 ** -22
    fma = torch.zeros(M, N, device="cuda")
    for k in range(K1 + K2):     # a chain of FP32 products and sums
        fma = torch.addcmul(fma, A[:, k:k + 1], Bt[None, :, k])
    rel = lambda x: float((x.double() - exact).norm() / exact.norm())  # noqa: E731
    print(f"M {M} N {N} K {K1}+{K2} span 2^{span}: {float((e / (c * scale)).max()):.3f} of the "
          f"bound; 2-norm error {rel(out):.2e}, FP32 chain {rel(fma):.2e}")
    assert bool((e <= c * scale).all())
    if span == 0 and M > 1:
        assert rel(out) <= 1.25 * rel(fma)
