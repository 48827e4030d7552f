"""Elementary arithmetic of the GEMMs against 64 bits: the sigmoids of their epilogues, every float."""
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
