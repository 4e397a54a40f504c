"""The branch-free reciprocal of the multi-step kernel and of the backward step
(rcp_rn, rcp_neg) is the correctly rounded one for every FP32 mantissa, the
all-ones one included, which the theorem behind it leaves open: multi-step and
single steps, which use the library's reciprocal, give the same bits only then."""
import os
import subprocess

import pytest

from paper_2210_10377_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_every_mantissa_at_a_range_of_exponents(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    exe = str(tmp_path / "reciprocal")
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "reciprocal_harness.cu"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout.split()
    assert int(out[0]) >= 20 << 23 and int(out[1]) == 0
