"""Training on a cluster of 8 CTAs (csrc/sp_model.cu, for devices that take no
cluster of 16): the cost model built with 8 as the largest size, against the
FP64 oracle at the sizes of test_gpu_train.py (shares and slices differ from
those of 16)."""
import ctypes
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")

import test_gpu_train as full  # noqa: E402
from paper_1011_4046_gb300 import build, sp  # noqa: E402

pytestmark = pytest.mark.gpu

MODEL = ("create", "destroy", "get_params", "set_params", "predict", "grad", "adam_step", "train", "save", "load")


@pytest.fixture(scope="module")
def lib8(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    out = str(tmp_path_factory.mktemp("eight") / "libsp_model8.so")
    subprocess.run([build.nvcc(), *build._flags(["-DSP_TRAIN_CTAS=8"]), "-shared", "-cudart", "static",
                    os.path.join(build.CSRC, "sp_model.cu"), "-o", out], check=True)
    lib, ref = ctypes.CDLL(out), sp.load()
    for name in MODEL:
        getattr(lib, "sp_model_" + name).argtypes = getattr(ref, "sp_model_" + name).argtypes
    lib.sp_strerror = ref.sp_strerror
    return lib


@pytest.mark.parametrize("n, batch", [(7, 3), (40, 16), (515, 256), (530, 257), (1400, 700), (4100, 4096)])
def test_training_steps_match_oracle_on_eight_ctas(lib8, monkeypatch, n, batch):
    monkeypatch.setattr(sp, "_lib", lib8)
    full.test_training_steps_match_oracle(n, batch)
