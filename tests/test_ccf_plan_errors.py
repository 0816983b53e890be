"""A device allocation that fails while the FP64 CCF is planned ends the call with its status; it is not
taken for a mask that the form does not apply to.  Without a GPU every allocation fails."""
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parents[1]


def test_failed_allocation_is_returned(tmp_path):
    torch = pytest.importorskip("torch")
    if torch.cuda.is_available():
        pytest.skip("allocations succeed")
    from paper_2301_04259_gb300 import _build
    lib = _build.build()
    exe = tmp_path / "plan"
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, str(ROOT / "tests/native/ccf_ramp_plan.cu"), "-o",
                    str(exe), str(lib), "-Xlinker", f"-rpath={lib.parent}"], check=True, capture_output=True)
    status, lines, text = subprocess.run([str(exe)], check=True, capture_output=True,
                                         text=True).stdout.split(maxsplit=2)
    assert int(status) != 0 and int(lines) == 0 and "cudaMalloc" in text
