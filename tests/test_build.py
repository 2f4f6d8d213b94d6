"""The build refuses device code whose result the language leaves open: a
function that returns a value on some paths only."""
import shutil
import subprocess

import pytest

from paper_1802_07871_gb300 import build


@pytest.mark.parametrize("end,ok", [("", False), ("  return true;\n", True)])
def test_a_missing_return_is_an_error(tmp_path, end, ok):
    if not (shutil.which("nvcc") or shutil.which("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no nvcc")
    src = tmp_path / "f.cu"
    src.write_text("__device__ bool f(int n) {\n  for (int k = 0; k < n; ++k)\n    if (k > 7) return false;\n"
                   f"{end}}}\n__global__ void g(int n, int* o) {{ *o = f(n); }}\n")
    r = subprocess.run([build._nvcc(), *build._flags(), "-c", str(src), "-o", str(tmp_path / "f.o")],
                       capture_output=True, text=True)
    assert (r.returncode == 0) == ok, r.stdout + r.stderr
