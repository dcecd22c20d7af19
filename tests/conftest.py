import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA GPU (GB300, sm_103a) and the built library")
    config.addinivalue_line("markers", "slow: oracle checks that take more than a few seconds on the CPU")


@pytest.fixture(scope="session")
def cuda_program(tmp_path_factory):
    """Compile a CUDA program against the built library's own headers and symbols: for what no public call reaches
    by itself.  Returns a function from the program's text to its executable."""
    from paper_1111_6288_gb300 import build

    def compile_program(text):
        where = tmp_path_factory.mktemp("program")
        src, exe = where / "program.cu", where / "program"
        src.write_text(text)
        subprocess.run([build.nvcc(), build.ARCH, "-std=c++17", "-I", build.CSRC, "-I",
                        os.path.join(build.ROOT, "include"), str(src), build.LIB, "-Xlinker",
                        "-rpath=" + os.path.dirname(build.LIB), "-o", str(exe)], check=True)
        return exe

    return compile_program
