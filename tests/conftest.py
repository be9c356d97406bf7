import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def pytest_configure(config):
    config.addinivalue_line("markers", "gpu: needs a CUDA device (B200); run with -m gpu")


def pytest_collection_modifyitems(config, items):
    import torch
    if torch.cuda.is_available():
        return
    skip = pytest.mark.skip(reason="no CUDA device")
    for item in items:
        if "gpu" in item.keywords:
            item.add_marker(skip)


@pytest.fixture
def tuning():
    """Apply overrides of the library's launch planner for one test: tuning(splits=3, kernel=2). Reset afterwards."""
    from paper_2508_02558_b200 import binding as B
    B.tuning_reset()

    def apply(**kw):
        for name, value in kw.items():
            B.tuning_set(name, value)
    yield apply
    B.tuning_reset()


@pytest.fixture
def host_program(tmp_path):
    """Compile a program of tests/native/ against the library's headers and libsdllm.so (host code only); returns its path."""
    def compile_program(source: str) -> str:
        import subprocess
        from paper_2508_02558_b200 import build as libbuild
        lib = libbuild.build()
        include = [os.path.join(ROOT, "include"), libbuild.CSRC, os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")]
        exe = str(tmp_path / source.split(".")[0])
        subprocess.run([os.environ.get("CXX", "g++"), "-O1", "-std=c++17", *(f"-I{d}" for d in include), "-o", exe,
                        os.path.join(ROOT, "tests", "native", source), lib, f"-Wl,-rpath,{os.path.dirname(lib)}"], check=True)
        return exe
    return compile_program
