"""The library's host-side services (device memory pool, transfers, result buffers, mailboxes) under several threads and
without host memory, and the layout of small scoring batches and their answers, on the CPU: host_services_check.cpp defines
the CUDA runtime calls they make."""
import subprocess
from pathlib import Path

import pytest

from paper_2004_13940_b200 import build as B


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = tmp_path_factory.mktemp("host_services") / "check"
    cuda = Path(B._nvcc()).resolve().parent.parent / "include"
    subprocess.run(["g++", "-O1", "-std=c++17", "-pthread", "-I", str(cuda), "-I", str(B.CSRC), "-o", str(exe),
                    str(Path(__file__).with_name("host_services_check.cpp"))], check=True)
    return lambda what: subprocess.run([str(exe), what], capture_output=True, text=True, timeout=120)


@pytest.mark.parametrize("what", ["transfers-in", "transfers-out", "threads", "no-host-memory", "requests", "scores"])
def test_host_services(check, what):
    r = check(what)
    assert r.returncode == 0, r.stdout + r.stderr
