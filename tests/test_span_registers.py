"""Register use of the general-layout bodies with run-time extents (every shape that has no
instantiation of its own): the compiler must not spill their fibers to local memory."""
import re
import subprocess

from paper_1304_7054_gb300 import build as libbuild


def test_runtime_extent_bodies_do_not_spill(tmp_path):
    cmd = [libbuild.nvcc(), *libbuild.NVCC_FLAGS, "-Xptxas", "-v", "-cubin", "-o", str(tmp_path / "s.cubin"),
           libbuild.CSRC + "/kron_span_f32_d2.cu"]
    log = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True, check=True).stdout
    spills = re.findall(r"entry function '\S*span_kernelIfLi(\d+)ELi0E\S*'.*?(\d+) bytes spill stores", log, re.S)
    assert sorted(int(ni) for ni, _ in spills) == [4, 8, 12, 16]
    assert all(int(n) == 0 for _, n in spills), spills
