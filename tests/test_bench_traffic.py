"""The DRAM traffic the benchmark reports belongs to the kernel's whole source: a
header that it includes, directly or through another, counts as the kernel."""
import hashlib
import os

import pytest

import bench

FILES = {"cd_flow.cu": b'#include "cd_core.cuh"\n#include <cuda_runtime.h>\nflow\n',
         "cd_sweep.cu": b'  # include "cd_inner.cuh"\nsweep\n',
         "cd_core.cuh": b'#include "cd_inner.cuh"\n#include "cd_api.h"\ncore\n',
         "cd_inner.cuh": b"inner\n", "cd_other.cuh": b"other\n"}


def tree(root, shas, changed=None):
    csrc = os.path.join(root, "paper_1104_3516_gb300", "csrc")
    os.makedirs(csrc)
    os.makedirs(os.path.join(root, "profiles"))
    for name, src in FILES.items():
        with open(os.path.join(csrc, name), "wb") as f:
            f.write(src + (b"// changed\n" if name == changed else b""))
    with open(os.path.join(root, "profiles", "k_sweep_traffic.txt"), "w") as f:
        for (kernel, sha), traffic in zip(shas.items(), (11, 22)):
            f.write(f"kernel={kernel} n=5 precision=f64 traffic_bytes_per_launch={traffic} src_sha256={sha}\n")


@pytest.mark.parametrize("changed, flow, sweep", [
    (None, 11.0, 22.0), ("cd_other.cuh", 11.0, 22.0), ("cd_core.cuh", None, 22.0), ("cd_inner.cuh", None, None),
    ("cd_flow.cu", None, 22.0), ("cd_sweep.cu", 11.0, None)])
def test_a_changed_header_invalidates_the_figure(tmp_path, monkeypatch, changed, flow, sweep):
    sha = lambda *names: hashlib.sha256(b"".join(FILES[n] for n in names)).hexdigest()[:16]  # noqa: E731
    tree(str(tmp_path), {"k_flow<2,double>": sha("cd_flow.cu", "cd_core.cuh", "cd_inner.cuh"),
                         "k_sweep<2,double>": sha("cd_sweep.cu", "cd_inner.cuh")}, changed)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench.profiled_traffic("k_flow<2,double>", "f64", 5) == flow
    assert bench.profiled_traffic("k_sweep<2,double>", "f64", 5) == sweep


def test_the_sources_of_the_solve_kernels():
    for kernel, own in (("k_flow<2,double>", b"k_flow("), ("k_sweep<2,double>", b"k_sweep(")):
        src = bench.kernel_source(kernel)
        assert own in src and b"__device__ __forceinline__ double abs_of_pair" in src and b"struct CdCtrl {" in src
