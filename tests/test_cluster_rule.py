"""Which items a batch gives to thread-block clusters: only where the device takes the cluster."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROBE = r"""
#include <cstdio>
#include "rdm_internal.h"
int main() {
  for (int c_log = 0; c_log <= 5; ++c_log) {
    rdm::Layout L{};
    L.n_bits = rdm::kTileBits + c_log;
    L.D = int64_t(1) << L.n_bits;
    L.DS = 2;
    L.precision = RDM_FP32;
    L.elem = 4;
    L.VW = 4;
    L.B = L.Bs = 8;
    L.n_slices = 1;
    L.TPR = 2;
    rdm::TiledTerms t{};
    t.ready = 1;
    t.dg.n_entries = 8;
    std::printf("%d", rdm::pass1_cluster_fits(L, t) ? 1 : 0);
  }
}
"""


def test_clusters_only_where_the_device_takes_them(tmp_path):
    """Without a device (as on one that cannot hold the cluster) no item takes the cluster
    launch, so a batch runs the packed units instead of failing; with a whole GPU the sizes
    2^10 .. 2^14 take it and 2^15 does not."""
    import torch

    from paper_2204_08147_gb300 import build
    if not os.path.exists(build.LIB):
        build.build_library()
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    inc = [os.path.join(ROOT, "include"), build.CSRC, os.path.join(build._cuda_home(build._nvcc()), "include")]
    subprocess.run([cxx, "-std=c++17", str(src), "-o", str(exe), *[f"-I{d}" for d in inc], build.LIB,
                    f"-Wl,-rpath,{build.PKG}"], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    assert out == ("111110" if torch.cuda.is_available() else "000000")
