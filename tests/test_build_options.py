"""The path kernels' sources compile for sm_103a with each of their build
options, and with the debug and counter builds'."""
import subprocess

import pytest

from paper_2503_12174_gb300 import build as b

SRC = """
#include "tile.cuh"
namespace dpcs {
__global__ void lanes(const RenderArgs a, const Ray r, Hit *h) {
    Cnt cnt;
    traverse(a.nodes, a.tris, a.root, a.T, r, 1.0f, false, *h, a.status, cnt);
}
__global__ void tiles(const RenderArgs a, const Ray r, float *o) {
    Cnt cnt;
    int pos = -1;
    float t = 1.0f, u, v;
    tree_walk<true>(a, r, false, a.root, pos, t, u, v, cnt);
    o[threadIdx.x] = pos + t + u + v;
}
}
"""


@pytest.mark.parametrize("option", ["", "DPCS_SLAB_FMA=0", "DPCS_WATERTIGHT=0", "DPCS_WATERTIGHT=2",
                                    "DPCS_SLAB_MINMAX3=0", "DPCS_MT_DETCHECK=1", "DPCS_FUSION_BY_COMPILER",
                                    "DPCS_CHECK", "DPCS_COUNTERS"])
def test_option_compiles(tmp_path, option):
    try:
        nvcc = b.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src = tmp_path / "option.cu"
    src.write_text(SRC)
    p = subprocess.run([nvcc, "-c", str(src), "-o", str(tmp_path / "option.o"), "-std=c++17", "-Xptxas", "-O0", *b.ARCH,
                        "-I", b.INCLUDE, "-I", b.CSRC, "--expt-relaxed-constexpr", *([f"-D{option}"] if option else [])],
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
