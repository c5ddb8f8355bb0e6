"""What the bench says of the plane kernel: its shapes are those of the CUDA source, the bytes
and flops of a launch are those of the path that ran, and the memory plan sizes the ring by it.
"""
import os
import shutil
import subprocess
import types

import numpy as np
import pytest

import bench
from paper_1408_7060_gb300.inputs import icosphere, place_grid

LENGTHS = (16, 32, 64, 128, 144, 192, 256)


def test_plane_shapes_are_the_kernels(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    pairs = [(L, lz) for L in LENGTHS if L != 144 for lz in LENGTHS if lz <= L]
    rows = "".join(f'  row<{L}, {lz}, {c}>("{c}");\n' for L, lz in pairs for c in ("float2", "double2"))
    (tmp_path / "shapes.cu").write_text(f'''#include <cstdio>
#include "plane.cuh"
template <int L, int LZ, class C> void row(const char* c) {{
  constexpr PlaneOrder o = plane_order<L, LZ, C>();
  std::printf("%d %d %s %zu %d %d\\n", L, LZ, c, PlaneCfg<L, LZ, C>::smem, o.stored * o.cw, (int)plane_fits<L, LZ, C>());
}}
int main() {{
{rows}}}
''')
    exe = str(tmp_path / "shapes")
    inc = [f"-I{bench.CSRC}", f"-I{os.path.join(bench.ROOT, 'include')}"]
    # operator.h's SlabList is a parameter of a kernel in the header
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode=arch=compute_103a,code=sm_103a", *inc,
                    "-include", "aim_internal.h", "-include", "operator.h", "-o", exe, str(tmp_path / "shapes.cu"),
                    "-lcudart"], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    assert len(out) == 2 * len(pairs)
    for line in out:
        L, lz, c, smem, cols, fits = line.split()
        esz = 8 if c == "float2" else 16
        assert bench.plane_shape(int(L), int(lz), esz) == (int(smem), int(cols)), line
        assert bench.plane_fits(int(L), int(lz), esz) == bool(int(fits)), line


def test_ring_limit_is_the_librarys():
    src = open(os.path.join(bench.CSRC, "operator.cu")).read()
    assert "kPlaneRingMax = size_t(64) << 30;" in src and bench.PLANE_RING_MAX == 64 << 30


def workload(grid, z=1.0):
    V, F = icosphere(4, 1.0)
    V = V * np.array([1.0, 1.0, z])
    h, origin = place_grid(V, grid)
    return types.SimpleNamespace(mesh=(V, F), grid_n=grid, h=h, origin=origin)


def test_memory_plan_holds_z_spectra_on_the_plane_kernel():
    w = workload(96)
    assert bench.box_depth(w)[1] == 192
    ring = 7 * 4 * 192 ** 3 * 8
    step = bench.context_bytes(w, 7, 0, 5) - bench.context_bytes(w, 7, 0, 4)
    assert ring < step < 1.25 * ring                         # no padded slab beside it
    # past 64 GiB the library runs the separate passes: slabs of the box planes, and the padded slab
    b = (64 << 30) // ring
    nz = bench.box_depth(w)[0]
    assert bench.context_bytes(w, 7, 0, b + 1) < bench.context_bytes(w, 7, 0, b)
    step = bench.context_bytes(w, 7, 0, b + 2) - bench.context_bytes(w, 7, 0, b + 1)
    slab = 4 * nz * 192 ** 2 * 8
    assert 8 * slab < step < 10 * slab


def test_chunk_fits():
    for w in (workload(64), workload(96), workload(128, 0.4)):
        for total in (20e9, 150e9, 284e9):
            nb = bench.chunk_size(w, 7, 4, total)
            assert nb == 1 or bench.context_bytes(w, 7, 4, nb) + 6e9 <= total
            assert bench.context_bytes(w, 7, 4, nb + 1) + 6e9 > total


def test_bytes_and_flops_follow_the_path():
    args = dict(N=64, ns=7680, nnz=200000, ng=7, nb=4, box=(62, 62, 62), lz=128, n_active=100000)
    A, slab, spec = 4 * 62 * 64 * 128 * 8 * 4, 4 * 62 * 128 ** 2 * 8 * 4, 4 * 128 ** 3 * 8 * 4
    plane = {k: bench.kernel_bytes(k, plane=True, **args) for k in ("zconv", "zrhs", "zfwd", "yfft_fwd", "yfft_inv")}
    assert plane["yfft_fwd"] is None and plane["yfft_inv"] is None
    assert 2 * A < plane["zconv"] < 2 * slab and plane["zfwd"] == A + spec
    assert 9 * spec + A < plane["zrhs"] < 9 * spec + A + 7 * 2 * 65 * 128 * 128 * 8
    assert bench.kernel_bytes("zconv", **args) == 2 * slab + 2 * 65 ** 2 * 65 * 8
    flops = lambda kind, **kw: bench.kernel_flops(kind, 64, 4, 7, 128, **kw)
    rows = 4 * 4 * 128 * 62 * 5 * 128 * 7
    assert flops("zconv", plane=True, bz=62) == flops("zconv") + 2 * rows
    assert flops("zrhs") == 4 * 4 * 128 ** 2 * (5 * 128 * 7 + 8 * 7 * 128)       # spectra: one inverse
    assert bench.kernel_flops("zrhs", 96, 1, 7, 192) > 7 * 4 * 192 ** 2 * 5 * 192 * 7
    assert bench.alu_kernels(144, False) == ("zconv", "zrhs") and bench.alu_kernels(192, True) == ("zconv",)
