"""Which pipelined step-kernel shapes exist for which populations: the library's own block-layout rule
(pipe_layout), compiled for the host, at the shared memory of an sm_103a SM.  No GPU needed."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1301_3423_gb300 import builder

SMEM_PER_SM, SMEM_PER_BLOCK = 228 * 1024, 227 * 1024
Q = {3: 128, 2: 66}
ELEM = {"f64": 8, "f32": 4, "f16dev": 2}
# (order, storage): the variants whose stages fit; narrower rows for double, whose stages are twice as large
SHAPES = {
    (3, "f64"): {7, 11},
    (3, "f32"): {4, 5, 6, 7, 8, 9, 12, 13, 15, 16, 17, 18, 19, 21, 22},
    (3, "f16dev"): set(range(4, 20)) | {21, 22, 23},
    (2, "f64"): set(range(4, 20)),
    (2, "f32"): {4, 5, 6, 7, 8, 9, 12, 13, 15, 16, 17, 18, 19, 21, 22, 23},
    (2, "f16dev"): set(range(4, 20)) | {21, 22, 23},
}


@pytest.fixture(scope="module")
def layout(tmp_path_factory):
    d = tmp_path_factory.mktemp("layout")
    src = d / "layout.cpp"
    src.write_text('#include "rlb_launch.h"\n'
                   'extern "C" int layout(int v, int q, int elem, int* out) {\n'
                   "  rlb::PipeLayout l{};\n"
                   "  if (!rlb::pipe_layout(v, q, elem, %d, %d, &l)) return 0;\n"
                   "  const int r[] = {l.tx, l.rows, l.nstage, l.groups, l.producers, l.threads, l.smem, l.split};\n"
                   "  for (int k = 0; k < 8; ++k) out[k] = r[k];\n"
                   "  return 1;\n}\n"
                   'extern "C" int max_warps(int elem, int split) { return rlb::pipe_max_warps(elem, split); }\n'
                   % (SMEM_PER_SM, SMEM_PER_BLOCK))
    cuda = os.path.dirname(os.path.dirname(builder._nvcc()))
    subprocess.check_call([shutil.which("g++") or "g++", "-std=c++17", "-shared", "-fPIC", "-I", builder.CSRC, "-I",
                           os.path.join(cuda, "include"), "-o", str(d / "layout.so"), str(src)])
    lib = ctypes.CDLL(str(d / "layout.so"))

    def ask(v, order, storage):
        out = (ctypes.c_int * 8)()
        if not lib.layout(v, Q[order], ELEM[storage], out):
            return None
        return dict(zip(("tx", "rows", "nstage", "groups", "producers", "threads", "smem", "split"), out))
    ask.max_warps = lambda storage, lay: lib.max_warps(ELEM[storage], lay["split"])
    return ask


@pytest.mark.parametrize("order,storage", sorted(SHAPES))
def test_shapes_exist(layout, order, storage):
    got = {}
    for v in range(24):
        lay = layout(v, order, storage)
        if lay:
            got[v] = lay
    assert set(got) == SHAPES[order, storage]
    for lay in got.values():
        assert lay["threads"] <= 32 * layout.max_warps(storage, lay)
        assert lay["nstage"] >= 2 and lay["nstage"] % lay["groups"] == 0 and lay["smem"] <= SMEM_PER_BLOCK
        assert 1 <= lay["producers"] <= lay["threads"] // 32 - 1


@pytest.mark.parametrize("order,storage", sorted(SHAPES))
def test_units_built_are_the_ones_a_shape_needs(layout, order, storage):
    needed = {(lay["tx"], lay["rows"]) for lay in (layout(v, order, storage) for v in range(24)) if lay}
    s = list(ELEM).index(storage)
    assert sorted(needed) == sorted((tx, rows) for o, t, tx, rows in builder.PIPE_UNITS if (o, t) == (order, s))


def test_built_tree_is_small():
    """The library's folder travels with the tree: no objects are left in it, and it stays far below the
    few hundred megabytes that a copy of the tree may have."""
    builder.build()
    files = [os.path.join(d, f) for d, _, fs in os.walk(builder.BUILD) for f in fs]
    assert not [f for f in files if f.endswith(".o")]
    assert sum(os.path.getsize(f) for f in files) < 100e6
