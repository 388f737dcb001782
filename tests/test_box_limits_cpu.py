"""Which kernels the adjoint takes (box_limits.h), compiled for the host: the whole-face
kernel forms its offsets in 32 bits, so boxes above 1290^3 keep the quadrant kernels."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2311_01492_gb300", "csrc")


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("box_limits")
    src, lib = str(d / "s.cpp"), str(d / "s.so")
    with open(src, "w") as f:
        # a catalogue of half-widths 40, 20 and 10, a third each
        f.write('#include "%s/box_limits.h"\n'
                'extern "C" int max_box() { return asora::kMaxBox32; }\n'
                'extern "C" void plan(int ns, int nmax, int faces, int exit, int* out) {\n'
                '  auto ff = [&](int h) { return h >= 40 ? 0 : h >= 20 ? ns / 3 : h >= 10 ? '
                '2 * ns / 3 : ns; };\n'
                '  auto p = asora::adjoint_plan(ns, nmax, faces, exit, 40, 16, 27, ff);\n'
                '  out[0] = p.face_begin; out[1] = p.quads; out[2] = p.split; out[3] = p.leftover;\n'
                '}\n' % CSRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", src, "-o",
                    lib], check=True)
    so = C.CDLL(lib)

    def call(ns, nmax, faces, exit):
        out = (C.c_int * 4)()
        so.plan(ns, nmax, faces, exit, out)
        return tuple(out)
    call.max_box = so.max_box()
    return call


def test_the_largest_box_is_the_last_cube_of_31_bits(plan):
    n = plan.max_box
    assert n ** 3 <= 2 ** 31 - 1 < (n + 1) ** 3


@pytest.mark.parametrize("nmax", [2, 250, 1290, 1291, 1300, 4096])
@pytest.mark.parametrize("exit", [0, 1])
@pytest.mark.parametrize("faces", [0, 1])
def test_the_adjoint_takes_whole_faces_only_where_32_bits_hold_an_offset(plan, nmax, exit, faces):
    ns = 900
    face_begin, quads, split, leftover = plan(ns, nmax, faces, exit)
    if not faces or nmax > 1290:
        assert (face_begin, quads, split, leftover) == (ns, ns, 300, 0)
    elif exit:  # all by faces, what is too wide may come back
        assert (face_begin, quads, split, leftover) == (0, ns, 300, 1)
    else:       # half-widths up to 16 by faces
        assert (face_begin, quads, split, leftover) == (600, 600, 300, 0)
