"""The host rules that shape the launches (CPU: the library's functions, no device): z planes per thread of the shell
kernels, planes per batch of loads of the one-cell ones, planes per thread of the design-E kernels.  Sizes lie on
either side of each line."""
import ctypes as C

import pytest

from paper_2305_00234_gb300 import _native, build


@pytest.fixture(scope="module", autouse=True)
def built():
    build.build()


class ShellBoxes(C.Structure):
    _fields_ = [("n", C.c_int), ("b", C.c_int * 6 * 6), ("first", C.c_uint * 7), ("kz", C.c_int), ("pz", C.c_int), ("pair", C.c_int)]


def shape(boxes, pair, type_bytes=4, cells=0, beside=False):
    s = ShellBoxes(n=len(boxes), pair=int(pair))
    for q, b in enumerate(boxes):
        s.b[q][:] = b
    f = _native.load_library()._ZN4fdtd11shell_shapeERNS_10ShellBoxesEimb
    f.argtypes, f.restype = [C.POINTER(ShellBoxes), C.c_int, C.c_size_t, C.c_bool], None
    f(C.byref(s), type_bytes, cells, beside)
    blocks = [-(-((b[1] - b[0]) // (2 if pair else 1) * (b[3] - b[2])) // 128) * -(-(b[5] - b[4]) // s.kz) for b in boxes]
    assert list(s.first[:len(boxes) + 1]) == [sum(blocks[:q]) for q in range(len(boxes) + 1)]
    return s.kz, s.pz


def around(n, ib):
    """The boxes around an interior box, as the library splits the grid."""
    return [(0, n[0], 0, n[1], 0, ib[4]), (0, n[0], 0, n[1], ib[5], n[2]), (0, n[0], 0, ib[2], ib[4], ib[5]),
            (0, n[0], ib[3], n[1], ib[4], ib[5]), (0, ib[0], ib[2], ib[3], ib[4], ib[5]), (ib[1], n[0], ib[2], ib[3], ib[4], ib[5])]


# beside an interior kernel: columns shorter than 8 planes only in one round, or where 8 would make 1.2 to 1.6 rounds of blocks
@pytest.mark.parametrize("n,ib,kz", [((328, 376, 306), (8, 324, 5, 372, 5, 302), 8), ((260, 252, 240), (16, 240, 11, 235, 11, 230), 8),
                                     ((280, 280, 280), (8, 264, 5, 276, 5, 276), 6), ((244, 247, 247), (8, 232, 5, 243, 5, 243), 8),
                                     ((244, 244, 244), (8, 232, 5, 229, 5, 240), 5), ((228, 204, 224), (16, 208, 9, 185, 9, 216), 4),
                                     ((128, 128, 128), (32, 120, 9, 120, 9, 120), 4),
                                     ((220, 260, 240), (8, 200, 3, 258, 3, 238), 8), ((296, 296, 296), (16, 272, 9, 281, 9, 288), 9)])
def test_columns_beside_an_interior_kernel(n, ib, kz):
    assert shape(around(n, ib), True, 4, n[0] * n[1] * n[2], True)[0] == kz


def test_whole_grid_columns():
    assert shape([(0, 48, 0, 48, 0, 48)], True)[0] == 1
    assert shape([(0, 96, 0, 170, 0, 170)], True)[0] == 9                    # one full round of blocks
    assert shape([(0, 600, 0, 600, 0, 600)], True)[0] <= 8


@pytest.mark.parametrize("type_bytes,cells,planes", [(4, 2499999, 1), (4, 2500000, 2), (8, 1000, 2), (8, 10 ** 8, 2)])
def test_planes_per_batch(type_bytes, cells, planes):
    assert shape([(0, 101, 0, 99, 0, 50)], False, type_bytes, cells)[1] == planes


@pytest.mark.parametrize("columns,nz,f64,other,planes", [(12 * 24, 24, False, 0, 1), (16 * 32, 31, False, 1024, 2), (32 * 64, 72, False, 0, 2),
                                                         (64 * 128, 128, False, 0, 3), (128 * 256, 192, False, 0, 5),
                                                         (64, 21845, False, 0, 5), (256, 24, True, 0, 1), (64 * 256, 192, True, 0, 8)])
def test_design_columns(columns, nz, f64, other, planes):
    f = _native.load_library()._ZN4fdtd13design_planesEiibj
    f.argtypes, f.restype = [C.c_int, C.c_int, C.c_bool, C.c_uint], C.c_int
    assert f(columns, nz, f64, other) == planes
