"""The dispatch of complex64 products (host logic, no GPU): every size has a kernel that is instantiated,
and the line between the packed 64 x 64 tiles and smaller ones is one."""
import ctypes

import pytest

SMALL_K, DOT, PACKED, SKINNY, TILE = range(5)


def gemm_route(mb, nb, kb, n_items, sms=152):
    """(kind, row edge, column edge) of the kernel a 2^mb x 2^kb x 2^nb product over n_items items takes."""
    from paper_2110_09894_gb300 import qx
    f = qx.load().qx_internal_gemm_route
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_int] * 3 + [ctypes.c_int64, ctypes.c_int]
    r = f(mb, nb, kb, n_items, sms)
    return r // 100, r // 10 % 10, r % 10


@pytest.mark.parametrize("sms", [1, 76, 152, 600])
def test_every_product_has_a_kernel(sms):
    for mb in range(0, 13):
        for nb in range(0, 13):
            for kb in range(0, 14):
                for items in (1, 2, 17, 151, 152, 153, 512, 4097, 65535):
                    kind, bm, bn = gemm_route(mb, nb, kb, items, sms)
                    if kind == SMALL_K:
                        assert kb <= 2 and nb >= 5
                    elif kind == DOT:
                        assert mb + nb <= 4 and kb >= 8
                    elif kind == PACKED:  # whole tiles, whole stages of 8 k
                        assert (bm, bn) in ((6, 6), (6, 5), (5, 6), (5, 5)) and mb >= bm and nb >= bn and kb >= 3
                    elif kind == SKINNY:
                        assert min(mb, nb) <= 4 and kb >= 3
                    else:
                        assert kind == TILE and 4 <= bm <= 6 and 4 <= bn <= 6 and (bm, bn) != (6, 6)


def test_the_lines_between_the_tiles():
    assert gemm_route(6, 6, 6, 152) == (PACKED, 6, 6) and gemm_route(6, 6, 6, 151)[0] == TILE
    assert gemm_route(8, 7, 3, 19) == (PACKED, 6, 6) and gemm_route(8, 7, 3, 18)[0] == TILE
    assert gemm_route(5, 5, 7, 512) == (PACKED, 5, 5) and gemm_route(5, 5, 7, 511)[0] == TILE
    assert gemm_route(7, 5, 4, 256) == (PACKED, 6, 5) and gemm_route(7, 5, 4, 255)[0] == TILE
    assert gemm_route(5, 9, 9, 64) == (PACKED, 5, 6) and gemm_route(5, 9, 9, 63)[0] == TILE
