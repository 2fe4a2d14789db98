"""Tile widths of the matrix products (csrc/gemm_tiles.h), against the widths that were measured on both sides of every line."""
import ctypes as C
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2512_04939_b200", "csrc")


@pytest.fixture(scope="module")
def columns(tmp_path_factory):
    d = tmp_path_factory.mktemp("tiles")
    (d / "tiles.cpp").write_text('#include "gemm_tiles.h"\nextern "C" int columns(long long m, long long n, long long k, int heads) {'
                                 " return lv::gemm_tile_columns(m, n, k, heads != 0, 148); }\n")
    so = str(d / "tiles.so")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "tiles.cpp"), "-o", so], check=True)
    fn = C.CDLL(so).columns
    return lambda m, n, k, heads=False: fn(C.c_longlong(m), C.c_longlong(n), C.c_longlong(k), int(heads))


@pytest.mark.parametrize("m,n,k", [(5601, 2048, 512), (12545, 1536, 512), (3553, 1536, 512),  # short k
                                   (17153, 3072, 768), (17153, 3072, 1024), (34561, 1536, 1024), (17153, 3072, 1536)])  # thirteen waves
def test_no_half_chunks_where_they_were_slower(columns, m, n, k):
    assert columns(m, n, k) % 64 == 0


@pytest.mark.parametrize("m,n,k,want", [(3360, 1024, 4096, 224), (2305, 1024, 4096, 160), (14209, 1024, 4096, 224), (34561, 1536, 4096, 224),
                                        (1777, 4096, 1024, 224), (4737, 4096, 1024, 224), (2305, 1024, 1024, 160), (7409, 1024, 1024, 224)])
def test_half_chunks_where_they_were_faster(columns, m, n, k, want):
    assert columns(m, n, k) == want


def test_tiles_of_whole_heads_have_multiples_of_64_columns(columns):
    widths = {columns(m, 3072, 1024, heads=True) for m in range(1, 40000, 61)}
    assert widths <= {0, 64, 128, 192, 256} and len(widths) > 2
