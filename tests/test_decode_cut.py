"""The cut of the decode scan's work, walked on the host for every block of the grid: each page is scanned once, each row is
stored or merged once, and a merge waits for the blocks that arrive and reads the partials that they stored."""
import ctypes as C
import os
import random
import subprocess

import pytest

from conftest import ROOT

SMS = 148
# launch shapes of the kernels: warps, blocks per SM, long pages, several layers end to end, tensor-memory kernel
SHAPES = {"d256": (8, 1, 0, 0, 0), "d256_two": (4, 2, 0, 0, 0), "d128_one": (16, 1, 0, 0, 0), "d128": (8, 2, 0, 0, 0),
          "long_d128": (12, 1, 1, 0, 0), "long_d256": (8, 1, 1, 0, 0), "tensor_memory": (16, 1, 0, 0, 1),
          "flat_d256": (8, 1, 0, 1, 0), "flat_d256_two": (4, 2, 0, 1, 0), "flat_d128": (8, 2, 0, 1, 0), "flat_d128_one": (16, 1, 0, 1, 0),
          "flat_long_d128": (12, 1, 1, 1, 0), "flat_long_d256": (8, 1, 1, 1, 0)}


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("cut") / "cut_walk.so")
    subprocess.run([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(ROOT, "paper_2608_23834_b200", "csrc"),
                    "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "cut_walk.cu"), "-o", so], check=True)
    return C.CDLL(so)


@pytest.fixture(scope="module")
def walk(lib):
    def run(shape, lens, hkv, n_layers=1):
        warps, per_sm, long_pages, flat, tensor_memory = SHAPES[shape]
        out = [C.c_int() for _ in range(3)]
        why = C.create_string_buffer(200)
        rc = lib.cut_walk((C.c_int * len(lens))(*lens), len(lens), hkv, SMS * per_sm, n_layers, flat, warps, per_sm, long_pages,
                          tensor_memory, *(C.byref(x) for x in out), why, len(why))
        assert rc == 0, (shape, lens, hkv, n_layers, why.value.decode())
        return [x.value for x in out]           # blocks without a page, most pages in a block, blocks

    return run


def _length(rng, longest):
    return max(0, int(longest ** rng.random()) - rng.randint(0, 1))


def _batch(rng):
    """Few or many requests; alike, spread over their logarithm, or long ones with a few of one to four pages between."""
    kind, longest = rng.randint(0, 2), rng.choice([200, 3200, 16000, 60000])
    n = rng.choice([1, 2, 3, 4, 6, 9, rng.randint(1, 80)])
    if kind == 0:
        return [longest - rng.randint(0, 40) for _ in range(n)]
    lens = [_length(rng, longest) for _ in range(n)]
    if kind == 2:
        lens = [max(x, longest // 2) for x in lens] + [rng.randint(0, 64) for _ in range(rng.randint(1, 3))]
        rng.shuffle(lens)
    return lens


@pytest.mark.parametrize("shape", list(SHAPES))
def test_every_page_once_and_every_row_merged_once(walk, shape):
    rng = random.Random(7)
    for _ in range(400):
        walk(shape, _batch(rng), rng.choice([1, 1, 2, 4, 8]), rng.choice([4, 16]) if SHAPES[shape][3] else 1)


@pytest.mark.parametrize("shape", ["d256", "d256_two", "d128_one", "d128", "tensor_memory"])
def test_a_short_row_beside_long_ones(walk, shape):
    """A row's share of the blocks counts what opening it costs; it must not get more blocks than it has pages."""
    rng = random.Random(11)
    for lens in ((4000, 32), (2098, 25), (36, 2846), (3000, 40, 3000), (32, 8000), (17, 961), (32, 16000), (16000, 32)):
        for hkv in (1, 2, 4):
            walk(shape, lens, hkv)
    for _ in range(400):
        lens = [rng.randint(200, 3200) for _ in range(rng.randint(2, 7))] + [rng.randint(17, 64)]
        walk(shape, lens, rng.choice([1, 2, 4]))


@pytest.mark.parametrize("B,hkv,tiles", [(1024, 32, 65535), (1024, 33, 65535), (300, 128, 65535), (1024, 8, 65535), (1024, 32, 256),
                                         (1, 32700, 65535)])
def test_positions_of_a_launch_fit_32_bits(lib, B, hkv, tiles):
    """The largest tables that a call accepts: where the positions of all requests pass 2^31 they are decoded in several
    launches, none of which does; smaller ones take one launch."""
    lib.cut_most_positions.restype = C.c_longlong
    most = lib.cut_most_positions(B, hkv, tiles)
    assert 0 < most < 2 ** 31
    one_launch = B * hkv * (tiles + 8 + 3 * 16)
    assert (most == one_launch) == (one_launch < 2 ** 31)
