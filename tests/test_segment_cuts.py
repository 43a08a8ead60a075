"""How one long sequence is cut into segments, over layers of few and of many heads: the longest segment is what a pass takes."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_11231_b200", "csrc")
SMS = 148


@pytest.fixture(scope="module")
def cuts(tmp_path_factory):
    d = tmp_path_factory.mktemp("cuts")
    src = d / "cuts.cpp"
    src.write_text('#include "segments.h"\n'
                   'static int out(const lkv::Cut &c, int *at) { for (int i = 0; i <= c.n; ++i) at[i] = c.at[i]; return c.n; }\n'
                   'extern "C" int gdn(int b, int h, int s, int *at) { return out(lkv::gdn_cut_blocks(b, h, s), at); }\n'
                   'extern "C" int ssd(int b, int p, int s, int *at) { return out(lkv::ssd_cut_blocks(b, p, s), at); }\n')
    so = d / "cuts.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(src)], check=True)
    lib = ctypes.CDLL(str(so))

    def cut(f, blocks, heads):
        at = (ctypes.c_int * 17)()
        n = f(blocks, heads, SMS, at)
        assert 1 <= n <= 16 and at[0] == 0 and at[n] == blocks
        sizes = [at[i + 1] - at[i] for i in range(n)]
        assert min(sizes) >= 1
        return sizes

    return lambda name, blocks, heads: cut(getattr(lib, name), blocks, heads)


@pytest.mark.parametrize("blocks", [1, 15, 16, 17, 31, 40, 52, 64, 100, 128, 256, 257, 384, 1000])
def test_gdn_cut(cuts, blocks):
    for heads in range(1, 150):
        sizes = cuts("gdn", blocks, heads)
        n, longest = len(sizes), max(sizes)
        if n == 1:
            continue
        slots = SMS // heads
        # one round of CTAs in both passes; a CTA that runs the short segment's state and then its transition is no longer than the rest
        assert n <= slots and (2 * n - 3 <= slots or (2 * n - 3 == slots + 1 and 2 * sizes[n - 2] <= longest + 1))
        assert sizes[n - 2] <= longest and all(s == longest for s in sizes[:n - 2] + sizes[n - 1:])
        assert 2 * longest + (n - 2) < blocks, (heads, sizes)   # shorter than the plain scan's chain
        assert longest <= 2 * blocks // (2 * n - 1) + 1         # no segment takes what the others leave


def test_gdn_cut_of_a_long_sequence_uses_the_gpu(cuts):
    """16384 tokens: the fewer the heads, the more segments (up to 16), never a longer chain than a layer of more heads has."""
    chain = [2 * max(s) if len(s) > 1 else 256 for s in (cuts("gdn", 256, h) for h in range(1, 149))]
    assert chain == sorted(chain)
    assert chain[0] == chain[3] == 2 * 16 and chain[31] == 2 * 74
    assert chain[48] == 2 * 86 and chain[73] == 256   # three CTAs a head: three segments; two: not enough for any


@pytest.mark.parametrize("blocks", [1, 23, 24, 64, 65, 129, 192, 1000])
def test_ssd_cut(cuts, blocks):
    for pairs in range(1, 150):
        sizes = cuts("ssd", blocks, pairs)
        n = len(sizes)
        if n > 1:
            assert n <= SMS // pairs and max(sizes) == sizes[0] <= blocks // n + n and min(sizes[:-1]) == sizes[0]
