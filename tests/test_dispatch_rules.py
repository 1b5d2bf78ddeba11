"""The rules that choose a kernel's variant (csrc/dispatch.h), compiled for the host: which side
a call of given sizes takes, at the measured crossings and beyond."""

import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_28699_gb300", "csrc")
SOURCE = r"""
#include "dispatch.h"
extern "C" {
void plan(int batch, int heads, int max_pages, int scheme, int bits, int group, int append, long available, long* out) {
    const wc::DecodePlan p = wc::plan_decode(batch, heads, max_pages, 152, scheme, bits, group, append != 0, (size_t)available);
    out[0] = p.splits, out[1] = p.pages_per_split, out[2] = (long)p.total, out[3] = p.two_per_sm;
}
int repair_wide(long cells, int threads) { return wc::repair_wide(cells, threads); }
int write_two_tasks(int scheme, int bits, long n_tok, long heads) { return wc::write_two_tasks(scheme, bits, n_tok, heads); }
int pairs_wide(int n_tok, int aligned, int heads, int resident) { return wc::pairs_wide(n_tok, aligned != 0, heads, resident); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{CSRC}", "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    return ctypes.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("cells,threads,wide", [(28, 1024, 1), (152, 1024, 1), (153, 1024, 0), (280, 512, 1), (448, 512, 0),
                                                (1216, 128, 1), (2800, 128, 0), (8400, 64, 0), (229376, 64, 0)])
def test_repair_ctas_are_wide_while_the_chip_is_half_full(lib, cells, threads, wide):
    """One warp per small cell left a few cells with long chains: 28 of 128 pages took 7.5 us, 4.8 before."""
    assert lib.repair_wide(ctypes.c_long(cells), threads) == wide


@pytest.mark.parametrize("scheme,bits,n_tok,heads,two", [
    (0, 8, 15, 8, 0), (0, 8, 16, 8, 1), (1, 8, 16, 1, 1),
    (0, 10, 15, 64, 0), (0, 10, 700, 8, 0), (0, 10, 1064, 8, 0), (0, 10, 1065, 8, 1), (0, 10, 8512, 1, 0), (0, 10, 32768, 4, 1),
    (2, 8, 2047, 8, 0), (2, 8, 2048, 8, 1), (2, 8, 131072, 1, 1)])
def test_write_tasks(lib, scheme, bits, n_tok, heads, two):
    """700 x 8 tokens and heads at 10 bits: 5.8 us with two tasks, 4.6 with one."""
    assert lib.write_two_tasks(scheme, bits, ctypes.c_long(n_tok), ctypes.c_long(heads)) == two


@pytest.mark.parametrize("n_tok,aligned,heads,resident,wide", [
    (4095, 1, 4, 14, 0), (4096, 1, 4, 14, 1), (4096, 0, 4, 14, 0), (4096, 1, 14, 14, 1), (4096, 1, 15, 14, 0),
    (65536, 1, 32, 14, 0),                     # more clusters than fit at once: 93 us, 80 narrow
    (65536, 1, 1, 0, 0), (65536, 1, 8, 4, 0)])   # a device that cannot place them: the narrow cluster serves
def test_pair_clusters_are_wide_while_resident(lib, n_tok, aligned, heads, resident, wide):
    assert lib.pairs_wide(n_tok, aligned, heads, resident) == wide


def _plan(lib, batch, heads, max_pages, scheme=0, bits=8, group=1, append=0, available=-1):
    out = (ctypes.c_long * 4)()
    lib.plan(batch, heads, max_pages, scheme, bits, group, append, ctypes.c_long(available), out)
    return list(out)


@pytest.mark.parametrize("scheme,batch,heads,max_pages,group,append,flat", [
    (0, 32, 8, 40, 1, 0, 0), (0, 32, 8, 41, 1, 0, 1), (0, 1, 8, 400, 7, 0, 0),
    (0, 75, 8, 5, 1, 0, 0), (0, 76, 8, 5, 1, 0, 1), (0, 76, 8, 5, 3, 0, 1), (0, 76, 8, 5, 4, 0, 0),   # 608 units: few query heads
    (0, 189, 8, 5, 5, 0, 0), (0, 190, 8, 5, 5, 0, 1), (0, 190, 8, 5, 6, 0, 0), (0, 1000, 8, 4, 8, 0, 0),
    (0, 19, 8, 5, 8, 1, 0), (0, 20, 8, 5, 8, 1, 1), (0, 1000, 8, 4, 8, 1, 1),                          # the append
    (2, 1000, 8, 30, 1, 0, 0), (2, 20, 8, 31, 1, 0, 1), (1, 1000, 8, 400, 1, 0, 0)])
def test_short_block_tables(lib, scheme, batch, heads, max_pages, group, append, flat):
    """200 sequences of 5 pages over 8 KV heads of one query head: 48.1 us split, 39.5 before, 38.5 flattened."""
    assert (_plan(lib, batch, heads, max_pages, scheme, group=group, append=append)[1] == 0) == bool(flat)


def test_workspace_does_not_depend_on_the_variant(lib):
    for scheme, bits in ((0, 8), (0, 10), (2, 8), (1, 8)):
        for batch in (1, 2, 19, 20, 76, 200, 1000):
            for heads in (1, 4, 8):
                for pages in (1, 5, 30, 31, 40, 41, 500):
                    plans = [_plan(lib, batch, heads, pages, scheme, bits, g, a) for g in (1, 3, 4, 5, 8) for a in (0, 1)]
                    assert len({p[2] for p in plans}) == 1
                    for splits, pps, total, _ in plans:
                        partials = splits + batch * heads if pps == 0 else splits * batch * heads
                        assert 256 + partials * 8 * 140 * 4 <= total
                        assert pps == 0 or splits * pps >= pages


@pytest.mark.parametrize("batch,heads,max_pages,two", [
    (37, 8, 5, 0), (38, 8, 5, 1), (38, 8, 24, 1), (38, 8, 25, 0), (76, 8, 48, 1), (76, 8, 49, 0), (300, 4, 94, 1), (300, 4, 95, 0),
    (400, 4, 38, 1), (1000, 1, 16, 1), (1000, 8, 4, 1), (16, 4, 20, 0), (32, 8, 5, 0), (1, 304, 24, 1)])
def test_ten_bit_short_sequences_take_two_ctas_per_sm(lib, batch, heads, max_pages, two):
    """400 sequences of 2 pages over 4 KV heads: 70 us on warp pairs with one CTA per SM, 47 with two."""
    splits, pps, total, got = _plan(lib, batch, heads, max_pages, 0, 10)
    assert got == two
    assert not two or pps > 0
    for scheme, bits in ((0, 8), (1, 8), (2, 8)):
        assert _plan(lib, batch, heads, max_pages, scheme, bits)[3] == 0


def test_ten_bit_plans_fit_what_they_are_given(lib):
    """A workspace of the size the 10-bit dither was first given holds whatever plan it then gets."""
    for batch in (2, 16, 76, 100, 200, 400, 1000):
        for heads in (1, 2, 4, 8):
            for pages in (1, 5, 20, 41, 60, 100, 400, 2048):
                want = _plan(lib, batch, heads, pages, 0, 10)
                small = _plan(lib, batch, heads, pages, 0, 10, available=0)
                assert small[2] <= want[2]
                again = _plan(lib, batch, heads, pages, 0, 10, available=small[2])
                assert again == small
                for splits, pps, total, two in (want, small):
                    partials = splits + batch * heads if pps == 0 else splits * batch * heads
                    assert 256 + partials * 8 * 140 * 4 <= total
