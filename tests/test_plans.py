"""The launch plans (csrc/plans.h, host arithmetic) over devices of many sizes,
compiled on their own."""

import ctypes
import glob
import os
import re
import subprocess

import pytest

from paper_2607_13205_gb300.build import CSRC

SHIM = r"""
#include "plans.h"
using namespace rolekv;
extern "C" {
int score(int varlen, long units, int chunks, int tiles, int sms) { return score_parts(varlen, units, chunks, tiles, sms); }
long decode(int varlen, long heads, long b, long m_max, long total, int d, int G, int fine, int sms) {
  return decode_split_rows(varlen, heads, b, m_max, total, d, G, fine, sms);
}
void quest(int varlen, long heads, long b, long n_max, long T, long page, long rows, int d, int sms, long* out) {
  const QuestSplit q = quest_split(varlen, heads, b, n_max, T, page, rows, d, sms);
  out[0] = q.ctas;
  out[1] = q.pages;
}
// clusters held, as a GB300 answers (152 SMs), other devices in proportion; or none
void select_(int n_max, long units, int sms, int clusters, int* out) {
  const SelectRoute r = select_route(n_max, units, sms, [&](const SelectRoute& x, bool alone) {
    const int two = x.threads == 512 && !alone;
    return clusters ? static_cast<int64_t>(sms) * (x.ranks == 4 ? (two ? 74 : 36) : (two ? 36 : 15)) / 152 : int64_t{0};
  });
  out[0] = r.mode; out[1] = r.ranks; out[2] = r.threads; out[3] = r.groups; out[4] = r.wide;
}
}
"""

SMS = (1, 7, 14, 30, 76, 132, 148, 152, 160)
ONE, CLUSTER, STREAM = 0, 1, 2


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    d = tmp_path_factory.mktemp("plans")
    src, so = os.path.join(d, "shim.cpp"), os.path.join(d, "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-shared", "-fPIC", "-I", CSRC, "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    L, I = ctypes.c_long, ctypes.c_int
    lib.score.argtypes = [I, L, I, I, I]
    lib.decode.argtypes = [I, L, L, L, L, I, I, I, I]
    lib.decode.restype = L
    lib.quest.argtypes = [I, L, L, L, L, L, L, I, I, ctypes.POINTER(L)]
    lib.quest.restype = None
    lib.select_.argtypes = [I, L, I, I, ctypes.POINTER(I)]
    lib.select_.restype = None
    return lib


def _quest(plans, *args):
    out = (ctypes.c_long * 2)()
    plans.quest(*args, out)
    return out[0], out[1]


def _select(plans, *args):
    out = (ctypes.c_int * 5)()
    plans.select_(*args, out)
    return list(out)


def test_one_source_of_the_sm_count():
    """The device's size is asked for on each call (the current device may
    change), in one place."""
    code = "".join(open(f).read() for f in glob.glob(os.path.join(CSRC, "*")))
    assert len(re.findall(r"cudaDevAttrMultiProcessorCount", code)) == 1
    assert not re.search(r"static int \w*sm\w*|kSms\b", code)


@pytest.mark.parametrize("sms", SMS)
def test_score_gangs_are_resident(plans, sms):
    for chunks in range(1, min(8, sms) + 1):
        for tiles in (1, 4, 5, 33, 64, 200):
            for units in (1, 2, 8, 76, 160, 256, 4096):
                for varlen in (0, 1):
                    x = plans.score(varlen, units, chunks, tiles, sms)
                    assert 1 <= x <= max(1, sms // chunks) and x <= (tiles + 3) // 4


@pytest.mark.parametrize("sms", SMS)
def test_decode_splits(plans, sms):
    for heads, b in ((1, 1), (8, 4), (64, 64)):
        for m in (0, 1, 63, 64, 65, 820, 3277, 131072):
            for varlen in (0, 1):
                for d in (64, 128):
                    coarse = plans.decode(varlen, heads, b, m, m * b, d, 8, 0, sms)
                    fine = plans.decode(varlen, heads, b, m, m * b, d, 8, 1, sms)
                    for r in (coarse, fine):
                        assert 64 <= r <= 1024 and r % 64 == 0
                    # a workspace of the fine splits holds the coarse ones' partials
                    assert -(-m // fine) >= -(-m // coarse)


def test_decode_splits_fill_whole_waves(plans):
    """152 SMs hold 760 CTAs of eight heads' sums at d = 64 (912 of four): the
    splits of 152 units make whole waves of those."""
    for m in (1638, 3277):
        for G, slots in ((4, 912), (8, 760)):
            ctas = 152 * -(-m // plans.decode(0, 152, 1, m, 152 * m, 64, G, 1, 152))
            assert ctas <= slots or ctas % slots > slots // 2 or ctas % slots == 0
    # short packed rows, whose merge costs more than the balance gains
    assert plans.decode(1, 8, 64, 300, 9600, 64, 4, 1, 152) >= 300


@pytest.mark.parametrize("sms", SMS)
def test_quest_splits_cover_the_pages(plans, sms):
    for heads, b in ((1, 1), (8, 4), (512, 1), (7, 64)):
        for n in (1, 15, 512, 2000, 65536):
            for page in (1, 16, 4096):
                for varlen in (0, 1):
                    ctas, per = _quest(plans, varlen, heads, b, n, n * b, page, 128, 128, sms)
                    pages = -(-n // page)
                    assert 1 <= ctas <= pages and ctas * per >= pages and (ctas - 1) * per < pages


def test_quest_splits_fit_the_page_size(plans):
    """152 SMs, three CTAs of eight warps each."""
    # one long packed sequence of small pages takes as many CTAs as the SMs hold
    for n in (65536, 131072, 300000):
        for page in (1, 4, 16):
            ctas, per = _quest(plans, 1, 1, 1, n, n, page, 128, 128, 152)
            assert ctas >= min(256, -(-n // page) // 8) and per * page <= 1024
    # a batch that fills the SMs is not cut into CTAs of fewer pages than warps,
    # nor where the starts cost more than the balance gains
    assert _quest(plans, 0, 256, 1, 4096, 256 * 4096, 512, 128, 128, 152)[0] == 1
    assert _quest(plans, 1, 1, 256, 4096, 256 * 4096, 512, 128, 128, 152)[0] == 1
    assert _quest(plans, 0, 256, 1, 2000, 256 * 2000, 64, 256, 128, 152)[0] == 1
    # one-token pages are bound by their number, not by their bytes
    assert _quest(plans, 0, 300, 1, 1500, 300 * 1500, 1, 128, 128, 152)[0] >= 3


@pytest.mark.parametrize("sms", SMS)
def test_select_routes(plans, sms):
    for n in (0, 1, 2048, 8192, 16384, 16385, 32768, 40960, 40961, 65536, 131072, 131137, 163840, 262144):
        for units in (1, 8, 38, 39, 76, 77, 152, 1024):
            mode, ranks, threads, groups, wide = _select(plans, n, units, sms, 1)
            assert groups * 4 * ranks >= n + 3
            assert mode == STREAM or groups * 4 <= 40960 + 128       # a rank's keys fit its shared memory
            assert (mode == CLUSTER) == (ranks > 1) and ranks in (1, 2, 4, 8)
            assert threads in ((512, 1024) if mode == CLUSTER else (1024,) if wide else (256, 512))
            assert wide or groups * 4 <= 16384 + 128
            # a device that holds no such cluster: another route, not a refusal
            mode, ranks, threads, groups, wide = _select(plans, n, units, sms, 0)
            assert mode == (STREAM if n > 40960 else ONE) and ranks == 1


def test_select_routes_by_waves(plans):
    """A cluster that has no SM of its own left, or a wave too many, is slower
    than one CTA or streaming."""
    def mode(n, units, sms=152):
        return _select(plans, n, units, sms, 1)[:2]
    assert mode(16385, 36) == [CLUSTER, 4] and mode(16385, 38) == [ONE, 1] and mode(24000, 38) == [ONE, 1]
    assert mode(32768, 38) == [CLUSTER, 4] and mode(32768, 39) == [ONE, 1]
    assert mode(40961, 72) == [CLUSTER, 4] and mode(40961, 76) == [STREAM, 1] and mode(65536, 76) == [STREAM, 1]
    assert mode(100000, 64) == [CLUSTER, 4] and mode(100000, 76) == [STREAM, 1]
    assert mode(150000, 14) == [CLUSTER, 8] and mode(150000, 20) == [CLUSTER, 4]
    assert mode(262144, 38) == [CLUSTER, 8]
    # the plan follows the device
    assert mode(65536, 57) == [CLUSTER, 4] and mode(65536, 57, 76) == [STREAM, 1]
    # threads: one CTA of a row just beyond 16384 tokens, alone on its SM
    assert _select(plans, 16385, 39, 152, 1)[2] == 1024 and _select(plans, 16385, 300, 152, 1)[2] == 512
    assert _select(plans, 16384, 39, 152, 1)[2] == 512
