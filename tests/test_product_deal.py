"""No GPU needed: how the products of a launch are dealt out to thread blocks (fft_deal, fft_dealt of csrc/d2mhe_fft.cuh)."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_04604_b200", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include <vector>
#include "d2mhe_fft.cuh"
static FftWork work(const char* s) {
  return !strcmp(s, "share") ? FFT_WORK_SHARE : !strcmp(s, "share32") ? FFT_WORK_SHARE32 : !strcmp(s, "boot") ? FFT_WORK_BOOT : FFT_WORK_CONVERT;
}
int main() {
  char kind[16];
  unsigned places, rows, parties;
  while (scanf("%15s %u %u %u", kind, &places, &rows, &parties) == 4) {
    const FftDeal d = fft_deal(places, rows, parties, work(kind));
    std::vector<unsigned> seen((size_t)rows * parties);
    bool ok = true;
    for (unsigned b = 0; b < d.blocks; ++b) {
      unsigned first, step;
      const unsigned row = d.whole ? fft_dealt<true>(d, b, first, step) : fft_dealt<false>(d, b, first, step);
      if (row >= rows || first >= parties || step == 0) { ok = false; break; }
      for (unsigned a = first; a < parties; a += step) ++seen[(size_t)row * parties + a];
    }
    for (unsigned n : seen) ok = ok && n == 1;
    printf("%u %u %u %d\n", d.whole, d.split, d.blocks, (int)ok);
  }
}
"""
# transforms that a block of the kernel makes: before its loop over the parties, and in one pass of it
TRANSFORMS = {"share": (2, 2), "share32": (1, 1), "boot": (2, 2), "convert": (2, 4)}


@pytest.fixture(scope="module")
def deal(tmp_path_factory):
    d = tmp_path_factory.mktemp("deal")
    (d / "d.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(d / "d.cc"), "-o", str(d / "d")], check=True)

    def run(calls):
        text = "".join("%s %d %d %d\n" % c for c in calls)
        out = subprocess.run([str(d / "d")], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]

    return run


def _schedule(kind, places, rows, parties, whole, split):
    fixed, each = TRANSFORMS[kind]
    waves = -(-(rows - whole) * split // places)
    return whole // places * (fixed + each * parties) + waves * (fixed + each * -(-parties // split))


@pytest.mark.parametrize("places", [148, 296, 592])
def test_the_calls_compared_with_the_oracle_on_the_gpu_have_mixed_deals(deal, places):
    """The sizes of the GPU tests of just over a wave of blocks, with the 148 multiprocessors of a B200."""
    parties, extra = {592: (7, 38), 296: (5, 14), 148: (4, 16)}[places]
    calls = [("convert", places, places + 2, 2), ("boot", places, places + 2, 2), ("share", places, places + extra, parties)]
    calls += [("share32", 148, 164, 4)]
    assert all(whole == p for (_, p, _, _), (whole, _, _, _) in zip(calls, deal(calls)))


@pytest.mark.parametrize("kind", sorted(TRANSFORMS))
@pytest.mark.parametrize("places", [148, 296, 592])
def test_every_product_is_dealt_once_and_no_even_split_is_shorter(deal, kind, places):
    calls = [(kind, places, rows, parties) for parties in (1, 2, 3, 7, 10, 17, 50)
             for rows in sorted({1, 2, 5, places // 5, places // 2, places - 1, places, places + 1, 2 * places - 1, 2 * places,
                                 2 * places + 2, 3 * places + 7} | set(range(places // 4, 3 * places, 13)) | {176, 88, 355})]
    for (_, _, rows, parties), (whole, split, blocks, ok) in zip(calls, deal(calls)):
        assert ok and whole % places == 0 and blocks == whole + (rows - whole) * split, (rows, parties)
        assert parties > 1 or whole == 0  # one product a row: the kernels have no mixed instance for it
        best = min(_schedule(kind, places, rows, parties, 0, c) for c in range(1, min(parties, 16) + 1))
        assert _schedule(kind, places, rows, parties, whole, split) <= best, (rows, parties, whole, split)
