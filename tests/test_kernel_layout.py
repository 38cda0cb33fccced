"""Layout identities of the kernels, on the constants and index functions of the CUDA headers as they
are compiled (a host program prints them): which line elements and frequencies a thread's registers
hold, where the half chirp table is read, which registers are the middle half P/4 .. 3P/4, and that
the exchanges of the long lines are free of shared-memory bank conflicts."""

import json
import os
import subprocess

import pytest

from paper_2407_20304_gb300 import build as bld

LENGTHS = [1 << k for k in range(4, 13)] + [3 << k for k in range(4, 11)]
PROGRAM = """
#include <cstdio>
#include "holo_kernels.cuh"
using namespace holo;
template <int P> void dump() {
  using L = Line<P>;
  std::printf("\\"%d\\": {\\"E\\": %d, \\"T\\": %d, \\"smem\\": %d, \\"r3\\": %d, \\"half\\": %d, "
              "\\"row_pitch\\": %d, \\"row_unit\\": %d, \\"row_threads\\": %d, "
              "\\"cols\\": %d, \\"col_threads\\": %d, \\"col_pitch\\": %d, \\"dcols\\": %d, "
              "\\"dcol_threads\\": %d, \\"dcol_pitch\\": %d",
              P, L::E, L::T, L::SMEM, (int)L::R3, (int)half_form_ok<P>(), RowCfg<P>::LS,
              RowCfg<P>::U, RowCfg<P>::NT, ColCfg<P>::C, ColCfg<P>::NT, ColCfg<P>::LS,
              DColCfg<P>::C, DColCfg<P>::NT, DColCfg<P>::LS);
  if constexpr (!L::R3) {
    std::printf(", \\"R\\": %d, \\"RS\\": %d, \\"at\\": [", L::R, L::RS);
    for (int k = 0; k < L::E; ++k) std::printf("%s%d", k ? "," : "", L::at(k));
    std::printf("]");
  }
  std::printf(", \\"map\\": [");  // element, frequency, chirp entry, middle half
  for (int t = 0; t < L::T; ++t)
    for (int c = 0; c < L::E; ++c)
      std::printf("%s[%d,%d,%d,%d]", t + c ? "," : "", L::pos(t, c), L::fpos(t, c),
                  ChirpAt<P>::at(t, c), (int)mid_reg<P>(c));
  std::printf("]}");
}
int main() {
  std::printf("{");
%s
  std::printf("}");
}
"""


@pytest.fixture(scope="module")
def layouts(tmp_path_factory):
    nvcc = bld.nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except OSError:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("layout")
    body = '  std::printf(",");\n'.join(f"  dump<{P}>();\n" for P in LENGTHS)
    (d / "layout.cu").write_text(PROGRAM.replace("%s\n", body, 1))
    subprocess.run([nvcc, "-std=c++17", *bld.ARCH, "-I", os.path.join(bld.ROOT, "include"), "-I",
                    bld.CSRC, str(d / "layout.cu"), "-o", str(d / "layout")], check=True)
    out = subprocess.run([str(d / "layout")], capture_output=True, text=True, check=True).stdout
    return {int(k): v for k, v in json.loads(out).items()}


@pytest.mark.parametrize("P", LENGTHS)
def test_elements_frequencies_and_chirp_entries(layouts, P):
    L = layouts[P]
    assert L["E"] * L["T"] == P and L["smem"] >= P
    pos, freq, chirp, mid = zip(*L["map"])
    assert sorted(pos) == list(range(P)) and sorted(freq) == list(range(P))
    assert all(e == min(f, P - f) for e, f in zip(chirp, freq))
    if not L["r3"]:
        assert pos == freq and sorted(L["at"]) == list(range(L["E"]))
        assert all(m == (P // 4 <= x < 3 * P // 4) for x, m in zip(pos, mid))
    if L["half"]:
        assert not L["r3"] and (P // 2) % L["cols"] == 0


@pytest.mark.parametrize("P", LENGTHS)
def test_blocks_are_whole_warps(layouts, P):
    """Tensor memory is read by whole warps, and units of the row passes synchronise by themselves."""
    L = layouts[P]
    assert L["cols"] * L["T"] == L["col_threads"] and L["dcols"] * L["T"] == L["dcol_threads"]
    assert L["col_threads"] % 32 == 0
    if not L["r3"]:
        assert L["row_unit"] % 32 == 0 and L["row_threads"] % L["row_unit"] == 0
        assert L["row_unit"] % L["T"] == 0


def conflicts(P, L, C, pitch):
    """Extra passes of a warp's accesses to the exchange buffer, lanes t * C + g (g the line of a
    column pass; rows: C = 1): 8-byte accesses go by half warps, 16-byte ones by quarter warps."""
    E, T, R, RS = L["E"], L["T"], L["R"], L["RS"]

    def extra(addr, words, group):
        worst = 0
        for l0 in range(0, T * C, group):
            banks = {}
            for lane in range(l0, min(l0 + group, T * C)):
                a = 2 * (addr(lane // C) + pitch * (lane % C))
                for i in range(words):
                    banks.setdefault((a + i) % 32, set()).add(a + i)
            worst = max(worst, max(len(b) for b in banks.values()) - 1)
        return worst

    out = [extra(lambda t: 5 * RS + t, 2, 16)]                         # exchange 1, writes
    if R == 1:
        out.append(extra(lambda t: t * RS + 2, 4, 8))                  # rows, two values a read
    else:
        out.append(extra(lambda t: t % E * RS + t // E + R * 3, 2, 16))
        out.append(extra(lambda t: t % E * RS + t // E * R + 2 * R * R + 1, 2, 16))
    return out


# T >= 16 (with fewer threads to a line the many columns of a block meet on some banks)
@pytest.mark.parametrize("P", [512, 768, 1024, 2048, 4096])
def test_exchanges_are_free_of_bank_conflicts(layouts, P):
    L = layouts[P]
    if L["T"] >= 32:
        assert not any(conflicts(P, L, 1, L["row_pitch"]))
    assert not any(conflicts(P, L, L["cols"], L["col_pitch"]))
    assert not any(conflicts(P, L, L["dcols"], L["dcol_pitch"]))
