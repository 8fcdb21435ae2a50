"""The sizes of an index build's partition (csrc/xm_plan.cuh, host arithmetic):
for every zone count the library accepts and row counts over every
power-of-two window, the bins fit the shared-memory arrays that count them."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1611_08494_gb300", "csrc")

PLAN = r"""
#include <stdio.h>
#include <vector>
#include "xm_plan.cuh"
using namespace xm;
int main() {
    std::vector<int64_t> rows = {0, 1, 2147483647LL};
    for (int b = 1; b < 31; b++)
        for (int64_t k = 0; k < 32; k++) {  // the window [2^b, 2^(b+1)) and its edges
            const int64_t n = (1LL << b) + ((k << b) >> 5);
            rows.push_back(n);
            rows.push_back(n - 1);
        }
    const int64_t more[] = {384000, 3000000, 12000000, 12000031, 25000000, 50000000, 100000000,
                            200000000, 300000000};
    for (int64_t n : more) rows.push_back(n);
    long most = 0;
    for (int32_t nz = 18; nz <= kMaxZones; nz++)
        for (int64_t n : rows) {
            const BuildPlan p = build_plan(n, nz);
            bool ok = p.cells_cap >= nz;
            if (!p.two) {
                ok &= p.units_cap <= kMaxUnits && p.nbins == 0;
            } else {
                // the digit of the last zone's sources, were they the last rows
                const int64_t last = (n >> p.kb) + ((nz - 1) >> kBinZoneBits);
                ok &= p.kb >= kUnitRowBits && p.kb < 32 && p.nbins <= kMaxBins && last < p.nbins;
            }
            if (!ok) {
                printf("n %lld nz %d: kb %d, %d bins, %lld units\n", (long long)n, nz, p.kb, p.nbins,
                       (long long)p.units_cap);
                return 1;
            }
            if (p.nbins > most) most = p.nbins;
        }
    printf("at most %ld bins\n", most);
    return 0;
}
"""


def test_bins_fit_their_arrays(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "plan.cpp"
    src.write_text(PLAN)
    exe = str(tmp_path / "plan")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I" + CSRC, "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


FOLD = r"""
#include <stdio.h>
#include "xm_plan.cuh"
using namespace xm;
// Two 16-bit counters of a word under the order of events that holds a fold back
// the longest: all that is added between two barriers, then the folds.
int main() {
    const uint32_t per = kCountThreads * kCountLoads * kFoldLoops;
    for (int which = 0; which < 2; which++)
        for (uint32_t step = 1; step <= per; step = step < 3 ? step + 1 : step * 3) {
            uint32_t word = 0, other = 0x7FFF;
            word += other << (16 * !which);  // the neighbour's count, which must not change
            uint64_t added = 0, folded = 0;
            const int sh = 16 * which;
            for (int window = 0; window < 40; window++) {
                const uint32_t n = per - (window * step) % per;
                uint32_t folds = 0;
                for (uint32_t k = 0; k < n; k++) {
                    folds += ((word >> sh) & 0xFFFFu) == 0x7FFFu;
                    word += 1u << sh;
                }
                added += n;
                for (uint32_t k = 0; k < folds; k++) {
                    word -= 0x8000u << sh;
                    folded += 0x8000;
                }
                if (((word >> (16 * !which)) & 0xFFFFu) != other ||
                    folded + ((word >> sh) & 0xFFFFu) != added) {
                    printf("window %d of %u sources\n", window, n);
                    return 1;
                }
            }
        }
    return 0;
}
"""


def test_counters_of_zones_hold(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "fold.cpp"
    src.write_text(FOLD)
    exe = str(tmp_path / "fold")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I" + CSRC, "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
