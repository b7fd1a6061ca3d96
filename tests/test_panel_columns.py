"""The panel kernel's bitmaps of tableau columns (csrc/gbs_colbits.h), on the CPU.

An overlapped panel lists the 16-byte vectors that hold a column it does not
leave out, in shared memory sized for the tableau's own vectors.  Panels that get
every column and panels that do not follow one another in any order here, at
widths around a whole word and a whole vector, with random columns basic.
"""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1804_04737_gb300", "csrc")

PANELS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "gbs_colbits.h"

int main() {
    unsigned rng = 12345u;
    auto rnd = [&]() { return rng = rng * 1664525u + 1013904223u, rng >> 16; };
    const int widths[] = {1, 2, 3, 4, 5, 17, 30, 31, 32, 33, 34, 36, 63, 64, 65, 95, 97, 1000, 4097, 4609};
    int bad = 0;
    for (int VW : {2, 4})
        for (int N : widths) {
            const int nwords = (N + 31) / 32, nvec = (N + VW - 1) / VW;
            std::vector<unsigned> prev(nwords, ~0u), stay(nwords);
            std::vector<char> was(N, 1), is(N);  // columns unchanged in the panel before, in this one
            for (int panel = 0; panel < 60; ++panel) {
                const bool all = rnd() % 3 == 0;
                const int dense = rnd() % 3;  // no column stays, every one, some
                for (int w = 0; w < nwords; ++w) stay[w] = gbs::past_end(w, N);
                for (int j = 0; j < N; ++j) {
                    is[j] = dense == 1 || (dense == 2 && rnd() % 4 != 0);
                    if (is[j]) stay[j / 32] |= 1u << (j % 32);
                }
                int listed = 0;
                for (int w = 0; w < nwords; ++w) {
                    const unsigned out = gbs::left_out_of_panel(prev[w], stay[w], all, gbs::past_end(w, N));
                    for (int u = 0; u < 32 / VW; ++u) {
                        const int v = w * (32 / VW) + u;
                        bool want = false;  // a column of the tableau that changed in either panel
                        for (int j = v * VW; j < (v + 1) * VW && j < N; ++j) want |= !(was[j] && is[j]);
                        const bool kept = gbs::vector_kept(out, u, VW);
                        if (kept != want || (kept && v >= nvec)) ++bad;
                        listed += kept;
                    }
                }
                if (listed > nvec) ++bad;
                for (int j = 0; j < N; ++j) was[j] = all ? 0 : is[j];
            }
        }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""

BASIS = r"""
#include <climits>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include "gbs_colbits.h"

int main() {
    int bad = 0;
    for (int N : {1, 31, 32, 33, 70}) {
        const int nwords = (N + 31) / 32;
        for (int leaving : {0, N / 2, N - 1, N, N + 1, 32 * nwords, 1 << 20, INT_MAX, -1, -33, INT_MIN}) {
            unsigned mem[16], want[16];  // guards, basic, guards, stay, guards
            for (unsigned &w : mem) w = 0xffffffffu;
            std::memcpy(want, mem, sizeof mem);
            unsigned *basic = mem + 2, *stay = mem + 9;
            const int entering = N / 3;
            basic[entering / 32] &= ~(1u << entering % 32);
            want[2 + entering / 32] |= 1u << entering % 32;
            if (leaving >= 0 && leaving < N) {
                if (leaving != entering) want[2 + leaving / 32] &= ~(1u << leaving % 32);
                want[9 + leaving / 32] &= ~(1u << leaving % 32);
            }
            gbs::change_basis(basic, stay, leaving, entering, N);
            bad += std::memcmp(mem, want, sizeof mem) != 0;
        }
    }
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def _run(tmp_path, source):
    src, exe = tmp_path / "cols.cpp", tmp_path / "cols"
    src.write_text(source)
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=undefined", "-fno-sanitize-recover=all",
                    "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], capture_output=True, text=True)


def test_panels_list_only_their_own_vectors(tmp_path):
    r = _run(tmp_path, PANELS)
    assert r.returncode == 0, r.stdout + r.stderr


def test_leaving_column_out_of_range_marks_nothing(tmp_path):
    r = _run(tmp_path, BASIS)
    assert r.returncode == 0, r.stdout + r.stderr
