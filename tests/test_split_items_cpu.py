"""The split Hamiltonian's work items (csrc/partition.cpp): every pair of functions of a batch is computed
exactly once per K segment, in no more items than the blocks need."""
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent
CSRC = ROOT / "paper_1912_06636_gb300" / "csrc"

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "nao_internal.h"
int main(int argc, char **argv) {
    const int TN = atoi(argv[1]), S = atoi(argv[2]), F = atoi(argv[3]), P = atoi(argv[4]);
    BlockPairs kept;
    for (int a = 5; a < argc; a++) {
        const int N = atoi(argv[a]), nseg = nao_split_h_nseg(P, S, F), nr = (N + 31) / 32;
        std::vector<HTask> items;
        nao_split_h_items(7, P, N, TN, S, items, kept, F);
        std::vector<unsigned char> hit((size_t)nseg * N * N, 0);
        for (const HTask &t : items) {
            if (t.batch != 7 || t.seg() >= nseg) return 2;
            for (int x = 0; x < 4; x++) {
                const uint32_t r = t.row(x);
                if (r == kNoRows) continue;
                if ((int)r >= nr) return 3;
                for (int i = (int)r * 32; i < (int)r * 32 + 32 && i < N; i++)
                    for (int j = t.tj() * TN; j < (t.tj() + 1) * TN && j < N; j++) {
                        // the kernel's rule: off-diagonal blocks of the 32-wide form are whole, the rest j >= i
                        if (!(TN == 32 && (int)r != t.tj()) && j < i) continue;
                        unsigned char &h = hit[((size_t)t.seg() * N + (i < j ? i : j)) * N + (i < j ? j : i)];
                        if (h++) return 4;
                    }
            }
        }
        for (int q = 0; q < nseg; q++)
            for (int i = 0; i < N; i++)
                for (int j = i; j < N; j++)
                    if (hit[((size_t)q * N + i) * N + j] != 1) return 5;
        const int need = nr * (nr + 1) / 2;
        if (TN == 32 && (int)items.size() != nseg * (need > 4 * nr ? (need + 3) / 4 : nr)) return 6;
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("items")
    (d / "main.cpp").write_text(MAIN)
    cmd = ["g++", "-O2", "-std=c++17", f"-I{ROOT / 'include'}", f"-I{CSRC}", "-I/usr/local/cuda/include", str(d / "main.cpp"),
           str(CSRC / "partition.cpp"), "-o", str(d / "items")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return str(d / "items")


@pytest.mark.parametrize("TN,S,F,P", [(32, 14, 1, 200), (32, 12, 0, 200), (32, 12, 0, 512), (48, 10, 0, 200), (48, 4, 0, 512)])
def test_every_pair_once(program, TN, S, F, P):
    # edges of the 32- and 48-function blocks and of 128 rows, odd and even block counts, large bases
    sizes = [1, 15, 16, 31, 32, 33, 47, 48, 49, 64, 65, 95, 96, 97, 127, 128, 129, 160, 161, 200, 224, 225, 256, 257, 320, 384,
             440, 510, 570, 768, 1000, 1343]
    r = subprocess.run([program, str(TN), str(S), str(F), str(P), *map(str, sizes)], capture_output=True)
    assert r.returncode == 0, r.returncode
