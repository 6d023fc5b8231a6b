"""The z chunk of the moment kernel (moment_chunk in lbgb_moment.cu), compiled
for the host: the choice of an exhaustive search over the numbers of chunks,
found without looking at all of them (a long lattice has as many as planes, and
the choice is made in every step: 2000 steps of 2^20 planes in 2 s at most)."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
struct Lattice { int nz; };
static int sms = 152;
static int device_sms() { return sms; }
%s
static int exhaustive(const Lattice& L, long long tiles, int per_sm) {
    const long long R = (long long)device_sms() * per_sm;
    int best = L.nz;
    long long cost = -1;
    for (int n = 1; n <= L.nz; n++) {
        const int zc = (L.nz + n - 1) / n;
        const long long B = tiles * ((L.nz + zc - 1) / zc), c = ((B + R - 1) / R) * (zc + 4);
        if (cost < 0 || c < cost) cost = c, best = zc;
        if (zc <= 2) break;
    }
    return best;
}
int main() {
    long long tiles = 1;
    for (int nz = 4; nz < 1200; nz++)
        for (int k = 0; k < 12; k++) {
            tiles = (tiles * 48271 + 11) %% (k < 6 ? 61 : 20011) + 1;
            const Lattice L = {nz};
            if (moment_chunk(L, tiles, 3 + k %% 2) != exhaustive(L, tiles, 3 + k %% 2)) return printf("nz %%d tiles %%lld\n", nz, tiles), 1;
        }
    const auto t0 = std::chrono::steady_clock::now();
    long long sum = 0;
    for (int k = 0; k < 2000; k++) sum += moment_chunk(Lattice{(1 << 20) + k}, 1 + k %% 9, 3);
    const double t = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    printf("%%lld %%g s\n", sum, t);
    return t > 2.0;
}
"""


def test_moment_chunk(tmp_path):
    with open(os.path.join(ROOT, "paper_2004_04080_gb300", "csrc", "lbgb_moment.cu")) as f:
        fn = re.search(r"static int moment_chunk\(.*?\n}\n", f.read(), flags=re.S).group(0)
    src, exe = tmp_path / "chunk.cpp", tmp_path / "chunk"
    src.write_text(PROGRAM % fn)
    subprocess.run(["g++", "-O2", "-o", str(exe), str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0, run.stdout
