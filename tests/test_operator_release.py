"""What a plan keeps when the autotuner gives its operators back (release_operators.h), on
the host with made-up pointers: the synthesis operators go on using the row offsets and
the tile list."""

import os
import subprocess

from helpers import ROOT

CSRC = os.path.join(ROOT, "paper_1904_10514_gb300", "csrc")
SRC = r"""
#include <cstdio>
#include <set>
#include "release_operators.h"
static hpx_plan_s* make(bool syn) {
    hpx_plan_s* P = new hpx_plan_s();
    char* at = nullptr;
    auto fake = [&](auto*& q) { at += 256; q = (std::remove_reference_t<decltype(q)>)at; };
    fake(P->fusedM); fake(P->fusedOff); fake(P->fusedTiles); fake(P->tcOff); fake(P->tcFirst);
    fake(P->tcRinv); fake(P->bscale); fake(P->bpk);
    if (syn) fake(P->synM);
    P->bytes = 100; P->fused_bytes = 60; P->use_tc = true;
    return P;
}
int main() {
    for (int syn = 0; syn < 2; ++syn) {
        hpx_plan_s* P = make(syn);
        void *off = P->fusedOff, *tiles = P->fusedTiles, *S = P->synM;
        std::multiset<void*> gone;
        hpx::release_operators(P, [&](void* q) { gone.insert(q); });
        printf("%d %d %d %d %d %d %d %d %d %d\n", (int)gone.size(), (int)gone.count(off), (int)gone.count(tiles),
               (int)gone.count(S), P->fusedOff == off, (void*)P->fusedTiles == tiles, P->synM == S,
               !P->fusedM && !P->bpk && !P->use_tc, (int)P->bytes, (int)P->flags);
    }
}
"""


def test_synthesis_keeps_offsets_and_tiles(tmp_path):
    src, exe = tmp_path / "release.cu", tmp_path / "release"
    src.write_text(SRC)
    r = subprocess.run([os.environ.get("NVCC", "nvcc"), "-std=c++17", "-I" + CSRC, "-o", str(exe), str(src)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split("\n")
    # without synthesis operators everything goes, with them the offsets and the tiles stay
    assert out[0] == "8 1 1 0 0 0 1 1 40 1"
    assert out[1] == "6 0 0 0 1 1 1 1 40 1"
