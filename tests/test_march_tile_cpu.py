"""The tiles of the marching level kernels over every pair of child and parent
grid an array can have, from equal grids to a parent a thousand times finer
(pitches of tens of wavelengths): the search ends, a CTA's threads and copies stay
within its bounds, and the column chunks and tap groups cover the row and the
stencil.  The host arithmetic (csrc/march_tile.h) is compiled here and fed the
stencil starts of the grids."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_21724_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "march_tile.h"
int main() {
  int kind, most, nk, hn, pack, nbox, nph, NT, width, boxcopies, extra;
  while (std::scanf("%d %d %d %d %d %d %d %d %d %d %d", &kind, &most, &nk, &hn, &pack, &nbox, &nph, &NT, &width, &boxcopies,
                    &extra) == 11) {
    std::vector<int> start(nph);
    for (int& s : start) if (std::scanf("%d", &s) != 1) return 1;
    int taps = width;
    const smr::MarchTile m =
        kind ? smr::anterp_tile(most, nk, hn, hn, pack, nbox, nph, NT, start, width, extra, &taps)
             : smr::march_tile(most, nk, hn, hn, pack, nbox, nph, NT, start, width, boxcopies, extra);
    std::printf("%d %d %d %d %d %d %d %d\n", taps, m.ncol, m.nck, m.cc, m.nbx, m.T, m.nbg, m.nhk);
  }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("tile")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "main")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(d / "main.cpp"), "-o", exe], check=True)
    return exe


def stencils(nc, npar):
    """First child column of every parent column's four phi taps, and first parent
    column and number of the transposed ones."""
    dphi = 2.0 * np.pi / nc
    start = np.floor(2.0 * np.pi * np.arange(npar) / npar / dphi).astype(int) - 1
    first, last = np.full(nc, 1 << 30), np.full(nc, -(1 << 30))
    for turn in (-1, 0, 1):
        for b in range(4):
            j = start + b + turn * nc
            ok = (j >= 0) & (j < nc)
            np.minimum.at(first, j[ok], np.arange(npar)[ok] + turn * npar)
            np.maximum.at(last, j[ok], np.arange(npar)[ok] + turn * npar)
    for j in range(nc):
        if last[j] < first[j]:
            first[j] = last[j] = first[j - 1] if j else 0
    return start, first, max(7, int((last - first).max()) + 1)


def test_tiles_of_every_grid_pair(program):
    asked, lines = [], []
    for L0 in (2, 3, 5, 10, 16, 40, 97):
        for L1 in sorted({max(2, int(round(L0 * f))) for f in np.geomspace(0.2, 1000, 40)} & set(range(2200))):
            nc, npar = 2 * L0 + 2, 2 * L1 + 2
            start, first, pm = stencils(nc, npar)
            for f64 in (0, 1):
                hn = 2 if f64 else 1
                for nbox, R in ((1, 1), (37, 3)):
                    for kind, most, nk, nph, s, width, bc, extra in (
                            (0, 224 if f64 else 128, 3, npar, start, 4, 4, 0),
                            (1, 192 if f64 else 128, 4 if pm <= 8 else 16, nc, first, pm, 1, hn)):
                        asked.append((kind, most, nk, hn, nbox, R, nph, s, width, bc, extra))
                        lines.append(" ".join(map(str, [kind, most, nk, hn, int(not f64), nbox, nph, hn * R, width, bc,
                                                        extra, *s.tolist()])))
    r = subprocess.run([program], input="\n".join(lines), capture_output=True, text=True, timeout=120)
    got = [tuple(map(int, ln.split())) for ln in r.stdout.splitlines()]
    assert len(got) == len(asked)
    for (kind, most, nk, hn, nbox, R, nph, s, width, bc, extra), (taps, ncol, nck, cc, nbx, T, nbg, nhk) in zip(asked, got):
        what = (kind, most, nph, width, nbox, R)
        assert 1 <= taps <= width and (kind == 1 or taps == width), what
        assert T <= most and T % 32 == 0 and nbx * ncol * hn <= T, what
        assert cc * (nbx * bc * hn + extra) <= nk * T, what           # every staged 16 bytes has its copy
        assert (nck - 1) * ncol < nph <= nck * ncol and nbg * nbx >= nbox and nhk * hn == hn * R, what
        assert nbx == 1 or nck == 1, what
        for p in range(0, nph, ncol):                                 # each column's taps are staged
            q = np.arange(p, min(nph, p + ncol))
            assert (s[q] >= s[p]).all() and (s[q] - s[p] + taps <= cc).all(), what
