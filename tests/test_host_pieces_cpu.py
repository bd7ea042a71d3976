"""The pieces of a host-buffer call (host_pieces.h), cut on the host: what each
compute piece waits for and when each host piece is complete, against the
definitions cell by cell and face by face, for orders that follow the cell order
and orders that do not."""
import os
import subprocess

import pytest

from tests.libutil import ROOT

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <random>

#include "host_pieces.h"

int main(int argc, char** argv) {
    const int nx = atoi(argv[1]), ny = atoi(argv[2]), k = atoi(argv[3]);
    const char order = argv[4][0];   // o: as the cells; i: two classes interleaved; r: random; x: domains too
    const int n = (k + 1) * (k + 2) / 2;
    hho_ops o;
    o.nc = (int64_t)nx * ny;
    std::vector<int64_t> pos(o.nc);
    std::mt19937 rng(1);
    o.cell_dom.resize(o.nc), o.cell_pos.resize(o.nc);
    int64_t count[2] = {};
    for (int64_t c = 0; c < o.nc; ++c) {   // upper half fluid
        o.cell_dom[c] = order == 'x' ? c & 1 : c < o.nc / 2;
        o.canon_off.push_back(o.n_canonical);
        o.n_canonical += (o.cell_dom[c] ? 5 : 3) * n;
        count[o.cell_dom[c]]++;
    }
    for (int d = 0; d < 2; ++d) {
        std::vector<int64_t> cells;
        for (int64_t c = 0; c < o.nc; ++c)
            if (o.cell_dom[c] == d) cells.push_back(c);
        if (order == 'i') std::stable_partition(cells.begin(), cells.end(), [](int64_t c) { return c & 1; });
        if (order == 'r' || order == 'x') std::shuffle(cells.begin(), cells.end(), rng);
        for (size_t i = 0; i < cells.size(); ++i) o.cell_pos[cells[i]] = (int32_t)i;
    }
    o.dev.Nf = (int)((count[0] + 31) / 32 * 32);
    o.dev.Ns = (int)((count[1] + 31) / 32 * 32);
    for (int y = 0; y < ny; ++y)
        for (int x = 0; x <= nx; ++x)
            for (int v = 0; v < 2; ++v) {   // faces across x, then across y
                const int64_t a = v == 0 ? (x > 0 ? (int64_t)y * nx + x - 1 : -1) : (x < nx && y > 0 ? (int64_t)(y - 1) * nx + x : -1);
                const int64_t b = x < nx ? (int64_t)y * nx + x : -1;
                o.face_cells.push_back(a), o.face_cells.push_back(b);
            }
    if (host_pieces(&o, 1, false, false) != 1) return 1;   // not cut yet
    cut_host_pieces(&o);
    const HostPieces& p = o.host_pieces;
    printf("%d\n", p.n);
    if (host_pieces(&o, 1, false, true) != 1 || host_pieces(&o, 0, false, false) != 1 ||
        host_pieces(&o, 1, true, false) != 1 || host_pieces(&o, 1, false, false) != p.n)
        return 2;
    o.prof_on = true;
    if (host_pieces(&o, 1, false, false) != 1) return 2;
    if (p.n == 1) return 0;
    const int warps = (o.dev.Nf + o.dev.Ns) / 32;
    if (p.blocks[0] || p.warps[0] || p.off[0] || p.warps[p.n] != warps || p.off[p.n] != o.n_canonical ||
        p.blocks[p.n] != (o.nc + STAGED_CELLS - 1) / STAGED_CELLS)
        return 3;
    std::vector<int> own(p.n, 0), need, at(p.n), last(p.n, 0);
    auto host = [&](int64_t c) { int h = 0; while (c / STAGED_CELLS >= p.blocks[h + 1]) ++h; return h; };
    auto piece = [&](int64_t c) {
        const int w = ((o.cell_dom[c] ? o.dev.Nf : 0) + o.cell_pos[c]) / 32;
        int d = 0;
        while (w >= p.warps[d + 1]) ++d;
        return d;
    };
    for (int64_t c = 0; c < o.nc; ++c) own[piece(c)] = std::max(own[piece(c)], host(c));
    need = own;
    for (size_t F = 0; F < o.face_cells.size(); F += 2)
        for (int s = 0; s < 2; ++s)
            if (o.face_cells[F] >= 0 && o.face_cells[F + 1] >= 0) {
                int& v = need[piece(o.face_cells[F + s])];
                v = std::max(v, own[piece(o.face_cells[F + 1 - s])]);
            }
    for (int i = 0; i < p.n; ++i) {
        at[p.order[i]] = i;
        if (i && need[p.order[i - 1]] > need[p.order[i]]) return 4;
    }
    for (int64_t c = 0; c < o.nc; ++c) last[host(c)] = std::max(last[host(c)], at[piece(c)]);
    for (int d = 0; d < p.n; ++d)
        if (p.own[d] != own[d] || p.need[d] != need[d] || p.last[d] != last[d]) return 5;
    for (int c = 1; c < p.n; ++c)
        if (p.warps[c] % 4 || p.off[c] != o.canon_off[(int64_t)p.blocks[c] * STAGED_CELLS]) return 6;
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("host_pieces")
    (d / "main.cpp").write_text(PROGRAM)
    exe = str(d / "main")
    csrc = os.path.join(ROOT, "paper_2505_15771_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I" + csrc, "-I" + os.path.join(ROOT, "include"), str(d / "main.cpp"),
                    "-o", exe], check=True)
    return exe


# the last ones: cells of both domains all over the canonical order, where nothing can start early
@pytest.mark.parametrize("nx,ny,k,order,pieces", [
    (1024, 512, 2, "o", 8), (1024, 512, 1, "o", 8), (723, 363, 2, "o", 4), (512, 272, 3, "o", 2),
    (512, 272, 2, "o", 1), (64, 64, 2, "o", 1), (1000, 700, 2, "i", 8), (1023, 513, 3, "r", 8), (723, 363, 3, "r", 4),
    (1023, 513, 2, "x", 1), (723, 363, 3, "x", 1)])
def test_pieces_follow_their_definition(program, nx, ny, k, order, pieces):
    r = subprocess.run([program, str(nx), str(ny), str(k), order], capture_output=True, text=True)
    assert r.returncode == 0 and int(r.stdout) == pieces


def test_operator_build_cuts_no_pieces():
    """The tables cost milliseconds on a large mesh and only pinned host-buffer calls read them."""
    src = open(os.path.join(ROOT, "paper_2505_15771_gb300", "csrc", "operators.cpp")).read()
    assert "cut_host_pieces" not in src
