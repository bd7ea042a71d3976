// The pieces of a host-buffer call (HostPieces, hho_internal.h), apart from the
// CUDA calls.
#pragma once

#include <algorithm>
#include <cstdint>
#include <memory>
#include <new>

#include "hho_internal.h"

// Cuts the pieces of an operator: where the cells of each are and which pieces
// their face neighbours lie in.  One pass over the cells and one over the faces,
// which only note which pieces meet: 1.3 ms of the host for the 524,288 cells of
// the 1024 x 512 bilayer, under the first call's 2 ms on the GPU (a build of the
// operator that updated the tables for each cell and face took 5 ms more of 65).
inline void cut_host_pieces(hho_ops* ops) {
    HostPieces& p = ops->host_pieces;
    const int Nf = ops->dev.Nf, warps = (Nf + ops->dev.Ns) / 32;
    const int64_t nc = ops->nc, blocks = (nc + STAGED_CELLS - 1) / STAGED_CELLS;
    p.n = 1;
    int n = 1;
    while (n < HostPieces::MAX && warps / HostPieces::WARPS >= 2 * n) n *= 2;
    if (n == 1 || (int64_t)sizeof(double) * ops->n_canonical < HostPieces::BYTES) return;
    std::unique_ptr<uint8_t[]> warp_piece(new (std::nothrow) uint8_t[warps]), cell_piece(new (std::nothrow) uint8_t[nc]);
    if (!warp_piece || !cell_piece) return;   // one piece
    for (int c = 0; c <= n; ++c) {
        p.blocks[c] = (int)(blocks * c / n);
        p.off[c] = c == n ? ops->n_canonical : ops->canon_off[(int64_t)p.blocks[c] * STAGED_CELLS];
        p.warps[c] = c == n ? warps : (int)((int64_t)warps * c / n) & ~3;   // whole thread blocks
        if (c > 0) std::fill(warp_piece.get() + p.warps[c - 1], warp_piece.get() + p.warps[c], (uint8_t)(c - 1));
    }
    uint32_t holds[HostPieces::MAX] = {}, meets[HostPieces::MAX] = {};   // compute pieces of a host piece; neighbours
    const int32_t *dom = ops->cell_dom.data(), *pos = ops->cell_pos.data();
    for (int h = 0; h < n; ++h) {
        const int64_t c1 = std::min(nc, (int64_t)p.blocks[h + 1] * STAGED_CELLS);
        uint32_t in = 0;
        for (int64_t c = (int64_t)p.blocks[h] * STAGED_CELLS; c < c1; ++c) {
            const uint8_t d = warp_piece[(uint32_t)((dom[c] == 0 ? 0 : Nf) + pos[c]) / 32];
            cell_piece[c] = d;
            in |= 1u << d;
        }
        holds[h] = in;
    }
    const int64_t* fc = ops->face_cells.data();
    const int64_t* end = fc + ops->face_cells.size() / 2 * 2;
    for (; fc < end; fc += 2) {
        if (fc[0] < 0 || fc[1] < 0) continue;
        const int a = cell_piece[fc[0]], b = cell_piece[fc[1]];
        if (a == b) continue;   // nearly all
        meets[a] |= 1u << b;
        meets[b] |= 1u << a;
    }
    for (int d = 0; d < n; ++d) {
        p.own[d] = 0;
        for (int h = 0; h < n; ++h)
            if ((holds[h] >> d) & 1) p.own[d] = h;
        p.order[d] = d;
    }
    for (int d = 0; d < n; ++d) {
        p.need[d] = p.own[d];
        for (int e = 0; e < n; ++e)
            if ((meets[d] >> e) & 1) p.need[d] = std::max(p.need[d], p.own[e]);
    }
    std::stable_sort(p.order, p.order + n, [&](int a, int b) { return p.need[a] < p.need[b]; });
    if (*std::min_element(p.own, p.own + n) == n - 1) return;   // nothing starts before the last arrival
    for (int h = 0; h < n; ++h) {
        p.last[h] = 0;
        for (int i = 0; i < n; ++i)
            if ((holds[h] >> p.order[i]) & 1) p.last[h] = i;
    }
    p.n = n;
}

// The pieces of a call that replays graphs or not (`graph`), on buffers that it
// has `made` or not.  Pieces not cut yet, or new buffers: one.  A copy by the copy
// engine into memory that was allocated just before waits 0.5 to 8 ms, while
// kernels run at full speed on it; the first call of an operator, 1024 x 512, k =
// 2, one FP64 step, took 2.2 to 10 ms in pieces and takes 2.5 to 3.7 in one (later
// calls 1.75 and 2.04).
inline int host_pieces(const hho_ops* ops, int64_t nsteps, bool graph, bool made) {
    return nsteps < 1 || ops->prof_on || graph || made ? 1 : std::max(1, ops->host_pieces.n);
}
