// The per-lane Verlet list build (the list of Sec. 3.1), shared by the
// list-build kernel and the pair kernel, which on a rebuild step builds the
// lists of its own lanes before walking them.
#pragma once

#include "launch.h"

namespace tdpd {

// The candidates of particle i over the rows r0, r0 + dr, ... < r1 of its cell
// stencil, in row order and slot order within a row: hit(ok, j0) for four
// candidate slots j0 .. j0 + 3 at a time, ok[u] set where slot j0 + u holds a
// partner within rlist. M: the stencil half-width when it is known at compile
// time (2, the default cell size), else 0 (read per replica).
//
// HALF: only the upper half of the stencil (rows from (2m+1)^2 / 2 on), so that
// every unordered pair is listed once. A cell's offset (dx, dy, dz) from particle
// i's cell has one representative in [-m, m]^3 (a periodic axis holds at least
// 2m + 1 cells), and the pair belongs to the side from which that offset is
// upper: rows with dz > 0, or dz = 0 and dy > 0 (the rows after the home row),
// and in the home row the cells with dx > 0 and, in i's own cell, the slots after
// i. Cells of a row are consecutive slots, so the home row's upper part is the
// slot range after i up to the row's end, plus the segment that wraps around to
// the right.
//
// ALL: every row of the (half) stencil (r0, r1, dr are not used): the rows of one
// z share their z part, the row's bound comes from a reciprocal square root (its
// error is far inside the margin eps), and the part that wraps around x is a
// second turn instead of a second copy of the loop. A build of 786k half lists in
// the pair kernel: 151 warp instructions per particle and 142 us (row by row: 177
// and 158); bound by issue (64 % of the slots) at 24 of 32 threads active, since
// rows differ in length.
template <int M, bool HALF, bool ALL, class Hit>
__device__ __forceinline__ void visit_rows(const RepParams &P, const float4 *pos, const int *cell_start, int i,
                                           int r0, int r1, int dr, float4 pi, Hit &&hit)
{
    const int m = M > 0 ? M : P.m_stencil, width = 2 * m + 1;
    const int cx = cell_coord(pi.x, P.cell_scale[0], P.nc[0]);
    const int cy = cell_coord(pi.y, P.cell_scale[1], P.nc[1]);
    const int cz = cell_coord(pi.z, P.cell_scale[2], P.nc[2]);
    const float oy = pi.y - (float)cy * P.h[1], oz = pi.z - (float)cz * P.h[2];
    const float eps = 1e-4f * fmaxf(P.h[0], fmaxf(P.h[1], P.h[2]));
    const float rl2 = P.rlist2;
    float4 pj[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) pj[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    // the candidates of slots [jb, je), four per trip with their loads in flight
    // together (a candidate past the end keeps stale y and z and gets an x far
    // away); the half shell's ranges never hold particle i itself
    auto walk = [&](int jb, int je, float px, float py, float pz) {
        for (int j0 = jb; j0 < je; j0 += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (j0 + u < je) pj[u] = pos[j0 + u];
                else pj[u].x = 1e30f;
            }
            bool ok[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float dx = px - pj[u].x, dy = py - pj[u].y, dz = pz - pj[u].z;
                ok[u] = dx * dx + dy * dy + dz * dz < rl2 && (HALF || j0 + u != i);
            }
            hit(ok, j0);
        }
    };
    if constexpr (ALL) {
        const float rtrim2 = rl2 * 1.0002f;
        const int nx = P.nc[0], ny = P.nc[1], nz = P.nc[2];
        const float hy = P.h[1], hz = P.h[2], sx = P.cell_scale[0], xs = pi.x * sx;
#pragma unroll 1
        for (int dz = HALF ? 0 : -m; dz <= m; ++dz) {
            const float az = dz == 0 ? 0.f : (dz > 0 ? (float)dz * hz - oz : oz - (float)(dz + 1) * hz);
            const float bz = fmaxf(az - eps, 0.f);
            const float remz = rtrim2 - bz * bz;
            int z = cz + dz;
            float pz = pi.z;
            bool okz = remz > 0.f;
            if (z < 0) { z += nz; pz += P.L[2]; okz = okz && P.periodic[2]; }
            else if (z >= nz) { z -= nz; pz -= P.L[2]; okz = okz && P.periodic[2]; }
            if (!okz) continue;
            const int *csz = cell_start + P.cell_base + z * ny * nx;
#pragma unroll 1
            for (int dy = HALF && dz == 0 ? 0 : -m; dy <= m; ++dy) {
                const float ay = dy == 0 ? 0.f : (dy > 0 ? (float)dy * hy - oy : oy - (float)(dy + 1) * hy);
                const float by = fmaxf(ay - eps, 0.f);
                const float rem = remz - by * by;
                if (!(rem > 0.f)) continue;
                int y = cy + dy;
                float py = pi.y;
                if (y < 0) { y += ny; py += P.L[1]; }
                else if (y >= ny) { y -= ny; py -= P.L[1]; }
                const float rx = (rem * rsqrtf(rem) + eps) * sx;
                const int x0 = max(cx - m, __float2int_rd(xs - rx)), x1 = min(cx + m, __float2int_rd(xs + rx));
                const int *cs = csz + y * nx;
                // the row's range, then where it wraps the part beyond the box;
                // half shell: the home row from the slot after i, and only the
                // part that wraps around to the right (dx > 0)
                const bool home = HALF && dy == 0 && dz == 0;
                int jb = home ? i + 1 : cs[max(x0, 0)], je = cs[min(x1, nx - 1) + 1];
                float px = pi.x;
                bool more = x1 >= nx || (x0 < 0 && !home);
#pragma unroll 1
                for (;;) {
                    walk(jb, je, px, py, pz);
                    if (!more) break;
                    more = false;
                    const bool right = x1 >= nx;
                    jb = cs[right ? 0 : nx + x0];
                    je = cs[right ? x1 - nx + 1 : nx];
                    px = pi.x + (right ? -P.L[0] : P.L[0]);
                }
            }
        }
    } else {
        for (int row = r0; row < r1; row += dr) {
            const int dy = row % width - m, dz = row / width - m;
            RowSeg g = {{0, 0}, {0, 0}, 0.f, 0.f, 0.f};
            if (!stencil_row_d(P, cell_start, pi, cx, cy, cz, dy, dz, m, oy, oz, eps, rl2 * 1.0002f, g)) continue;
            if (HALF && dy == 0 && dz == 0) {
                // the home row from the slot after i; a segment that wraps
                // around to the left (x shift +L) holds only cells with dx < 0
                g.jb[0] = i + 1;
                if (g.sx1 > 0.f) g.je[1] = g.jb[1];
            }
            const float py = pi.y + g.sy, pz = pi.z + g.sz;
#pragma unroll
            for (int sg = 0; sg < 2; ++sg) {
                const float px = pi.x + (sg ? g.sx1 : 0.f);
                walk(g.jb[sg], g.je[sg], px, py, pz);
            }
        }
    }
}

// The list of one pair lane (particle i, lane sub of LPP, thread gt of the pair
// kernel's layout), its count in nlc and, for lane 0, the build position xb[i].
// Used by k_list_build and, on rebuild steps, by the pair kernel for its own
// lanes.
template <int LPP, int M, bool HALF = false>
__device__ __forceinline__ void build_lane(const ListArgs &A, int gt, int i, int sub, float4 pi, int rep)
{
    const RepParams &P = A.reps[rep];
    const int m = M > 0 ? M : P.m_stencil, nrow = (2 * m + 1) * (2 * m + 1);
    int *out = A.nl + (size_t)(gt >> 5) * A.cap * 32 + (gt & 31);   // next entry
    const int cap = A.cap;
    int c = 0;
    // appended in order (the capacity test once per four while they fit)
    visit_rows<M, HALF, LPP == 1>(P, A.pos, A.cell_start, i, (HALF ? nrow / 2 : 0) + sub, nrow, LPP, pi,
                        [&](const bool (&ok)[4], int j0) {
        if (c + 4 <= cap) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (ok[u]) {
                    *out = j0 + u;
                    out += 32;
                    ++c;
                }
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (ok[u]) {
                    if (c < cap) {
                        *out = j0 + u;
                        out += 32;
                    }
                    ++c;
                }
        }
    });
    A.nlc[gt] = A.cap > 0 ? min(c, A.cap) : c;
    if (A.cap > 0 && c > A.cap) atomicOr(A.err + rep, 2u);
    if (sub == 0) A.xb[i] = pi;
}

}  // namespace tdpd
