// Verlet neighbour lists for the pair kernel (the list of Sec. 3.1 that is
// rebuilt every few steps rather than every step).
//
// A list holds, per lane of the pair kernel, the slots of the partners within
// rlist = rcut + skin of the particle at build time, found over the same cell
// stencil rows that lane would walk (rows s, s+LPP, ... of its particle). As
// long as no particle of the replica has moved more than skin/2 since the
// build, every pair closer than rcut is in the list. The pair kernel's
// epilogue records the largest displacement of each replica's next positions;
// the next step rebuilds exactly the replicas that crossed skin/2, so a
// replica's rebuild steps -- and its summation order -- do not depend on the
// other replicas of a batch.
//
// Layout: entry k of lane l of warp w at nl[(w * cap + k) * 32 + l], so the
// 32 lanes of a warp read one 128-byte line per entry.
//
// k_list_build counts the entries at commit; on a rebuild step and for a loaded
// state the pair kernel's one- and two-species forms build their own lanes' lists
// (list_lane.cuh). The kernels for more species read lists of another layout
// (list_striped.cuh), one per particle, which k_list_build_striped builds before
// them.
#include <algorithm>

#include "launch.h"
#include "list_lane.cuh"
#include "list_striped.cuh"

namespace tdpd {

// Threads per particle of a striped build, and the particles up to which it has more
// than one (measured, full lists of ten species, event time with 6 us of launch:
// 27k particles 43 us with four threads, 46 with eight, 67 with one; 41k at a density
// of 3: 48, 50, 59; 60k: 78, 80, 72; 286k: 213, 243, 169).
constexpr int STRIPED_SPLIT = 4, STRIPED_SPLIT_MAX = 50000;

__global__ void k_rebuild_decide(const uint32_t *__restrict__ disp, uint32_t *disp_clear, uint32_t *rb,
                                 const RepParams *__restrict__ reps, int n_rep, int force, uint32_t *step_ctr,
                                 uint32_t *builds)
{
    pdl_enter();
    int any = 0;
    for (int r = threadIdx.x; r < n_rep; r += blockDim.x) {
        const bool b = force || __uint_as_float(disp[r]) > reps[r].half_skin2;
        rb[r] = b ? 1u : 0u;
        disp_clear[r] = 0u;
        if (b) builds[r] += 1u;
        any |= b;
    }
    any = __syncthreads_or(any);
    if (threadIdx.x == 0) {
        rb[n_rep] = any ? 1u : 0u;
        *step_ctr += 1u;
    }
}

// Cell and rank of the position each particle of a rebuilding replica will
// have at the next force evaluation (the last pair epilogue wrote it, for every
// slot, into the other buffer: next_pos), for the sort of a rebuild step. A replica
// that keeps its list keeps its slots: its particles are not binned, and its whole
// count goes to its first cell, so that the scan still gives every replica its own
// slot range. With D.disp set (few replicas) the rebuild decision is taken here
// instead of in k_rebuild_decide: every CTA reads the replicas' maxima itself, and
// CTA 0 records the decision as k_rebuild_decide would; otherwise rb holds it.
// Bound by the ranks' round trip to the L2; two particles per thread and turn keep
// two in flight (786k particles: 21.6 us; one per thread, with the positions
// predicted again from three more arrays: 28.7). A step without a rebuild launches
// it too, so the grid is at most what the GPU holds at once.
constexpr int BIN_THREADS = 256, BIN_GRID_MAX = 152 * 8;
__global__ void __launch_bounds__(BIN_THREADS) k_bin_next(const float4 *__restrict__ next_pos,
                                                          const float4 *__restrict__ vel,
                                                          const RepParams *__restrict__ reps, int n_rep, int n,
                                                          int *count, int *tile_sum, int2 *cellrank,
                                                          const uint32_t *any, const uint32_t *__restrict__ rb,
                                                          DecideArgs D)
{
    pdl_enter();
    if (D.disp) {
        int a = 0;
        for (int r = threadIdx.x; r < D.n_rep; r += blockDim.x) {
            const bool rebuild = __uint_as_float(D.disp[r]) > reps[r].half_skin2;
            a |= rebuild;
            if (blockIdx.x == 0) {
                D.rb[r] = rebuild ? 1u : 0u;
                D.disp_clear[r] = 0u;
                if (rebuild) D.builds[r] += 1u;
            }
        }
        a = __syncthreads_or(a);
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            D.rb[D.n_rep] = a ? 1u : 0u;
            *D.step_ctr += 1u;
        }
        if (!a) return;
    } else if (!*any) {
        return;
    }
    const int G = gridDim.x * BIN_THREADS, first = blockIdx.x * BIN_THREADS + threadIdx.x;
    // (a turn's bound is the same for the lanes of a warp)
    for (int k0 = first; k0 - (int)(threadIdx.x & 31) < n; k0 += 2 * G) {
        int c[2], rank[2], r[2];
        float4 p[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = k0 + u * G;
            c[u] = -1;
            if (k < n) {
                r[u] = n_rep > 1 ? wbits(vel[k].w) : 0;
                p[u] = next_pos[k];
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int k = k0 + u * G;
            if (k >= n) continue;
            const RepParams &P = reps[r[u]];
            const bool rebuild = D.disp ? __uint_as_float(D.disp[r[u]]) > P.half_skin2 : rb[r[u]] != 0u;
            if (rebuild) {
                c[u] = cell_of(P, p[u].x, p[u].y, p[u].z);
                rank[u] = atomicAdd(count + c[u], 1);
            } else if (k == P.pbase) {
                atomicAdd(count + P.cell_base, P.n);
                atomicAdd(tile_sum + (P.cell_base >> SCAN_TILE_LOG2), P.n);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            add_tile_count(tile_sum, c[u]);
            if (c[u] >= 0) cellrank[k0 + u * G] = make_int2(c[u], rank[u]);
        }
    }
}

// One thread per pair lane.
template <int LPP, int M, bool HALF>
__global__ void __launch_bounds__(128) k_list_build(ListArgs A)
{
    pdl_enter();
    if (!A.rb[A.n_rep]) return;                       // no replica rebuilds
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = gt / LPP, sub = gt % LPP;
    if (i >= A.n) return;
    const float4 pi = A.pos[i];
    const int rep = wbits(A.vel[i].w);
    if (!A.rb[rep]) return;
    if (A.quar && A.quar[rep]) {                      // quarantined: an empty list
        A.nlc[gt] = 0;
        return;
    }
    build_lane<LPP, M, HALF>(A, gt, i, sub, pi, rep);
}

// The striped lists of the kernels with more than two species, B threads per
// particle (a power of two), in the stencil's row order for every B. One thread
// appends as it walks its rows; of several (small systems, where a thread per
// particle leaves the GPU idle) each takes one of the next B rows, keeps up to
// KEEP of its entries in shared memory until the B counts are known, and walks the
// row a second time only for the entries beyond them (consecutive parts of the rows
// per thread, each walked twice, 27k particles: 52 us against 43 -- the outer rows
// are short and their threads idled).
template <int M, bool HALF, int B>
__global__ void __launch_bounds__(128) k_list_build_striped(ListArgs A)
{
    constexpr int KEEP = 8;
    __shared__ int kept[B > 1 ? KEEP : 1][128];
    pdl_enter();
    if (!A.rb[A.n_rep]) return;                       // no replica rebuilds
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = gt / B, sub = gt % B;
    if (i >= A.n) return;
    const float4 pi = A.pos[i];
    const int rep = wbits(A.vel[i].w);
    if (!A.rb[rep]) return;
    if (A.quar && A.quar[rep]) {                      // quarantined: an empty list
        if (sub == 0) A.nlc[i] = 0;
        return;
    }
    const RepParams &P = A.reps[rep];
    const int m = M > 0 ? M : P.m_stencil, nrow = (2 * m + 1) * (2 * m + 1), first = HALF ? nrow / 2 : 0;
    // striped_row and striped_off by shifts (L is a power of two)
    const int L = A.lpp, kl = __ffs(L) - 1, cap = A.cap;
    int *list = A.nl + ((size_t)(i >> (5 - kl)) * (cap >> kl) * 32 + ((i & ((32 >> kl) - 1)) << kl));
    auto off = [&](int e) { return ((e >> kl) << 5) + (e & (L - 1)); };
    int total = 0;
    if constexpr (B > 1) {
        int *mine = &kept[0][threadIdx.x];
        const unsigned group = ((1u << B) - 1u) << (threadIdx.x & 31 & ~(B - 1));   // the particle's lanes
        for (int r0 = first; r0 < nrow; r0 += B) {
            const int row = r0 + sub, end = min(row + 1, nrow);
            int c = 0;
            visit_rows<M, HALF, false>(P, A.pos, A.cell_start, i, row, end, 1, pi, [&](const bool (&ok)[4], int j0) {
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (ok[u]) {
                        if (c < KEEP) mine[c * 128] = j0 + u;
                        ++c;
                    }
            });
            int x = c;
#pragma unroll
            for (int o = 1; o < B; o <<= 1) {
                const int v = __shfl_up_sync(group, x, o, B);
                if (sub >= o) x += v;
            }
            const int e = total + x - c, room = cap - e;          // the row's first entry, entries left from it
            for (int k = 0; k < min(min(c, KEEP), room); ++k) list[off(e + k)] = mine[k * 128];
            if (c > KEEP && room > KEEP) {
                int k = 0;
                visit_rows<M, HALF, false>(P, A.pos, A.cell_start, i, row, end, 1, pi,
                                           [&](const bool (&ok)[4], int j0) {
#pragma unroll
                    for (int u = 0; u < 4; ++u)
                        if (ok[u]) {
                            if (k >= KEEP && k < room) list[off(e + k)] = j0 + u;
                            ++k;
                        }
                });
            }
            total += __shfl_sync(group, x, B - 1, B);
        }
    } else {
        int at = 0;
        visit_rows<M, HALF, true>(P, A.pos, A.cell_start, i, 0, 0, 1, pi, [&](const bool (&ok)[4], int j0) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (ok[u]) {
                    if (total < cap) list[at] = j0 + u;
                    ++total;
                    at += (total & (L - 1)) ? 1 : 33 - L;
                }
        });
    }
    if (sub == 0) {
        A.nlc[i] = cap > 0 ? min(total, cap) : total;
        if (cap > 0 && total > cap) atomicOr(A.err + rep, 2u);
        A.xb[i] = pi;
    }
}

void launch_rebuild_decide(const uint32_t *disp, uint32_t *disp_clear, uint32_t *rb, const RepParams *reps,
                           int n_rep, int force, uint32_t *step_ctr, uint32_t *builds, cudaStream_t st)
{
    launch_pdl(k_rebuild_decide, 1, 256, st, disp, disp_clear, rb, reps, n_rep, force, step_ctr, builds);
}

void launch_bin_next(const float4 *next_pos, const float4 *vel, const RepParams *reps, int n_rep, int n, int *count,
                     int *tile_sum, int2 *cellrank, const uint32_t *rb, const uint32_t *any, cudaStream_t st,
                     const DecideArgs &d)
{
    if (n <= 0 && !d.disp) return;
    int g = std::max(1, (n + 2 * BIN_THREADS - 1) / (2 * BIN_THREADS));
    if (d.disp) g = std::min(g, BIN_GRID_MAX);       // (of many replicas one nearly always rebuilds)
    launch_pdl(k_bin_next, g, BIN_THREADS, st, next_pos, vel, reps, n_rep, n, count, tile_sum, cellrank, any, rb, d);
}

template <bool HALF>
static void launch_list_build_h(const ListArgs &a, int g, cudaStream_t st)
{
    if (a.m2) {
        switch (a.lpp) {
        case 1: launch_pdl(k_list_build<1, 2, HALF>, g, 128, st, a); break;
        case 2: launch_pdl(k_list_build<2, 2, HALF>, g, 128, st, a); break;
        case 4: launch_pdl(k_list_build<4, 2, HALF>, g, 128, st, a); break;
        case 8: launch_pdl(k_list_build<8, 2, HALF>, g, 128, st, a); break;
        case 16: launch_pdl(k_list_build<16, 2, HALF>, g, 128, st, a); break;
        default: launch_pdl(k_list_build<32, 2, HALF>, g, 128, st, a); break;
        }
        return;
    }
    switch (a.lpp) {
    case 1: launch_pdl(k_list_build<1, 0, HALF>, g, 128, st, a); break;
    case 2: launch_pdl(k_list_build<2, 0, HALF>, g, 128, st, a); break;
    case 4: launch_pdl(k_list_build<4, 0, HALF>, g, 128, st, a); break;
    case 8: launch_pdl(k_list_build<8, 0, HALF>, g, 128, st, a); break;
    case 16: launch_pdl(k_list_build<16, 0, HALF>, g, 128, st, a); break;
    default: launch_pdl(k_list_build<32, 0, HALF>, g, 128, st, a); break;
    }
}

template <int M, bool HALF>
static void launch_striped(const ListArgs &a, cudaStream_t st)
{
    // several threads per particle up to the particles that fill the GPU alone
    if (a.n <= STRIPED_SPLIT_MAX)
        launch_pdl(k_list_build_striped<M, HALF, STRIPED_SPLIT>, (int)(((long)STRIPED_SPLIT * a.n + 127) / 128), 128,
                   st, a);
    else
        launch_pdl(k_list_build_striped<M, HALF, 1>, (a.n + 127) / 128, 128, st, a);
}

void launch_list_build(const ListArgs &a, cudaStream_t st)
{
    if (a.n <= 0) return;
    if (a.striped) {
        if (a.m2) {
            if (a.half) launch_striped<2, true>(a, st);
            else launch_striped<2, false>(a, st);
        } else {
            if (a.half) launch_striped<0, true>(a, st);
            else launch_striped<0, false>(a, st);
        }
        return;
    }
    const int g = (int)(((long)a.n * a.lpp + 127) / 128);
    if (a.half) launch_list_build_h<true>(a, g, st);
    else launch_list_build_h<false>(a, g, st);
}

}  // namespace tdpd
