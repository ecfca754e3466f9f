// The list-mode pair kernel for more than two species: pairwise tDPD force (Eq. 3)
// and the fluxes of every species (Eq. 6, and Eq. 7), full or half shell, as k_pair
// (k_pair_impl.cuh), with another division of the work.
//
// A partner here is a row of concentrations beside its position: with one
// particle per lane (k_pair's layout) 32 lanes gather 32 rows that share no
// sector. So L lanes walk one particle's list together, L consecutive entries a
// trip: they are mostly consecutive slots, and the rows and the reductions of a
// trip fall into few sectors (measured: 16-byte gathers run at 225 G/s from
// scattered slots and at 640 G/s from runs of eight, 64-bit reductions at 206 and
// 509 G/s). A warp owns 32 / L x K consecutive particles and takes them 32 / L at
// a time, K rounds, so that its set-up is paid once. Lane s of a particle sums the
// entries s, s + L, ... in list order and a butterfly adds the lanes: the sum
// depends on the list and on L alone, not on K or on the particles that share the
// warp. (One and two species keep k_pair: there the rows are short, and the
// additional instructions per entry cost more than the gathers; with the random flux
// too, so that a replica's sums have one order whether or not another replica of its
// batch has the flux.)
//
// Ten species, 286k particles, full shell: 236 us (k_pair's layout 344). Ten
// species with the random flux, 41k particles, half shell: 108 us and 17 for the
// finishing pass (318 together). Bound by the latency of the rows, 41 % of the
// issue slots and 69 % of the L1 throughput: four CTAs per SM (128 registers) took
// 260 us, six (80, a few spilled) 303. The rows are read while the force pairs
// are queued; reading them a trip ahead needs ten more registers.
#pragma once

#include "k_pair_impl.cuh"
#include "list_striped.cuh"

namespace tdpd {

namespace {

template <int NS>
struct MultiSmem {
    WarpSmem w;                      // li, acc: by the particle's index within the warp
    float4 pos[32];
    int cnt[32];                     // list lengths
    float c[32 * NS], qs[32 * NS];   // predicted concentrations and own flux sums
};

// A replica with one type and no partner shares sums its fluxes without kappa and
// scales them at the end; its own parameters decide, so that it takes the same
// formula alone and beside other replicas.
template <bool HALF, bool QR>
__device__ __forceinline__ bool scaled_flux(const RepParams &P)
{
    return !HALF && P.ntypes == 1 && !(QR && P.qr_coef > 0.0f);
}

constexpr float ROUND_MAGIC = 12582912.0f;    // 1.5 x 2^23: x + M - M rounds x to an integer

}  // namespace

// NS: species; RT: up to NS of them, A.ns at run time. L: lanes per particle.
// QR: the random flux of Eq. 7.
template <int NS, bool RT, int L, bool HALF, bool QR>
__global__ void __launch_bounds__(128, NS <= 4 ? 6 : NS <= 10 ? 5 : 3) k_pair_multi(PairArgs A)
{
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int P1 = 32 / L;                     // particles of a round
    pdl_enter();
    __shared__ MultiSmem<NS> smem[4];
    const int ns = RT ? A.ns : NS;
    const int lane = threadIdx.x & 31, sub = lane % L, grp = lane / L;
    MultiSmem<NS> &M = smem[threadIdx.x >> 5];
    WarpSmem &W = M.w;
    const int K = 1 << A.klog, PW = P1 << A.klog;
    const int base = (blockIdx.x * 4 + (threadIdx.x >> 5)) * PW;
    if (base >= A.n) return;                       // (no barrier of the whole CTA follows)
    const float4 *__restrict__ pos = A.b.pos;
    const float4 *__restrict__ vt = A.b.vt;
    const float *__restrict__ Ct = A.b.Ct;
    const uint32_t step_ctr = *A.step_ctr;

    // lane p holds the warp's particle p before and after the walk
    const int i = base + lane;
    const bool valid = lane < PW && i < A.n;
    bool live;
    {
        const int ic = valid ? i : base;
        const float4 pi = pos[ic];
        const int rep = wbits(A.b.vel[ic].w);
        // a quarantined replica is neither evaluated nor moved
        live = valid && !(A.quar && A.quar[rep] != 0u);
        M.pos[lane] = pi;
        W.li[lane].vt = vt[ic];
        W.li[lane].wi = (uint32_t)wbits(pi.w);
        W.li[lane].rep = rep;
        W.acc[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        M.cnt[lane] = live ? A.nlc[i] : 0;
        // (the rows of the warp's particles are one contiguous range)
        for (int e = lane; e < min(PW, A.n - base) * ns; e += 32) {
            const int p = e / ns;
            M.c[p * NS + (e - p * ns)] = Ct[(size_t)base * ns + e];
        }
    }
    __syncwarp();

    float q[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) q[s] = 0.0f;
    int qhead = 0, qcount = 0;
    const int capb = A.cap / L;
    const int *ptr = A.nl + striped_row(base + grp, L, capb) + sub;
    int n = M.cnt[grp];
    int j0 = sub < n ? ptr[0] : -1, j1 = L + sub < n ? ptr[32] : -1;
    for (int k = 0; k < K; ++k) {
        // round k: lane group g walks the warp's particle k P1 + g
        const int cur = k * P1 + grp;
        float4 p0 = make_float4(0.f, 0.f, 0.f, 0.f), p1 = p0;
        if (j0 >= 0) p0 = pos[j0];
        const int nmax = __reduce_max_sync(FULL, n);
        const float4 xi = M.pos[cur];
        float ci[NS];
#pragma unroll
        for (int s = 0; s < NS; ++s) ci[s] = M.c[cur * NS + s];
        const int rep = W.li[cur].rep;
        const RepParams &P = A.reps[rep];
        const float Lx = P.L[0], Ly = P.L[1], Lz = P.L[2], iLx = P.inv_L[0], iLy = P.inv_L[1], iLz = P.inv_L[2];
        const float rc2 = P.rc2, rcc2 = P.rcc2, inv_rcc = P.inv_rcc, s_c = P.s_c;
        const bool sc2 = P.sc_is2, random = QR && P.qr_coef > 0.0f, scaled = scaled_flux<HALF, QR>(P);
        const float *kap_row = P.kappa + (int)((uint32_t)wbits(xi.w) >> 24) * P.ntypes * ns;
        for (int e = 0; e < nmax; e += L) {
            // the next trip's positions and the indices of the one after are in
            // flight during this trip's arithmetic
            if (j1 >= 0) p1 = pos[j1];
            const int j2 = e + 2 * L + sub < n ? ptr[64] : -1;
            ptr += 32;
            float dx = xi.x - p0.x, dy = xi.y - p0.y, dz = xi.z - p0.z;
            // (rounding by adding 1.5 x 2^23 instead of the conversion unit's
            // rint: the same integer but for ties, which are half a box away)
            dx = __fmaf_rn(-Lx, __fmaf_rn(dx, iLx, ROUND_MAGIC) - ROUND_MAGIC, dx);
            dy = __fmaf_rn(-Ly, __fmaf_rn(dy, iLy, ROUND_MAGIC) - ROUND_MAGIC, dy);
            dz = __fmaf_rn(-Lz, __fmaf_rn(dz, iLz, ROUND_MAGIC) - ROUND_MAGIC, dz);
            const uint32_t wj = (uint32_t)wbits(p0.w);
            const float r2 = dx * dx + dy * dy + dz * dz;
            const bool near = j0 >= 0 && r2 > 0.0f;
            const bool inc = near && r2 < rcc2;
            // the partner's row, in flight while the force pairs are queued
            float cj[NS];
            if (inc) {
                const float *row = Ct + (size_t)j0 * ns;
                if constexpr (!RT && NS % 2 == 0) {
#pragma unroll
                    for (int s = 0; s < NS; s += 2) {
                        const float2 v = *reinterpret_cast<const float2 *>(row + s);
                        cj[s] = v.x;
                        cj[s + 1] = v.y;
                    }
                } else {
#pragma unroll
                    for (int s = 0; s < NS; ++s) cj[s] = s < ns ? row[s] : 0.0f;
                }
            }
            const bool push = near && r2 < rc2;
            const unsigned bal = __ballot_sync(FULL, push);
            if (push) {
                const int slot = (qhead + qcount + __popc(bal & ((1u << lane) - 1u))) & (QCAP - 1);
                int4 *qe = reinterpret_cast<int4 *>(&W.q[slot]);
                qe[0] = make_int4(j0, (int)wj, cur, 0);
                qe[1] = make_int4(__float_as_int(dx), __float_as_int(dy), __float_as_int(dz), __float_as_int(r2));
            }
            qcount += __popc(bal);
            if (qcount >= 32) {
                __syncwarp();
                drain<HALF, false>(W, qhead, 32, A.reps, vt, step_ctr, lane, A.accF, A.err);
                qhead = (qhead + 32) & (QCAP - 1);
                qcount -= 32;
            }
            if (inc) {
                const float r = r2 * rsqrtf(r2);
                const float w = 1.0f - r * inv_rcc;
                const float wdc = sc2 ? w * w : __powf(w, s_c);
                if (scaled) {
#pragma unroll
                    for (int s = 0; s < NS; ++s) q[s] = __fmaf_rn(-wdc, ci[s] - cj[s], q[s]);
                } else {
                    const float *kap = kap_row + (int)(wj >> 24) * ns;
                    // random flux (Eq. 7): eps w_RC zeta / sqrt(dt), eps^2 =
                    // m_s^2 kappa rho (C_i + C_j), w_RC = w_DC^(1/2) (Eq. 8);
                    // one pair normal per species (the (cos, sin) pair of
                    // stream 6 + s/2), signed by the id order so that
                    // zeta_ji = -zeta_ij
                    const uint32_t idi = (uint32_t)wbits(xi.w) & ID_MASK, idj = wj & ID_MASK;
                    float amp = 0.0f;
                    if (random) amp = (idi < idj ? 1.0f : -1.0f) * P.qr_coef * sqrtf(wdc) * P.inv_sqrt_dt;
                    float2 z = make_float2(0.f, 0.f);
#pragma unroll
                    for (int s = 0; s < NS; ++s) {
                        if (RT && s >= ns) break;
                        const float ks = __ldg(kap + s);
                        // (rounded explicitly: the same bits in every form)
                        const float kw = __fmul_rn(ks, wdc), dc = __fsub_rn(ci[s], cj[s]);
                        float f;
                        if (random) {
                            if ((s & 1) == 0)
                                z = normal2(pair_bits(idi, idj, P.seed_lo, P.seed_hi, step_ctr + P.step0, 6u + (uint32_t)(s >> 1)));
                            const float fr = amp * sqrtf(fmaxf(ks * (ci[s] + cj[s]), 0.0f)) * ((s & 1) ? z.y : z.x);
                            f = __fmaf_rn(-kw, dc, fr);
                            q[s] = __fadd_rn(q[s], f);
                        } else {
                            f = -__fmul_rn(kw, dc);
                            q[s] = __fmaf_rn(-kw, dc, q[s]);
                        }
                        if (HALF) acc_add(A.accQ + (size_t)j0 * ns + s, -f, ACC_Q_SCALE, ACC_Q_LIMIT, A.err + rep);
                    }
                }
            }
            j0 = j1; p0 = p1;
            j1 = j2;
        }
        // the next round's first indices, and this round's own fluxes
        if (k + 1 < K) {
            ptr = A.nl + striped_row(base + cur + P1, L, capb) + sub;
            n = M.cnt[cur + P1];
            j0 = sub < n ? ptr[0] : -1;
            j1 = L + sub < n ? ptr[32] : -1;
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            if (RT && s >= ns) break;
            float t = q[s];
#pragma unroll
            for (int o = 1; o < L; o <<= 1) t += __shfl_xor_sync(FULL, t, o);
            if (sub == 0) M.qs[cur * NS + s] = t;
            q[s] = 0.0f;
        }
    }
    __syncwarp();
    if (qcount > 0) drain<HALF, false>(W, qhead, qcount, A.reps, vt, step_ctr, lane, A.accF, A.err);
    __syncwarp();

    const float4 fa = W.acc[lane];
    const int rep = W.li[lane].rep;
    float disp2 = 0.0f;
    const int count = min(PW, A.n - base);
    const unsigned mask = __ballot_sync(FULL, live);
    if constexpr (HALF) {
        // the own sums; k_pair_finish adds the partners' shares and applies the
        // epilogue
        if (live) A.fown[i] = make_float4(fa.x, fa.y, fa.z, 0.0f);
        for (int e = lane; e < count * ns; e += 32) {
            const int p = e / ns;
            if ((mask >> p) & 1u) A.qown[(size_t)base * ns + e] = M.qs[p * NS + (e - p * ns)];
        }
    } else {
        if (live) {
            const float4 pi = M.pos[lane];
            int cell = -1;
            epilogue<0, true, false>(A, A.reps[rep], i, pi, W.li[lane].vt, A.b.vel[i], (uint32_t)wbits(pi.w), rep, fa.x,
                                     fa.y, fa.z, nullptr, cell, disp2);
        }
        species_rows<RT ? 0 : NS>(A, base, count, mask, lane,
                                  [&](int p) { return make_int2(W.li[p].rep, (int)W.li[p].wi); },
                                  [&](int p, int s, size_t) {
                                      const float f = M.qs[p * NS + s];
                                      const RepParams &R = A.reps[W.li[p].rep];
                                      return scaled_flux<HALF, QR>(R) ? __fmul_rn(f, __ldg(R.kappa + s)) : f;
                                  },
                                  [&](int p, int s) { return M.c[p * NS + s]; });
        record_displacement(A.disp_next, rep, disp2, live, lane);
    }
}

template <int NS, bool RT, bool HALF, bool QR>
static void launch_multi_lanes(const PairArgs &a, cudaStream_t st)
{
    const int pw = (32 / a.lpp) << a.klog;
    const int g = (int)(((long)a.n + 4 * pw - 1) / (4 * pw));
    switch (a.lpp) {
    case 1: launch_pdl(k_pair_multi<NS, RT, 1, HALF, QR>, g, 128, st, a); break;
    case 2: launch_pdl(k_pair_multi<NS, RT, 2, HALF, QR>, g, 128, st, a); break;
    case 4: launch_pdl(k_pair_multi<NS, RT, 4, HALF, QR>, g, 128, st, a); break;
    case 8: launch_pdl(k_pair_multi<NS, RT, 8, HALF, QR>, g, 128, st, a); break;
    case 16: launch_pdl(k_pair_multi<NS, RT, 16, HALF, QR>, g, 128, st, a); break;
    default: launch_pdl(k_pair_multi<NS, RT, 32, HALF, QR>, g, 128, st, a); break;
    }
}

template <int NS, bool RT, bool QR>
static void launch_multi_ns(const PairArgs &a, cudaStream_t st)
{
    if (a.half) launch_multi_lanes<NS, RT, true, QR>(a, st);
    else launch_multi_lanes<NS, RT, false, QR>(a, st);
}

}  // namespace tdpd
