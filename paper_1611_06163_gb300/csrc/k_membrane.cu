// Membrane forces of the triangulated RBC model (Sec. 2.2, Eq. 10-16), one CTA or a
// cluster of CTAs per membrane (k_membrane):
//   - K-Gather of Sec. 3.3: the triangle areas and signed tetrahedron volumes and
//     the vertex centroid (the next step's reference point), binary32 terms in
//     compensated float-float sums, converted to binary64 once, and the
//     constraint coefficients they give;
//   - every edge once: the bond (WLC + POW, viscous and random parts) and the
//     dihedral of its two triangles, their forces on the edge's four vertices
//     left in shared memory;
//   - K-Apply: every vertex sums, over its one-ring fan, the forces of its bonds
//     and dihedrals and the area and volume gradients of its triangles. No
//     atomics, a fixed order. A lagged membrane uses the previous step's
//     coefficients, the others wait for this step's.
//
// The vertices' predicted positions and v~ come from arrays in load order (written
// by the previous step's pair kernel, or by the packing of a loaded state) and the
// force goes out in load order, so the kernel does not depend on the cell sort and
// runs beside it.
//
// Coordinates are taken relative to a per-membrane reference point with the
// minimum image, so a membrane may straddle the periodic boundary as long as
// it spans less than half a box. The vertex centroid is the next step's reference
// point; a loaded state's comes from k_mem_ref.
#include <cooperative_groups.h>

#include "launch.h"

namespace tdpd {

__device__ __forceinline__ float3 f3(float4 a) { return make_float3(a.x, a.y, a.z); }
__device__ __forceinline__ float3 sub(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 add(float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 scl(float s, float3 a) { return make_float3(s * a.x, s * a.y, s * a.z); }
__device__ __forceinline__ float dot(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross(float3 a, float3 b)
{
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}

__device__ __forceinline__ float3 rel_pos(const RepParams &P, float4 x, float4 ref)
{
    return make_float3(min_image(x.x - ref.x, P.L[0], P.periodic[0]),
                       min_image(x.y - ref.y, P.L[1], P.periodic[1]),
                       min_image(x.z - ref.z, P.L[2], P.periodic[2]));
}

constexpr int REF_THREADS = 256;

// Dynamic shared memory of one of the C CTAs of a membrane: every vertex's
// position and velocity, and for its share of the edges the force on each edge's
// four vertices (three planes of 4 x the share), of the triangles their area and
// volume.
__host__ __device__ constexpr int share_of(int n, int C) { return (n + C - 1) / C; }
static constexpr size_t membrane_smem(int nv, int C)
{
    return (size_t)nv * 32 + (size_t)share_of(3 * nv - 6, C) * 48 + (size_t)share_of(2 * nv - 4, C) * 8;
}
// The launch limits are those of the largest mesh, not of the handle that launches: a
// kernel's limit belongs to the process, and a handle with a smaller mesh in another
// thread would lower it between this one's setting and its launch.
constexpr size_t MEMBRANE_SMEM_MAX = membrane_smem(MESH_MAX_NV, 1);
static_assert(MEMBRANE_SMEM_MAX + 1024 <= 227 * 1024, "the largest mesh fits one CTA (with the static arrays)");

// The sums of K terms over n items, as SUM_THREADS threads would add them (item i by
// thread i mod SUM_THREADS, the threads by a tree): the T threads of the CTA take the
// parts of H of them side by side, so T does not change a bit. add(v, i): item i's
// terms. The sums are in lane 0 of warp 0. Every thread of the CTA calls it.
constexpr int SUM_THREADS = 512;
template <int T, int K, class Add>
__device__ __forceinline__ void totals(FF (&sum)[K], FF (*sh)[K], int n, Add &&add)
{
    constexpr int H = SUM_THREADS / T, NW = SUM_THREADS / 32;
    static_assert(SUM_THREADS % T == 0 && T % 32 == 0, "whole parts of whole warps");
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    FF v[H][K];
#pragma unroll
    for (int h = 0; h < H; ++h)
#pragma unroll
        for (int k = 0; k < K; ++k) v[h][k] = FF{0.0f, 0.0f};
    for (int i = threadIdx.x; i < n; i += SUM_THREADS)
#pragma unroll
        for (int h = 0; h < H; ++h)
            if (i + h * T < n) add(v[h], i + h * T);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
            for (int k = 0; k < K; ++k) v[h][k] = ff_add(v[h][k], ff_shfl_down(v[h][k], o));
    if (lane == 0)
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
            for (int k = 0; k < K; ++k) sh[h * (T / 32) + w][k] = v[h][k];
    __syncthreads();
    if (w != 0) return;
#pragma unroll
    for (int k = 0; k < K; ++k) sum[k] = lane < NW ? sh[lane][k] : FF{0.0f, 0.0f};
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < K; ++k) sum[k] = ff_add(sum[k], ff_shfl_down(sum[k], o));
}

// C CTAs (a thread-block cluster; CL false: one CTA) per membrane. Each stages all
// its vertices, computes a share of the edges and triangles and sums a share of
// the vertices, reading the other shares through distributed shared memory. Every
// sum has an order of its own, whatever C and T (the threads) are: the terms of a
// total are added as by SUM_THREADS threads, T of them at a time, a vertex's fan by
// eight lanes. So a membrane gives the same bits alone and in a batch.
//
// Every CTA adds the areas and volumes itself; a lagged membrane's are for the next
// step only, and one CTA of a cluster adds them while the others, which need not wait,
// sum the vertices.
//
// Bound by the arithmetic, above all the five TEA draws and ten normals of a
// bond's random force (about 650 of 900 instructions per edge). Computed from each
// of its ends, with the dihedral from each of its four vertices (eight lanes per
// vertex over its fan), this took 47 us on the 229 cells of 128 replicas after a
// K-Gather of 8 us; every edge once: 38 us in one launch. A single cell is a chain of
// latencies, split over the CTAs (membrane_ctas).
template <bool CL, int T>
__global__ void __launch_bounds__(T, 1024 / T) k_membrane(MemArgs A)
{
    namespace cg = cooperative_groups;
    pdl_enter();
    extern __shared__ float4 mem_sm[];
    __shared__ FF sh_av[SUM_THREADS / 32][2], sh_c[SUM_THREADS / 32][3];
    __shared__ float2 cgv_sh;
    cg::cluster_group cl = cg::this_cluster();
    const int C = CL ? (int)cl.num_blocks() : 1, rank = CL ? (int)cl.block_rank() : 0;
    const int b = blockIdx.x / C, tid = threadIdx.x;
    if (blockIdx.x == 0 && tid == 0) A.mem_ctr[1 - A.q] = A.mem_ctr[A.q] + 1u;   // the next evaluation's
    const RbcDev R = A.rbcs[b];
    const RepParams &P = A.reps[R.rep];
    const float4 ref = A.ref_in[b];
    const int es = share_of(R.ne, C), ts = share_of(R.ntri, C);
    float4 *xs = mem_sm, *vs = xs + R.nv;
    float *fx = reinterpret_cast<float *>(vs + R.nv);        // fy, fz: the next planes of 4 es
    float2 *tri_av = reinterpret_cast<float2 *>(fx + 12 * es);
    const int *tri = A.tri + R.tri_off;

    // vertices, and this CTA's first triangle and edge in flight with them
    const int t0 = rank * ts, t1 = min(t0 + ts, R.ntri), e0 = rank * es, e1 = min(e0 + es, R.ne);
    const int tp = t0 + tid, ep = e0 + tid;
    int3 tv = tp < t1 ? make_int3(tri[3 * tp], tri[3 * tp + 1], tri[3 * tp + 2]) : make_int3(0, 0, 0);
    int4 E = ep < e1 ? A.edge[R.edge_off + ep] : make_int4(0, 0, 0, 0);
    for (int k = tid; k < R.nv; k += T) {
        const float3 x = rel_pos(P, A.mx[R.gbase + k], ref);
        xs[k] = make_float4(x.x, x.y, x.z, 0.0f);
        vs[k] = A.mv[R.gbase + k];
    }
    __syncthreads();
    for (int t = tp; t < t1; t += T) {
        if (t != tp) tv = make_int3(tri[3 * t], tri[3 * t + 1], tri[3 * t + 2]);
        const float3 x0 = f3(xs[tv.x]), x1 = f3(xs[tv.y]), x2 = f3(xs[tv.z]);
        const float3 n = cross(sub(x1, x0), sub(x2, x0));
        tri_av[t - t0] = make_float2(0.5f * sqrtf(dot(n, n)), dot(x0, cross(x1, x2)) * (1.0f / 6.0f));
    }
    // edges (a, b), triangles (a, b, c) and (b, a, d)
    {
        const uint32_t step = A.mem_ctr[A.q] + P.step0;
        const int id0 = R.gbase - P.pbase;
        for (int e = ep; e < e1; e += T) {
            if (e != ep) E = A.edge[R.edge_off + e];
            const float2 bp = A.bond[R.bond_off + e];        // (l_m, k_p)
            const float3 xa = f3(xs[E.x]), xb = f3(xs[E.y]), xc = f3(xs[E.z]), xd = f3(xs[E.w]);
            const float3 d = sub(xb, xa);
            const float l2 = dot(d, d);
            // bond, the force on a: Eq. 10-13 (ue points from b to a)
            float3 f;
            {
                const float il = rsqrtf(l2);
                const float len = l2 * il;
                const float3 ue = scl(-il, d);
                const float x = len / bp.x;
                const float omx = 1.0f - x;
                const float pw = P.m_m == 2.0f ? len * len : __powf(len, P.m_m);
                const float dudl = P.m_wlc0 * (0.25f / (omx * omx) - 0.25f + x) - bp.y / pw;
                const float3 vij = sub(f3(vs[E.x]), f3(vs[E.y]));
                const float ve = dot(vij, ue);
                f = add(scl(-dudl, ue), add(scl(-P.m_gT, vij), scl(-P.m_gC * ve, ue)));
                float z[10];
#pragma unroll
                for (int s = 0; s < 5; ++s) {
                    const float2 g = normal2(pair_bits((uint32_t)(id0 + E.x), (uint32_t)(id0 + E.y), P.seed_lo,
                                                       P.seed_hi, step, 1u + s));
                    z[2 * s] = g.x;
                    z[2 * s + 1] = g.y;
                }
                const float tr = z[0] + z[4] + z[8];
                // (W^S - tr/3 I) e with W^S the symmetric part of Z
                const float s01 = 0.5f * (z[1] + z[3]), s02 = 0.5f * (z[2] + z[6]), s12 = 0.5f * (z[5] + z[7]);
                const float t3 = tr * (1.0f / 3.0f);
                const float3 we = make_float3((z[0] - t3) * ue.x + s01 * ue.y + s02 * ue.z,
                                              s01 * ue.x + (z[4] - t3) * ue.y + s12 * ue.z,
                                              s02 * ue.x + s12 * ue.y + (z[8] - t3) * ue.z);
                f = add(f, add(scl(P.m_rand_T, we), scl(P.m_rand_C * tr, ue)));
            }
            // dihedral: the gradients of the angle theta between the outward
            // normals (positive on a convex fold) times -kb sin(theta - theta0)
            const float3 n1 = cross(d, sub(xc, xa));
            const float3 n2 = cross(sub(xd, xb), d);
            const float n1s = dot(n1, n1), n2s = dot(n2, n2);
            const float le = sqrtf(l2), inv12 = rsqrtf(n1s * n2s);
            const float cos_t = dot(n1, n2) * inv12;
            const float sin_t = dot(cross(n1, n2), d) * inv12 / le;
            const float s = P.m_kb * (sin_t * P.m_cos0 - cos_t * P.m_sin0);
            const float3 u1 = scl(1.0f / n1s, n1), u2 = scl(1.0f / n2s, n2);
            const float a1 = dot(sub(xc, xb), d) / le, a2 = dot(sub(xd, xb), d) / le;
            const float b1 = dot(sub(xa, xc), d) / le, b2 = dot(sub(xa, xd), d) / le;
            const float3 fo[4] = {add(f, scl(s, add(scl(a1, u1), scl(a2, u2)))),
                                  sub(scl(s, add(scl(b1, u1), scl(b2, u2))), f), scl(s * le, u1), scl(s * le, u2)};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float *o = fx + k * es + (e - e0);
                o[0] = fo[k].x;
                o[4 * es] = fo[k].y;
                o[8 * es] = fo[k].z;
            }
        }
    }
    if (CL) cl.sync();
    else __syncthreads();

    // the area and the volume: by every CTA of the membrane, or by the last one of a
    // lagged membrane's, whose forces use the previous step's coefficients
    const bool lagged = P.m_lagged && A.cgv_lag, last = rank == C - 1;
    if (!lagged || last) {
        FF v[2];
        totals<T, 2>(v, sh_av, R.ntri, [&](FF (&u)[2], int t) {
            float2 av;
            if (CL) {
                const int r = t / ts;
                av = cl.map_shared_rank(tri_av, r)[t - r * ts];
            } else {
                av = tri_av[t];
            }
            u[0] = ff_add(u[0], av.x);
            u[1] = ff_add(u[1], av.y);
        });
        if (tid == 0) {
            const double Ab = ff_value(v[0]), Vb = ff_value(v[1]);
            // constraint coefficients of Eq. 14-15, once per membrane in binary64
            // (divisions by A0 and V0 were done once on the host)
            cgv_sh = make_float2((float)((Ab - R.A0) * R.kgA0), (float)((Vb - R.V0) * R.kvV0));
            if (last) {
                A.av_out[b] = make_double2(Ab, Vb);
                A.cgv_out[b] = cgv_sh;
            }
        }
        __syncthreads();
    }

    // a share of the vertices, eight lanes each over the fan
    const float2 coef = lagged ? A.cgv_lag[b] : cgv_sh;
    const float c_area = coef.x, c_vol = coef.y;
    const int parts = lagged && C > 1 ? C - 1 : C;
    const int vsh = share_of(R.nv, parts), v0 = rank * vsh, v1 = rank < parts ? min(v0 + vsh, R.nv) : v0;
    auto edge_force = [&](int code) {
        const int role = code >> 29, e = code & ((1 << 29) - 1);
        const float *o;
        if (CL) {
            const int r = e / es;
            o = cl.map_shared_rank(fx, r) + role * es + (e - r * es);
        } else {
            o = fx + role * es + e;
        }
        return make_float3(o[0], o[4 * es], o[8 * es]);
    };
    for (int k0 = v0; k0 < v1; k0 += T / 8) {
        const int k = k0 + (tid >> 3);
        float3 f = make_float3(0.f, 0.f, 0.f);
        if (k < v1) {
            const FanEntry *fan = A.fan + R.fan_off + (size_t)k * R.fan_stride;
            const float3 xv = f3(xs[k]);
            for (int l = tid & 7; l < R.fan_stride; l += 8) {
                const FanEntry F = fan[l];
                if (F.nb < 0) break;                      // past the vertex's degree
                f = add(f, add(edge_force(F.end), edge_force(F.opp)));
                // triangle (v, nb[l], nb[l+1]): Eq. 14-15
                const float3 xl = f3(xs[F.nb]), xn = f3(xs[F.nb_next]);
                const float3 n = cross(sub(xl, xv), sub(xn, xv));
                const float nn = sqrtf(dot(n, n));
                const float At = 0.5f * nn;
                const float a0 = A.a0j[R.a0j_off + F.tri];
                const float ca = c_area + P.m_kl * (At - a0) / a0;
                const float3 gA = scl(0.5f / nn, cross(n, sub(xn, xl)));
                const float3 gV = scl(1.0f / 6.0f, cross(xl, xn));
                f = sub(f, add(scl(ca, gA), scl(c_vol, gV)));
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            f.x += __shfl_xor_sync(0xffffffffu, f.x, o);
            f.y += __shfl_xor_sync(0xffffffffu, f.y, o);
            f.z += __shfl_xor_sync(0xffffffffu, f.z, o);
        }
        if (k < v1 && (tid & 7) == 0) A.fext[R.gbase + k] = make_float4(f.x, f.y, f.z, 0.0f);
    }
    if (last) {
        // the vertex centroid: the next reference point
        FF v[3];
        totals<T, 3>(v, sh_c, R.nv, [&](FF (&u)[3], int k) {
            const float4 x = xs[k];
            u[0] = ff_add(u[0], x.x);
            u[1] = ff_add(u[1], x.y);
            u[2] = ff_add(u[2], x.z);
        });
        if (tid == 0) {
            const double inv = R.inv_nv;
            float c3[3] = {(float)(ref.x + ff_value(v[0]) * inv), (float)(ref.y + ff_value(v[1]) * inv),
                           (float)(ref.z + ff_value(v[2]) * inv)};
            for (int c = 0; c < 3; ++c)
                if (P.periodic[c]) {
                    if (c3[c] < 0.0f) c3[c] += P.L[c];
                    else if (c3[c] >= P.L[c]) c3[c] -= P.L[c];
                }
            A.ref_out[b] = make_float4(c3[0], c3[1], c3[2], 0.0f);
        }
    }
    if (CL) cl.sync();                 // the shares stay until every CTA has read them
}

// Reference point of each membrane of a loaded state, from the uploaded
// load-order positions x3 (three floats per particle): the centroid of its
// vertices unwrapped along the mesh's edges from vertex 0 by the minimum
// image, folded into the box. Each round, every unlabelled vertex takes its
// image offsets k (per axis) from a labelled neighbour, k_u = k_v -
// rint((p_u - p_v) / L); for a mesh whose edges are shorter than half the
// box every path gives the same k. The coordinates relative to vertex 0,
// (p_u - p_0) + k_u L, are summed with float-float compensation in a fixed
// tree (as K-Gather sums its terms) and combined with p_0 once in binary64.
// All arithmetic but that last step is binary32 (the FP64 unit of this GPU
// is narrow). One CTA per membrane; the labels in shared memory (0: not
// reached; else the three offsets, biased by 64, in the low bytes and bit
// 24 set), and with STAGED the vertices' positions and neighbours too. A
// vertex no edge reaches is left out of the sum.
template <bool STAGED>
__global__ void __launch_bounds__(REF_THREADS) k_mem_ref(const float *__restrict__ x3,
                                                         const RbcDev *__restrict__ rbcs,
                                                         const FanEntry *__restrict__ fan,
                                                         const RepParams *__restrict__ reps, float4 *ref_out,
                                                         int max_nv, int max_stride)
{
    extern __shared__ int sm[];
    __shared__ FF wsum[REF_THREADS / 32][3];
    const int b = blockIdx.x;
    const RbcDev R = rbcs[b];
    const RepParams &P = reps[R.rep];
    const int nv = R.nv, stride = R.fan_stride;
    volatile int *lab = sm;
    float *ps = reinterpret_cast<float *>(sm + max_nv);             // STAGED: [3 nv]
    int *nbs = sm + 4 * max_nv;                                     // STAGED: [nv stride]
    const float *pg = x3 + 3 * (size_t)R.gbase;
    const FanEntry *fg = fan + R.fan_off;
    constexpr int SET = 1 << 24, ZERO = 64 | 64 << 8 | 64 << 16;
    if (STAGED) {
        for (int i = threadIdx.x; i < 3 * nv; i += blockDim.x) ps[i] = pg[i];
        for (int i = threadIdx.x; i < nv * stride; i += blockDim.x) nbs[i] = fg[i].nb;
    }
    for (int u = threadIdx.x; u < nv; u += blockDim.x) lab[u] = u == 0 ? (SET | ZERO) : 0;
    __syncthreads();
    const float *p = STAGED ? ps : pg;
    bool changed;
    do {
        changed = false;
        for (int u = threadIdx.x; u < nv; u += blockDim.x) {
            if (lab[u]) continue;
            for (int l = 0; l < stride; ++l) {
                const int v = STAGED ? nbs[u * stride + l] : fg[(size_t)u * stride + l].nb;
                if (v < 0) break;
                const int lv = lab[v];
                if (!lv) continue;
                int code = SET;
                for (int c = 0; c < 3; ++c) {
                    const int k = ((lv >> (8 * c)) & 255) - 64 - (int)rintf((p[3 * u + c] - p[3 * v + c]) * P.inv_L[c]);
                    code |= (k + 64) << (8 * c);
                }
                lab[u] = code;
                changed = true;
                break;
            }
        }
    } while (__syncthreads_or(changed));
    FF acc[3] = {FF{0.0f, 0.0f}, FF{0.0f, 0.0f}, FF{0.0f, 0.0f}};
    for (int u = threadIdx.x; u < nv; u += blockDim.x) {
        const int lu = lab[u];
        if (!lu) continue;
        for (int c = 0; c < 3; ++c)
            acc[c] = ff_add(acc[c], __fmaf_rn((float)(((lu >> (8 * c)) & 255) - 64), P.L[c], p[3 * u + c] - p[c]));
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        for (int c = 0; c < 3; ++c) acc[c] = ff_add(acc[c], ff_shfl_down(acc[c], o));
    if (lane == 0)
        for (int c = 0; c < 3; ++c) wsum[w][c] = acc[c];
    __syncthreads();
    if (threadIdx.x != 0) return;
    float cf[3];
    for (int c = 0; c < 3; ++c) {
        FF t = wsum[0][c];
        for (int k = 1; k < REF_THREADS / 32; ++k) t = ff_add(t, wsum[k][c]);
        double y = (double)p[c] + ff_value(t) / (double)nv;
        if (P.periodic[c]) y -= (double)P.L[c] * floor(y / (double)P.L[c]);
        cf[c] = (float)y;
        if (!(cf[c] < P.L[c])) cf[c] = 0.0f;      // rounded up onto L
    }
    ref_out[b] = make_float4(cf[0], cf[1], cf[2], 0.0f);
}

void launch_mem_ref(const float *x3, const RbcDev *rbcs, const FanEntry *fan, const RepParams *reps, float4 *ref_out,
                    int n_rbc, int max_nv, int max_stride, cudaStream_t st)
{
    if (n_rbc <= 0) return;
    constexpr size_t SMEM_MAX = 200 * 1024;
    const size_t staged = sizeof(int) * ((size_t)4 * max_nv + (size_t)max_nv * max_stride);
    const size_t plain = sizeof(int) * (size_t)max_nv;       // (at most 4 KB)
    if (staged <= SMEM_MAX) {
        // (the same limit for every handle, as for k_membrane)
        if (staged > 48 * 1024)
            cudaFuncSetAttribute(k_mem_ref<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_MAX);
        k_mem_ref<true><<<n_rbc, REF_THREADS, staged, st>>>(x3, rbcs, fan, reps, ref_out, max_nv, max_stride);
    } else {
        k_mem_ref<false><<<n_rbc, REF_THREADS, plain, st>>>(x3, rbcs, fan, reps, ref_out, max_nv, max_stride);
    }
}

// CTAs and threads per membrane: the most CTAs that leave one per SM (clusters of eight
// and four fill a little less than 152 SMs), since a second wave, or a second CTA on
// every SM, costs more than the split gains; beyond 152 membranes one, which then share
// the SMs two by two, and two for meshes so large that one CTA fills an SM's shared
// memory. Measured, launch by launch, us, with 1, 2, 4 and 8 CTAs of 512 threads (in
// brackets the two kernels with a lane per fan entry that this one replaced): 10 meshes
// of 500 vertices 26.6, 20.8, 16.4, 14.3 (22); 36 of 26.6, 20.7, 16.7, 18.4 (24); 76 of
// 26.6, 20.4, 28.7, 36.9 (32); 152 of 26.6, 28.7, 43, 60 (45); 153 of 37, 39, 43, 60
// (47); 300 of 41, 52, 72 (76). 10 of 1000 vertices 40.5, 30.7, 22.5, 18.4 (22); 153 of
// 82, 64, 66, 80 (76); 300 of 84, 82, 109 (129).
// Beside the half shell's walk a few membranes take smaller CTAs, which disturb it less
// (a cell in 20^3, eight lanes, us per step: 31.3 with 8 x 256 threads, 32.4 with
// 8 x 512, 31.9 with 4 x 512; the full shell, which waits for them, 36.4, 35.6 and 36.9).
// Many small meshes: with 128 threads eight of them share an SM (3,000 meshes of 12
// vertices 29 us, with 512 threads 78, the kernels before 71; 1,000 of 42 19, 35, 47).
struct MembraneSplit { int ctas, threads; };
constexpr size_t SMEM_PER_SM = 228 * 1024;
static MembraneSplit membrane_split(int n_rbc, int max_nv, bool beside_walk)
{
    if (n_rbc <= 16) return {8, beside_walk && max_nv <= 512 ? 256 : 512};
    if (n_rbc <= 152) return {n_rbc <= 36 ? 4 : n_rbc <= 76 ? 2 : 1, 512};
    if (membrane_smem(max_nv, 1) + 2048 > SMEM_PER_SM / 2) return {2, 512};
    return {1, max_nv <= 66 ? 128 : 512};
}

void launch_membrane(const MemArgs &a, cudaStream_t st, bool pdl, bool beside_walk)
{
    if (a.n_rbc <= 0) return;
    const MembraneSplit split = membrane_split(a.n_rbc, a.max_nv, beside_walk);
    const int C = split.ctas;
    auto kern = C == 1 ? (split.threads == 128 ? k_membrane<false, 128> : k_membrane<false, 512>)
                       : (split.threads == 256 ? k_membrane<true, 256> : k_membrane<true, 512>);
    const size_t smem = membrane_smem(a.max_nv, C);
    if (smem > 48 * 1024)
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MEMBRANE_SMEM_MAX);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = a.n_rbc * C;
    cfg.blockDim = split.threads;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    int n = 0;
    if (C > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = C;
        at[n].val.clusterDim.y = at[n].val.clusterDim.z = 1;
        ++n;
    }
    if (pdl) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    cudaLaunchKernelEx(&cfg, kern, a);
}

}  // namespace tdpd
