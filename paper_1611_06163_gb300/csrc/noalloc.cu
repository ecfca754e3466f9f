// Pair force + flux without any device allocation (tdpd_pair_forces_noalloc).
//
// Every scratch buffer this entry point needs -- the cell histogram and
// offsets, the sorted copy of the particle state, the slot maps -- lives
// in one file-scope __device__ array of fixed size, g_noalloc_scratch, which
// every GPU that loads the library holds until the process exits. The caller
// supplies inputs and outputs; nothing is allocated or freed per call.
//
// In host code the name g_noalloc_scratch is only a host-side stand-in for the
// symbol, not a device address: handing it to a kernel would fault or, where
// the GPU can reach host memory, silently use the wrong memory. The device
// address is obtained once per device with cudaGetSymbolAddress, with that
// device current, and cached.
#include <cmath>
#include <cstdio>
#include <mutex>

#include "launch.h"

using namespace tdpd;

namespace {

constexpr int NA_N = TDPD_NOALLOC_MAX_PARTICLES;
constexpr int NA_C = TDPD_NOALLOC_MAX_CELLS;
constexpr int NA_S = TDPD_NOALLOC_MAX_SPECIES;
constexpr int NA_TILES = (NA_C + SCAN_TILE - 1) / SCAN_TILE;
static_assert(NA_C % SCAN_TILE == 0, "the cell capacity is whole scan tiles");

// Layout of the scratch array (only its size and offsets are used on the host).
struct __align__(256) NoAllocLayout {
    RepParams params;
    float4 pos[NA_N], vt[NA_N], vel[NA_N], frc[NA_N];
    float C[NA_N * NA_S], Ct[NA_N * NA_S], Q[NA_N * NA_S];
    float4 fext[NA_N];
    int inv[NA_N];
    int2 cellrank[NA_N];
    int keys[NA_N];
    int count[NA_C];
    int cell_start[NA_C + 4];
    int tile_sum[2][NA_TILES];
    uint32_t err[4];
    uint32_t step_ctr[4];
};
static_assert(sizeof(NoAllocLayout) <= TDPD_NOALLOC_SCRATCH_BYTES, "scratch size as documented in tdpd.h");

static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocLayout)];

std::mutex g_mu;
constexpr int MAX_DEVICES = 64;
NoAllocLayout *g_dev_ptr[MAX_DEVICES] = {};

tdpd_status na_fail(tdpd_status code, const char *msg)
{
    set_thread_error(msg);
    return code;
}

// The inputs sorted by cell, and by id within a cell, straight from the caller's
// arrays: clear, bin, scan (k_scan), keys, place. Each launch is a few dependent
// loads long, so fewer of them is what helps (12,000 particles: 16.8 us; with the
// inputs first copied to a state buffer and gathered from there: 22.2; all of it in
// one thread-block cluster: 27 with counters in the L2, 35 with counters and keys in
// distributed shared memory, whose scattered atomics and loads are slower still).

// What the binning counts into, the input check word and the call's parameters
// (word by word: one thread's copy of the structure took 9 us).
__global__ void k_na_clear(const __grid_constant__ RepParams P, int n, int cells, uint32_t step, NoAllocLayout *S)
{
    pdl_enter();
    const int stride = gridDim.x * blockDim.x, g0 = blockIdx.x * blockDim.x + threadIdx.x;
    static_assert(sizeof(RepParams) % 4 == 0, "copied by words");
    for (int w = g0; w < (int)(sizeof(RepParams) / 4); w += stride)
        reinterpret_cast<uint32_t *>(&S->params)[w] = reinterpret_cast<const uint32_t *>(&P)[w];
    if (g0 == 0) {
        S->err[0] = S->err[1] = 0u;
        S->step_ctr[0] = step;
        S->cell_start[cells] = n;            // the end of the last scanned tile
    }
    for (int c = g0; c < cells; c += stride) S->count[c] = 0;
    for (int t = g0; t < 2 * NA_TILES; t += stride) S->tile_sum[t / NA_TILES][t % NA_TILES] = 0;
}

__global__ void k_na_bin(int n, const float *__restrict__ pos, NoAllocLayout *S)
{
    pdl_enter();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    int c = -1;
    if (k < n) {
        c = cell_of(S->params, pos[3 * k], pos[3 * k + 1], pos[3 * k + 2]);
        S->cellrank[k] = make_int2(c, atomicAdd(S->count + c, 1));
    }
    add_tile_count(S->tile_sum[0], c);
}

__global__ void k_na_keys(int n, NoAllocLayout *S)
{
    pdl_enter();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int2 cr = S->cellrank[k];
    S->keys[S->cell_start[cr.x] + cr.y] = k;
}

// The particle of slot d's key goes to its rank by id inside its cell.
__global__ void k_na_place(int n, int ns, const float *__restrict__ pos, const float *__restrict__ vel,
                           const float *__restrict__ conc, const int32_t *__restrict__ type, NoAllocLayout *S)
{
    pdl_enter();
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const int k = S->keys[e], c = S->cellrank[k].x;
    const int lo = S->cell_start[c], hi = S->cell_start[c + 1];
    float4 p = make_float4(pos[3 * k], pos[3 * k + 1], pos[3 * k + 2], 0.f);
    const float4 v = make_float4(vel[3 * k], vel[3 * k + 1], vel[3 * k + 2], __int_as_float(0));
    float cs[NA_S];
#pragma unroll
    for (int s = 0; s < NA_S; ++s) cs[s] = s < ns ? conc[(size_t)k * ns + s] : 0.f;
    int t = type[k], d = lo;
    for (int q = lo; q < hi; ++q) d += S->keys[q] < k;
    // a type outside [0, n_types) is recorded (the outputs become NaN)
    // and replaced by type 0, so that no table lookup leaves its range
    if (t < 0 || t >= S->params.ntypes) {
        atomicOr(&S->err[1], 4u);
        t = 0;
    }
    p.w = __int_as_float((int)((uint32_t)k | ((uint32_t)t << 24)));
    S->pos[d] = p;
    S->vel[d] = v;
    S->vt[d] = make_float4(v.x, v.y, v.z, __int_as_float(-1));
    S->frc[d] = make_float4(0.f, 0.f, 0.f, 0.f);
    S->inv[k] = d;
#pragma unroll
    for (int s = 0; s < NA_S; ++s)
        if (s < ns) {
            S->C[(size_t)d * ns + s] = cs[s];
            S->Ct[(size_t)d * ns + s] = cs[s];
            S->Q[(size_t)d * ns + s] = 0.f;
        }
}

// Load-order outputs; every output is NaN when an input type was out of
// range or some force came out non-finite (the caller checks the outputs).
__global__ void k_na_unpack(int n, int ns, const NoAllocLayout *S, float *force, float *flux)
{
    pdl_enter();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const bool bad = (S->err[0] | S->err[1]) != 0u;
    const float nan = __int_as_float(0x7fc00000);
    const int slot = S->inv[k];
    const float4 f = S->frc[slot];
    force[3 * k] = bad ? nan : f.x;
    force[3 * k + 1] = bad ? nan : f.y;
    force[3 * k + 2] = bad ? nan : f.z;
    for (int s = 0; s < ns; ++s) flux[(size_t)k * ns + s] = bad ? nan : S->Q[(size_t)slot * ns + s];
}

Buffers buffers(NoAllocLayout *S)
{
    Buffers B;
    B.pos = S->pos;
    B.vt = S->vt;
    B.vel = S->vel;
    B.frc = S->frc;
    B.C = S->C;
    B.Ct = S->Ct;
    B.Q = S->Q;
    return B;
}

}  // namespace

extern "C" tdpd_status tdpd_pair_forces_noalloc(const tdpd_config *cfg, const float *pair_coef,
                                                const float *kappa, int n, const float *pos,
                                                const float *vel, const float *conc,
                                                const int32_t *type, uint32_t step, float *force,
                                                float *flux, void *stream)
{
    if (!cfg || !pair_coef || !kappa) return na_fail(TDPD_EINVAL, "noalloc: null parameter pointer");
    if (n < 1 || n > NA_N) return na_fail(TDPD_EINVAL, "noalloc: particle count must be 1..TDPD_NOALLOC_MAX_PARTICLES");
    if (!pos || !vel || !conc || !type || !force || !flux) return na_fail(TDPD_EINVAL, "noalloc: null device array");
    const tdpd_config &c = *cfg;
    {
        // the checks of tdpd_create, then this entry point's own limits
        char why[200], msg[240];
        if (config_error(c, why, sizeof why)) {
            std::snprintf(msg, sizeof msg, "noalloc: %s", why);
            return na_fail(TDPD_EINVAL, msg);
        }
    }
    if (c.n_species > NA_S) return na_fail(TDPD_EINVAL, "noalloc: n_species must be 1..TDPD_NOALLOC_MAX_SPECIES");
    if (!c.periodic[2]) return na_fail(TDPD_EINVAL, "noalloc: the box must be periodic on every axis");
    const int m = c.cells_per_cutoff > 0 ? c.cells_per_cutoff : 2;
    const float rcut = c.rc > c.rcc ? c.rc : c.rcc;
    int nc[3];
    long ncell = 1;
    for (int k = 0; k < 3; ++k) {
        if (!(c.L[k] > 0) || (double)c.L[k] < 3.0 * rcut * 1.0001)
            return na_fail(TDPD_EINVAL, "noalloc: every box edge must hold three cut-offs");
        const double ncd = std::floor((double)c.L[k] * m / ((double)rcut * 1.0001));
        if (ncd > NA_C) return na_fail(TDPD_EINVAL, "noalloc: the box needs more than TDPD_NOALLOC_MAX_CELLS cells");
        nc[k] = (int)ncd;
        if (nc[k] < 2 * m + 1) return na_fail(TDPD_EINVAL, "noalloc: too few cells");
        ncell *= nc[k];
    }
    if (ncell > NA_C) return na_fail(TDPD_EINVAL, "noalloc: the box needs more than TDPD_NOALLOC_MAX_CELLS cells");

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES)
        return na_fail(TDPD_ECUDA, "noalloc: no usable current device");
    NoAllocLayout *S = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_dev_ptr[dev]) {
            void *p = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
            if (e != cudaSuccess || !p) return na_fail(TDPD_ECUDA, "noalloc: cudaGetSymbolAddress of the scratch array failed");
            g_dev_ptr[dev] = static_cast<NoAllocLayout *>(p);
        }
        S = g_dev_ptr[dev];
    }

    const int ns = c.n_species;
    const RepParams P = build_rep_params(c, pair_coef, kappa, nc, m, 0, 0, n);
    cudaStream_t st = (cudaStream_t)stream;
    const Buffers b1 = buffers(S);
    const RepParams *dP = &S->params;
    const int n_tiles = (int)((ncell + SCAN_TILE - 1) / SCAN_TILE), grid = (n + 255) / 256;
    launch_pdl(k_na_clear, 16, 256, st, P, n, n_tiles * SCAN_TILE, step, S);
    launch_pdl(k_na_bin, grid, 256, st, n, pos, S);
    launch_scan(S->count, S->cell_start, n_tiles, S->tile_sum[0], S->tile_sum[1], S->step_ctr, 0, st);
    launch_pdl(k_na_keys, grid, 256, st, n, S);
    launch_pdl(k_na_place, grid, 256, st, n, ns, pos, vel, conc, type, S);
    PairArgs a{};
    a.b = b1;
    a.fext = S->fext;
    a.reps = dP;
    a.cell_start = S->cell_start;
    a.count = S->count;
    a.cellrank = S->cellrank;
    a.tile_sum = S->tile_sum[1];
    a.err = S->err;
    a.step_ctr = S->step_ctr;
    a.n = n;
    a.ns = ns;
    a.integrate = 0;
    a.std_exp = c.s_f == 2.0f && c.s_c == 2.0f;
    // lanes per particle: the stencil's 25 rows are split over them, and while the
    // GPU is not full the rows left to each lane set the time (measured, pair
    // kernel: 648 particles 34 us with 8 lanes, 18 with 32; 4,000: 22.5 with 8,
    // 17.7 with 16, 19.8 with 32; 12,000: 24.5 with 8, 28.6 with 16)
    a.lpp = n <= 1500 ? 32 : n <= 6000 ? 16 : 8;
    launch_pair(a, st);
    launch_pdl(k_na_unpack, grid, 256, st, n, ns, S, force, flux);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return na_fail(TDPD_ECUDA, cudaGetErrorString(e));
    return TDPD_OK;
}
