// batch.cu -- batched calibration sweep: many independent pseudopotential lattices at once.
//
// The calibration runs the pseudopotential model needs (Sec. 3: sigma^Li, kappa^P and
// kappa^Li tuned against coexistence densities, interface width and surface tension; Secs.
// 5.1-5.2: its parameters are set from preliminary runs) are many small, independent
// lattices of uneven sizes and step counts.  Run one at a time, the small ones are
// launch-latency bound and the large ones leave most SMs idle.  Here they run together:
//
//   resident lattices  -- those of at most 4452 cells: one CTA per lattice runs every step of
//                         that lattice in shared memory and registers, in one persistent launch
//                         per size class (no HBM traffic per step);
//   tiled lattices     -- the rest: one launch per time step over a work table, replayed as
//                         captured 64-step CUDA graphs on a second stream, concurrently with
//                         the resident launch.  While the unfinished lattices hold many cells
//                         the table is one of (lattice, strip) items for the two-cells-per-lane
//                         TMA strip of the context path (pp_pair_strip), then one of tiles for
//                         CTAs that each take a run of them (pp_batch_tile).
//
// An autotuner picks the resident cells per thread and the strip height by timing short trials
// (cached per shape class for the process), and orders work longest-first.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "../../include/lbm.h"
#include "lbm_kernels.cuh"
#include "ring.cuh"
#include "step_pair.cuh"
#include "tile.h"
#include "rest_host.h"

namespace {

thread_local char g_batch_msg[256] = "";
int bfail(cudaError_t e, const char* what) {
    snprintf(g_batch_msg, sizeof(g_batch_msg), "%s: %s", what, cudaGetErrorString(e));
    return LBM_ERR_CUDA;
}
#define BCK(call)                                             \
    do {                                                      \
        cudaError_t e_ = (call);                              \
        if (e_ != cudaSuccess) return bfail(e_, #call);       \
    } while (0)

constexpr int kBPWarps = 4;
constexpr int kBPStages = 6;
static_assert(kBPStages >= 4, "the pseudopotential strip ring needs at least 4 stages");
using BPSmem = lbmk::WarpStripSmem<kBPWarps, kBPStages, 60>;
constexpr int kBPTX = BPSmem::TX;  // widest pair strip (240 columns)
constexpr int kChunk = 64;       // steps per captured graph
constexpr int kTileCtasPerSM = 4;          // resident CTAs of the tile kernel
// Unfinished cells from which strips are the faster step (24 lattices of 192^2 .. 512^2, 0.8 million
// cells: 6.5 ms with tiles, 10.4 with strips; 96 lattices, 3.9 million cells at first, 100 .. 400 steps:
// 27.2 ms with tiles only, 25.6 with strips only, 24.7 with this rule, 24.9 and 24.6 with 1.5 and 3.5
// million).
constexpr long long kStripCells = 2500000;
constexpr size_t kResidentSmemMax = 200 * 1024;

struct BatchLattice {
    lbmk::StepParams<float> P;  // physics and geometry (nx, ny, rows, pitch)
    float* buf[2];              // ping-pong stored populations
    float* scratch;             // 2 N floats: rho and psi for observables
    double* rho0;               // N initial densities (of their own, or in scratch: lbm_batch::rho0)
    double RT, a, b4;           // FP64 EOS constants for the observables (pressure jump)
    int nsteps;
    int geometry;
    int resident;
    int pad_;
};

struct BatchItem {
    int lat, x0, w, y0, y1;
};

size_t a256(size_t n) { return (n + 255) & ~size_t(255); }

// The size rule of resident lattices: 11 floats and an int16 per cell within kResidentSmemMax, that is up to
// kResidentCells (the kernel keeps 9 floats per cell in shared memory).
constexpr size_t resident_bytes(size_t N) { return 11 * N * sizeof(float) + ((2 * N + 15) & ~size_t(15)); }
constexpr int kResidentCells = 4452;
static_assert(resident_bytes(kResidentCells) <= kResidentSmemMax && resident_bytes(kResidentCells + 1) > kResidentSmemMax,
              "the largest resident lattice");
constexpr size_t resident_smem(int cells) { return 9 * sizeof(float) * (size_t)((cells + 3) & ~3); }

// One population buffer of a lattice: 9 FP32 planes plus the int16 rest plane (plane 9).
size_t buffer_bytes(long long pitch) { return a256(10 * (size_t)pitch * 4); }

}  // namespace

namespace lbmk {

// ------------------------------------------------------------------------------------
// Resident lattice: all steps on one SM.  A thread keeps PAIRS pairs of cells for the whole run: their
// rest populations and extensions are its own (in registers with one pair; with two 8 to 80 bytes a thread
// spill to local memory, with four, which lattices above 2048 cells need, 196 to 788), the eight moving
// populations are in shared memory in the stored layout S_i(x) (post-collision at the source cell).  Per step: (A) pull every cell's
// populations into registers and write psi; barrier; (B) collide from the neighbours' psi and write f*
// over S, which every thread has read by then; barrier.  So no population moves through global memory
// and each step has two barriers.  A pair is two cells of one row when nx is even, so that reads of
// unshifted columns and all writes are 8 bytes; otherwise the cells c and c + ceil(N/2).
//
// What bounds it: issue and the latency of the two phases at 16 warps per SM (128 registers a thread).
// The earlier kernel (one cell at a time, f* through a global buffer, three barriers) took 11.4 us per
// step for 64 x 64 cells on each of 152 SMs (54.8 GLUPS) and 12.5 us for 608 lattices of 256 x 4 (49.6);
// this one 6.8 us (91.5) and 7.4 us (84.4).
struct CellOff {  // steps to the wrapped neighbours of a cell, two 16-bit numbers each: columns, rows
    int lr, mp;
    __device__ __forceinline__ int dl() const { return (short)lr; }
    __device__ __forceinline__ int dr() const { return lr >> 16; }
    __device__ __forceinline__ int dm() const { return (short)mp; }
    __device__ __forceinline__ int dp() const { return mp >> 16; }
};
// left of cell c and right of cell d of the same row
__device__ __forceinline__ CellOff cell_off(int c, int d, int nx, int ny) {
    const int x = c % nx, y = c / nx;
    const int l = x == 0 ? nx - 1 : -1, r = d % nx == nx - 1 ? 1 - nx : 1;
    const int m = y == 0 ? (ny - 1) * nx : -nx, p = y == ny - 1 ? -(ny - 1) * nx : nx;
    return {(l & 0xffff) | r << 16, (m & 0xffff) | p << 16};
}

template <int PAIRS, int THREADS, bool EVEN>
__global__ void __launch_bounds__(THREADS, 1)
    pp_resident_kernel(const BatchLattice* __restrict__ lats, const int* __restrict__ ids, int step_limit) {
    extern __shared__ __align__(16) float rsm[];
    __shared__ StepParams<float> P;  // (read where they are used: registers are short)
    const BatchLattice& L = lats[ids[blockIdx.x]];
    for (int i = threadIdx.x; i < (int)sizeof(P) / 4; i += blockDim.x)  // (a CTA may be one warp)
        reinterpret_cast<int*>(&P)[i] = reinterpret_cast<const int*>(&L.P)[i];
    const int nx = L.P.nx, ny = L.P.ny, N = nx * ny, H = (N + 1) / 2;
    const int Ns = (N + 3) & ~3;  // plane stride
    const long long pitch = L.P.pitch;
    auto S = [&](int i) { return rsm + (i - 1) * Ns; };  // planes 1..8
    float* psi = rsm + 8 * Ns;
    const float* g0 = L.buf[0];
    for (int i = 1; i < 9; ++i)
        for (int c = threadIdx.x; c < N; c += blockDim.x) S(i)[c] = g0[i * pitch + c];
    // this thread's pairs (pair p: cells a(p), b(p); b may not exist when N is odd)
    auto cell_a = [&](int p) { return EVEN ? 2 * p : p; };
    auto cell_b = [&](int p) { return EVEN ? 2 * p + 1 : p + H; };
    F2 v[PAIRS][9];
    unsigned q[PAIRS];
    CellOff oa[PAIRS], ob[EVEN ? 1 : PAIRS];
#pragma unroll
    for (int j = 0; j < PAIRS; ++j) {
        const int p = threadIdx.x + j * blockDim.x, a = cell_a(p), b = cell_b(p);
        v[j][0] = F2::c(1.0f);
        q[j] = 0;
        if (p < H) {
            const short* ql = rest_lo_plane(g0, pitch);
            oa[j] = cell_off(a, EVEN ? b : a, nx, ny);
            if (!EVEN) ob[EVEN ? 0 : j] = cell_off(b < N ? b : a, b < N ? b : a, nx, ny);
            v[j][0] = F2(g0[a], g0[b < N ? b : a]);
            q[j] = (unsigned)(unsigned short)ql[a] | (unsigned)(unsigned short)ql[b < N ? b : a] << 16;
        }
    }
    __syncthreads();
    // both cells' values of a plane, dx columns and dy rows away
    auto at = [&](const float* f, int j, int p, int dx, int dy) {
        const CellOff A = oa[j];
        if constexpr (EVEN) {
            const int c = 2 * p + (dy < 0 ? A.dm() : dy > 0 ? A.dp() : 0);
            if (dx == 0) return F2(*reinterpret_cast<const float2*>(f + c));
            if (dx < 0) return F2(f[c + A.dl()], f[c]);
            return F2(f[c + 1], f[c + 1 + A.dr()]);
        } else {
            const CellOff B = ob[j];
            const int a = p + (dx < 0 ? A.dl() : dx > 0 ? A.dr() : 0) + (dy < 0 ? A.dm() : dy > 0 ? A.dp() : 0);
            const int b0 = p + H < N ? p + H : p;
            const int b = b0 + (dx < 0 ? B.dl() : dx > 0 ? B.dr() : 0) + (dy < 0 ? B.dm() : dy > 0 ? B.dp() : 0);
            return F2(f[a], f[b]);
        }
    };
    auto put = [&](float* f, int p, F2 w) {
        if constexpr (EVEN) {
            *reinterpret_cast<float2*>(f + 2 * p) = w.v;
        } else {
            f[p] = w.v.x;
            if (p + H < N) f[p + H] = w.v.y;
        }
    };
    const int nsteps = step_limit >= 0 ? min(step_limit, L.nsteps) : L.nsteps;
    for (int s = 0; s < nsteps; ++s) {
#pragma unroll
        for (int j = 0; j < PAIRS; ++j) {
            const int p = threadIdx.x + j * blockDim.x;
            if (p >= H) continue;
            F2* w = v[j];
            w[1] = at(S(1), j, p, -1, 0);
            w[2] = at(S(2), j, p, 0, -1);
            w[3] = at(S(3), j, p, 1, 0);
            w[4] = at(S(4), j, p, 0, 1);
            w[5] = at(S(5), j, p, -1, -1);
            w[6] = at(S(6), j, p, 1, -1);
            w[7] = at(S(7), j, p, 1, 1);
            w[8] = at(S(8), j, p, -1, 1);
            put(psi, p, pseudo_psi_v(sum9_v(w), P));
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < PAIRS; ++j) {
            const int p = threadIdx.x + j * blockDim.x;
            if (p >= H) continue;
            F2 pn[9], d0;
            pn[0] = at(psi, j, p, 0, 0);
            pn[1] = at(psi, j, p, 1, 0);
            pn[2] = at(psi, j, p, 0, 1);
            pn[3] = at(psi, j, p, -1, 0);
            pn[4] = at(psi, j, p, 0, -1);
            pn[5] = at(psi, j, p, 1, 1);
            pn[6] = at(psi, j, p, -1, 1);
            pn[7] = at(psi, j, p, -1, -1);
            pn[8] = at(psi, j, p, 1, -1);
            pp_collide_v<F2, true>(v[j], sum9_v(v[j]), pn[0], pn, P, &d0);
            q[j] = rest_update_pair(v[j][0], q[j], d0, P);
#pragma unroll
            for (int i = 1; i < 9; ++i) put(S(i), p, v[j][i]);
        }
        __syncthreads();
    }
    // final state to the buffer the tiled convention uses after nsteps steps
    float* g = L.buf[nsteps & 1];
    short* ql = rest_lo_plane(g, pitch);
#pragma unroll
    for (int j = 0; j < PAIRS; ++j) {
        const int p = threadIdx.x + j * blockDim.x, a = cell_a(p), b = cell_b(p);
        if (p >= H) continue;
        g[a] = v[j][0].v.x;
        ql[a] = (short)(q[j] & 0xffffu);
        if (b < N) {
            g[b] = v[j][0].v.y;
            ql[b] = (short)(q[j] >> 16);
        }
    }
    for (int i = 1; i < 9; ++i)
        for (int c = threadIdx.x; c < N; c += blockDim.x) g[i * pitch + c] = S(i)[c];
}

// Tiled lattices, two cells per lane: one strip of one lattice per CTA, one step per launch.
template <int NW, int S, bool NEAR>
__global__ void __launch_bounds__((NW + 1) * 32, 4)
    pp_batch_pair(const BatchLattice* __restrict__ lats, const BatchItem* __restrict__ items,
                  const int* __restrict__ state, int k, int* __restrict__ err) {
    using Smem = WarpStripSmem<NW, S, 60>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
    const BatchItem it = items[blockIdx.x];
    const BatchLattice& L = lats[it.lat];
    const int step = state[0] + k;
    if (step >= L.nsteps) return;
    // in shared memory, not in registers: 94 of them allow four CTAs per SM, 110 three (a sweep of 3.9
    // million cells: 25.6 ms against 29.1)
    __shared__ StepParams<float> P;
    static_assert(sizeof(P) / 4 <= (NW + 1) * 32, "one word per thread");
    if (threadIdx.x < sizeof(P) / 4)
        reinterpret_cast<int*>(&P)[threadIdx.x] = reinterpret_cast<const int*>(&L.P)[threadIdx.x];
    __syncthreads();
    pp_pair_strip<NW, S, false, NEAR>(L.buf[step & 1], L.buf[(step + 1) & 1], P, it.x0, it.w, it.y0, it.y1, sm, err);
}

// The same lattices in tiles of kBatchTileRows rows, one row per warp (step_tile.cuh): CTA b takes its
// share of the tiles of the unfinished lattices, which head the table (state[1] of them), one after the
// other.  Neighbouring tiles follow each other, so their common halo rows are still in L1; a lattice's
// constants are read from shared memory where they are used, because held in registers they would cost
// CTAs per SM.  (Copying the next tile's rows to shared memory ahead, two cp.async stages per warp, made
// a sweep that exceeds L2 3% faster and a small one 8% slower; the strips are faster there.)
constexpr int kBatchTileRows = 4;
__global__ void __launch_bounds__(32 * (kBatchTileRows + 2))
    pp_batch_tile(const BatchLattice* __restrict__ lats, const BatchItem* __restrict__ tiles,
                  const int* __restrict__ state, int k) {
    constexpr int R = kBatchTileRows;
    __shared__ F2 s_psi[2][R + 2][32];
    __shared__ StepParams<float> P;
    const int step = state[0] + k, count = state[1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = 2 * lane - 2;
    const int i1 = (int)((long long)count * (blockIdx.x + 1) / gridDim.x);
    int lat = -1, par = 0;
    bool done = false;
    const float* fin = nullptr;
    float* fout = nullptr;
    for (int i = (int)((long long)count * blockIdx.x / gridDim.x); i < i1; ++i) {
        const BatchItem it = tiles[i];
        if (it.lat != lat) {
            lat = it.lat;
            const BatchLattice& L = lats[lat];
            done = step >= L.nsteps;
            fin = L.buf[step & 1];
            fout = L.buf[(step + 1) & 1];
            __syncthreads();  // every warp is done with the previous lattice's constants
            static_assert(sizeof(P) / 4 <= 32 * (R + 2), "one word per thread");
            if (threadIdx.x < sizeof(P) / 4)
                reinterpret_cast<int*>(&P)[threadIdx.x] = reinterpret_cast<const int*>(&L.P)[threadIdx.x];
            __syncthreads();
        }
        if (done) continue;
        const int nx = P.nx, ny = P.ny, y = it.y0 - 1 + warp;
        F2 v[9], rho = F2::c(1.0f), psi = F2::c(0.0f);
        unsigned qw = 0;
        const bool out_row = warp >= 1 && y < it.y1;
        const bool out = out_row && c >= 0 && c < it.w;
        const long long oc = (long long)y * nx + it.x0 + c;
        if (y < it.y1 + 1 && c < it.w + 2) {
            // lattices of the table are at least 8 wide and 4 tall: one wrap each way
            const int yr = wrap_once(y, ny), xa = wrap_once(it.x0 + c, nx);
            const int xl = xa == 0 ? nx - 1 : xa - 1, xr = wrap_once(xa + 2, nx);
            const long long o0 = (long long)yr * nx, om = yr == 0 ? (long long)(ny - 1) * nx : o0 - nx,
                            op = yr == ny - 1 ? 0 : o0 + nx;
            pull_tile<true>(fin, P.pitch, xl, xa, xa + 1, xr, om, o0, op, v);
            if (out) qw = __ldg(reinterpret_cast<const unsigned*>(rest_lo_plane(fin, P.pitch) + oc));
            rho = sum9_v(v);
            psi = pseudo_psi_v(rho, P);
        }
        F2(*s)[32] = s_psi[par];  // two buffers: the next tile's psi may be written before this one's is read
        par ^= 1;
        s[warp][lane] = psi;
        __syncthreads();
        if (!out_row) continue;
        F2 pn[9];
        neighbours(shifted(s[warp - 1][lane]), shifted(psi), shifted(s[warp + 1][lane]), pn);
        tile_collide_pp<-1>(v, rho, pn, F2::c(P.fx), F2::c(P.fy), qw, P, Exchange{});
        if (out) {
#pragma unroll
            for (int j = 0; j < 9; ++j) *reinterpret_cast<float2*>(fout + j * P.pitch + oc) = v[j].v;
            *reinterpret_cast<unsigned*>(rest_lo_plane(fout, P.pitch) + oc) = qw;
        }
    }
}

// Start (by < 0) or advance the tiled lattices' clock: state[0] the steps done, state[1] the tiles of
// the lattices (order: their step counts and tiles) that are not finished by then.
__global__ void batch_clock_kernel(int* state, int by, const int2* __restrict__ order, int n) {
    const int base = by < 0 ? 0 : state[0] + by;
    int tiles = 0;
    for (int i = threadIdx.x; i < n; i += 32) tiles += order[i].x > base ? order[i].y : 0;
    tiles = __reduce_add_sync(0xffffffffu, tiles);
    if (threadIdx.x == 0) {
        state[0] = base;
        state[1] = tiles;
    }
}

// Cells of every lattice in runs of kRunCells, one CTA each (lattice, run of it): the kernels off the step
// path work on these, so that a 512 x 512 lattice does not wait for one CTA (observables of the 96-lattice
// sweep: 1.25 ms with a CTA per lattice, 0.33 with these).
constexpr unsigned kRunCells = 2048;
// The cells of a run, [first, end) of N.  32-bit numbers without sign: a lattice that fits the device has
// less than 2^32 cells (88 bytes each), but may have more than 2^31.
struct Run {
    unsigned N, first, end;
    __device__ __forceinline__ Run(int2 run, int nx, int ny)
        : N((unsigned)nx * (unsigned)ny), first((unsigned)run.y * kRunCells), end(first + min(kRunCells, N - first)) {}
};

// f = f^eq(rho0, u = 0) of every lattice from its initial densities on the device.
__global__ void __launch_bounds__(256)
    batch_init_kernel(const BatchLattice* __restrict__ lats, const int2* __restrict__ runs) {
    const int2 run = runs[blockIdx.x];
    const BatchLattice& L = lats[run.x];
    const int nx = L.P.nx, ny = L.P.ny;
    const Run R(run, nx, ny);
    for (long long c = R.first + threadIdx.x; c < R.end; c += blockDim.x)
        init_cell(L.rho0, L.buf[0], LBM_PSEUDOPOTENTIAL, nx, ny, L.P.pitch, L.P.rest_inv, c);
}

// Observables, the definitions of lbm_observables, in three launches: rho and psi of the final state into
// the lattice scratch; per run the sums and maxima of u (Eq. 6b with the Shan-Chen force), mass and probes;
// per lattice their total in run order, tangent width, pressure jump and equimolar radius.
__global__ void __launch_bounds__(256)
    batch_fields_kernel(const BatchLattice* __restrict__ lats, const int2* __restrict__ runs) {
    const int2 run = runs[blockIdx.x];
    const BatchLattice& L = lats[run.x];
    const StepParams<float> P = L.P;
    const int nx = P.nx, ny = P.ny;
    const Run R(run, nx, ny);
    const float* f = L.buf[L.nsteps & 1];
    float* psi = L.scratch + R.N;
    for (unsigned k = threadIdx.x; k < R.end - R.first; k += blockDim.x) {
        const unsigned c = R.first + k;
        float v[9];
        pull_cell(f, P.pitch, (int)(c % nx), (int)(c / nx), nx, ny, v);
        const float r = sum9_rest(v, rest_lo_plane(f, P.pitch)[c], P);
        L.scratch[c] = r;
        psi[c] = pseudo_psi(r, P);
    }
}

constexpr int kRunSums = 6;  // mass, liquid and vapour probes, bad cells; max u^2, max slope
__global__ void __launch_bounds__(256)
    batch_sums_kernel(const BatchLattice* __restrict__ lats, const int2* __restrict__ runs, double* __restrict__ sums) {
    const int2 run = runs[blockIdx.x];
    const BatchLattice& L = lats[run.x];
    const StepParams<float> P = L.P;
    const int nx = P.nx, ny = P.ny;
    const Run R(run, nx, ny);
    const float* f = L.buf[L.nsteps & 1];
    const float* rho = L.scratch;
    const float* ps = L.scratch + R.N;
    double m = 0.0, u2 = 0.0, bad = 0.0, liq = 0.0, vap = 0.0, dmax = 0.0;
    for (unsigned k = threadIdx.x; k < R.end - R.first; k += blockDim.x) {
        const unsigned c = R.first + k;
        const int x = (int)(c % nx), y = (int)(c / nx);
        float v[9], an[9];
        pull_cell(f, P.pitch, x, y, nx, ny, v);
        gather8(ps, x, y, nx, ny, an);
        const float w1 = 1.0f / 3.0f, w2 = 1.0f / 12.0f;
        const float gx = (an[1] - an[3]) * w1 + ((an[5] - an[7]) + (an[8] - an[6])) * w2;
        const float gy = (an[2] - an[4]) * w1 + ((an[5] - an[7]) + (an[6] - an[8])) * w2;
        const float r = rho[c];
        const float Fx = an[0] * gx + P.fx, Fy = an[0] * gy + P.fy;
        const float jx = (v[1] - v[3]) + (v[5] - v[6]) + (v[8] - v[7]);
        const float jy = (v[2] - v[4]) + (v[5] + v[6]) - (v[7] + v[8]);
        const double ux = (jx + 0.5f * Fx) / r, uy = (jy + 0.5f * Fy) / r;
        const double q = ux * ux + uy * uy;
        if (!(r > 0.0f) || !isfinite(r) || !isfinite(q)) bad += 1.0;
        m += r;
        u2 = fmax(u2, isfinite(q) ? q : 0.0);
        if (L.geometry == 0) {
            if (x == nx / 2 - 1 || x == nx / 2) liq += r;
            if (x == 0 || x == nx - 1) vap += r;
        } else {
            const int cx0 = nx / 2 - 2, cy0 = ny / 2 - 2;
            if (x >= cx0 && x < cx0 + 4 && y >= cy0 && y < cy0 + 4) liq += r;
            if ((x < 4 || x >= nx - 4) && (y < 4 || y >= ny - 4)) vap += r;
        }
        const int prow = L.geometry == 0 ? 0 : ny / 2;
        if (y == prow) {
            const float* row = rho + (size_t)y * nx;
            const double a = row[x == nx - 1 ? 0 : x + 1], b = row[x == 0 ? nx - 1 : x - 1];
            dmax = fmax(dmax, fabs(a - b) * 0.5);
        }
    }
    __shared__ double red[kRunSums][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        m += __shfl_down_sync(0xffffffffu, m, o);
        liq += __shfl_down_sync(0xffffffffu, liq, o);
        vap += __shfl_down_sync(0xffffffffu, vap, o);
        bad += __shfl_down_sync(0xffffffffu, bad, o);
        u2 = fmax(u2, __shfl_down_sync(0xffffffffu, u2, o));
        dmax = fmax(dmax, __shfl_down_sync(0xffffffffu, dmax, o));
    }
    if (lane == 0) {
        red[0][wid] = m;
        red[1][wid] = liq;
        red[2][wid] = vap;
        red[3][wid] = bad;
        red[4][wid] = u2;
        red[5][wid] = dmax;
    }
    __syncthreads();
    if (threadIdx.x < kRunSums) {
        double t = red[threadIdx.x][0];
        for (int w = 1; w < 8; ++w)
            t = threadIdx.x < 4 ? t + red[threadIdx.x][w] : fmax(t, red[threadIdx.x][w]);
        sums[kRunSums * (size_t)blockIdx.x + threadIdx.x] = t;
    }
}

// first[i], first[i + 1]: the runs of lattice i (one warp per lattice).
__global__ void __launch_bounds__(32)
    batch_obs_kernel(const BatchLattice* __restrict__ lats, const int* __restrict__ first,
                     const double* __restrict__ sums, double* __restrict__ out) {
    const BatchLattice& L = lats[blockIdx.x];
    const int nx = L.P.nx, ny = L.P.ny, lane = threadIdx.x;
    const unsigned N = (unsigned)nx * (unsigned)ny;
    double s[kRunSums] = {0, 0, 0, 0, 0, 0};
    for (int r = first[blockIdx.x] + lane; r < first[blockIdx.x + 1]; r += 32)
        for (int j = 0; j < kRunSums; ++j) {
            const double t = sums[kRunSums * (size_t)r + j];
            s[j] = j < 4 ? s[j] + t : fmax(s[j], t);
        }
    for (int o = 16; o > 0; o >>= 1)
        for (int j = 0; j < kRunSums; ++j) {
            const double t = __shfl_xor_sync(0xffffffffu, s[j], o);
            s[j] = j < 4 ? s[j] + t : fmax(s[j], t);
        }
    if (lane == 0) {
        const double nl = L.geometry == 0 ? 2.0 * ny : 16.0, nv = L.geometry == 0 ? 2.0 * ny : 64.0;
        const double rl = s[1] / nl, rv = s[2] / nv;
        auto pcs = [&](double r) {
            const double e = L.b4 * r, om = 1.0 - e;
            return r * L.RT * (1.0 + e + e * e - e * e * e) / (om * om * om) - L.a * r * r;
        };
        double* o = out + 8 * blockIdx.x;
        o[0] = rl;
        o[1] = rv;
        o[2] = (rl - rv) / s[5];
        o[3] = pcs(rl) - pcs(rv);
        o[4] = sqrt(s[4]);
        o[5] = s[0];
        o[6] = L.geometry == 1 ? sqrt(fmax(s[0] - rv * (double)N, 0.0) / (3.14159265358979323846 * (rl - rv))) : nan("");
        o[7] = s[3];
    }
}

}  // namespace lbmk

// --------------------------------------------------------------------------------------
// Host side

namespace {
// Resident lattices that run as one launch on a stream of its own: CTAs of threads x pairs cells.
struct ResidentGroup {
    std::vector<int> ids;  // longest first
    int max_cells;
    bool even;             // even widths
    int pairs, threads;    // chosen by the autotuner
    int* d_ids;
    cudaStream_t stream;
    cudaEvent_t done;
};
}  // namespace

struct lbm_batch {
    int n;
    std::vector<lbm_batch_lattice> spec;
    std::vector<BatchLattice> lat;       // host copy of the device table
    std::vector<ResidentGroup> groups;   // resident lattices by size and parity of the width
    std::vector<BatchItem> items;        // strips, sorted by lattice nsteps, longest first
    std::vector<BatchItem> tiles;        // tiles, in the same order of lattices
    std::vector<int2> order;             // tiled lattices in that order: steps, tiles
    int max_tiled_steps;
    int strip_rows;
    char* pool;
    BatchLattice* d_lat;
    BatchItem* d_items;
    BatchItem* d_tiles;
    int2* d_order;
    int* d_step;
    int* d_err;
    double* d_obs;
    std::vector<double> h_obs;
    cudaStream_t s_tile;
    cudaGraphExec_t chunk[2];            // kChunk steps with strips, with tiles
    bool ran;
    std::vector<int2> runs;                 // cells in runs of kRunCells: lattice, run of it
    int2* d_runs;
    int* d_first;                           // each lattice's first run (n + 1)
    double* d_sums;                         // kRunSums per run
    std::vector<std::vector<double>> rho0;  // initial densities, where the device cannot hold them between runs
    cudaEvent_t ready;                      // the initial state is there (for the resident groups)
};

namespace {

struct TuneKey {
    int kind, a, b;
    bool operator<(const TuneKey& o) const {
        return kind != o.kind ? kind < o.kind : (a != o.a ? a < o.a : b < o.b);
    }
};
std::map<TuneKey, int> g_tune_cache;
std::mutex g_tune_mu;

// f^eq(rho0) for every lattice and the clock at 0, enqueued behind whatever ran before.
int batch_init_state(lbm_batch* b) {
    BCK(cudaMemsetAsync(b->d_err, 0, sizeof(int) * 16, b->s_tile));
    for (size_t i = 0; i < b->rho0.size(); ++i)
        BCK(cudaMemcpyAsync(b->lat[i].rho0, b->rho0[i].data(), sizeof(double) * b->rho0[i].size(),
                            cudaMemcpyHostToDevice, b->s_tile));
    if (b->d_order) lbmk::batch_clock_kernel<<<1, 32, 0, b->s_tile>>>(b->d_step, -1, b->d_order, (int)b->order.size());
    lbmk::batch_init_kernel<<<(unsigned)b->runs.size(), 256, 0, b->s_tile>>>(b->d_lat, b->d_runs);
    BCK(cudaGetLastError());
    BCK(cudaEventRecord(b->ready, b->s_tile));
    for (const ResidentGroup& g : b->groups) BCK(cudaStreamWaitEvent(g.stream, b->ready, 0));
    return LBM_OK;
}

// The runs of all lattices and their initial densities, to the device.
int upload_state(lbm_batch* b, const double* const* rho0) {
    std::vector<int> first;
    for (int i = 0; i < b->n; ++i) {
        const size_t cells = (size_t)b->lat[i].P.nx * b->lat[i].P.ny;
        first.push_back((int)b->runs.size());
        for (size_t c = 0; c < cells; c += lbmk::kRunCells) b->runs.push_back(make_int2(i, (int)(c / lbmk::kRunCells)));
        if (b->rho0.empty())
            BCK(cudaMemcpyAsync(b->lat[i].rho0, rho0[i], sizeof(double) * cells, cudaMemcpyHostToDevice, b->s_tile));
    }
    first.push_back((int)b->runs.size());
    BCK(cudaMalloc(&b->d_runs, sizeof(int2) * b->runs.size()));
    BCK(cudaMalloc(&b->d_first, sizeof(int) * first.size()));
    BCK(cudaMalloc(&b->d_sums, sizeof(double) * lbmk::kRunSums * b->runs.size()));
    BCK(cudaMemcpyAsync(b->d_runs, b->runs.data(), sizeof(int2) * b->runs.size(), cudaMemcpyHostToDevice, b->s_tile));
    BCK(cudaMemcpyAsync(b->d_first, first.data(), sizeof(int) * first.size(), cudaMemcpyHostToDevice, b->s_tile));
    BCK(cudaStreamSynchronize(b->s_tile));  // the caller's arrays have been read
    return LBM_OK;
}

// The resident kernel's forms by pairs per thread; the widest block holds the largest resident lattice.
using ResidentKernel = void (*)(const BatchLattice*, const int*, int);
ResidentKernel resident_kernel(int pairs, bool even, int threads) {
    if (pairs == 1) return even ? lbmk::pp_resident_kernel<1, 512, true> : lbmk::pp_resident_kernel<1, 512, false>;
    if (pairs == 2) return even ? lbmk::pp_resident_kernel<2, 512, true> : lbmk::pp_resident_kernel<2, 512, false>;
    if (threads <= 512)
        return even ? lbmk::pp_resident_kernel<4, 512, true> : lbmk::pp_resident_kernel<4, 512, false>;
    return even ? lbmk::pp_resident_kernel<4, 576, true> : lbmk::pp_resident_kernel<4, 576, false>;
}
// Threads of a CTA whose threads hold `pairs` pairs of a lattice of `cells` cells.
int resident_threads(int cells, int pairs) { return ((cells + 1) / 2 + 32 * pairs - 1) / (32 * pairs) * 32; }

int launch_resident(const lbm_batch* b, const ResidentGroup& g, int step_limit) {
    const ResidentKernel k = resident_kernel(g.pairs, g.even, g.threads);
    // the limit belongs to the kernel, not to this launch: the same for every batch, since a smaller batch on
    // another thread would lower it under this launch
    BCK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)resident_smem(kResidentCells)));
    k<<<(unsigned)g.ids.size(), g.threads, resident_smem(g.max_cells), g.stream>>>(b->d_lat, g.d_ids, step_limit);
    BCK(cudaGetLastError());
    return LBM_OK;
}

// Groups of the resident lattices: CTAs of one launch have the same shared memory and threads, so
// lattices of up to 1152, 2304 and 4608 cells run as separate launches, and odd widths apart.
int build_groups(lbm_batch* b) {
    for (int cls = 0; cls < 6; ++cls) {
        ResidentGroup g{};
        g.even = cls % 2 == 0;
        const int hi = 1152 << cls / 2, lo = cls < 2 ? 0 : hi / 2;
        for (int i = 0; i < b->n; ++i) {
            if (!b->lat[i].resident) continue;
            const int nx = b->lat[i].P.nx, cells = nx * b->lat[i].P.ny;
            if ((nx % 2 == 0) == g.even && cells > lo && cells <= hi) {
                g.ids.push_back(i);
                g.max_cells = std::max(g.max_cells, cells);
            }
        }
        if (g.ids.empty()) continue;
        std::stable_sort(g.ids.begin(), g.ids.end(), [&](int x, int y) {
            return (long long)b->lat[x].nsteps * b->lat[x].P.nx * b->lat[x].P.ny >
                   (long long)b->lat[y].nsteps * b->lat[y].P.nx * b->lat[y].P.ny;
        });
        b->groups.push_back(g);  // (owned by the batch from here on, whatever fails below)
        ResidentGroup& o = b->groups.back();
        BCK(cudaStreamCreateWithFlags(&o.stream, cudaStreamNonBlocking));
        BCK(cudaEventCreateWithFlags(&o.done, cudaEventDisableTiming));
        BCK(cudaMalloc(&o.d_ids, sizeof(int) * o.ids.size()));
        BCK(cudaMemcpyAsync(o.d_ids, o.ids.data(), sizeof(int) * o.ids.size(), cudaMemcpyHostToDevice, b->s_tile));
    }
    return LBM_OK;
}

int launch_tile_step(lbm_batch* b, int k, cudaStream_t s) {
    const int grid = (int)std::min<size_t>(b->tiles.size(), 152 * kTileCtasPerSM);
    lbmk::pp_batch_tile<<<grid, 32 * (lbmk::kBatchTileRows + 2), 0, s>>>(b->d_lat, b->d_tiles, b->d_step, k);
    BCK(cudaGetLastError());
    return LBM_OK;
}

// The strip kernel that addresses every lattice of the batch.
decltype(&lbmk::pp_batch_pair<kBPWarps, kBPStages, true>) strip_kernel(const lbm_batch* b) {
    for (const auto& l : b->lat)
        if (!lbmk::near_buffer(l.P.pitch)) return lbmk::pp_batch_pair<kBPWarps, kBPStages, false>;
    return lbmk::pp_batch_pair<kBPWarps, kBPStages, true>;
}

int launch_tiled_step(lbm_batch* b, int k, cudaStream_t s) {
    if (b->items.empty()) return LBM_OK;
    const auto kernel = strip_kernel(b);
    kernel<<<(unsigned)b->items.size(), (kBPWarps + 1) * 32, sizeof(BPSmem), s>>>(b->d_lat, b->d_items, b->d_step, k,
                                                                                  b->d_err);
    BCK(cudaGetLastError());
    return LBM_OK;
}

// Tiles of every tiled lattice, longest lattice first, and the lattices in that order.
int build_tiles(lbm_batch* b) {
    std::vector<int> ids;
    for (int i = 0; i < b->n; ++i)
        if (!b->lat[i].resident) ids.push_back(i);
    if (ids.empty()) return LBM_OK;
    std::stable_sort(ids.begin(), ids.end(), [&](int x, int y) { return b->lat[x].nsteps > b->lat[y].nsteps; });
    for (int i : ids) {
        const int nx = b->lat[i].P.nx, ny = b->lat[i].P.ny, wb = lbmk::tile_columns<float>(0, nx);
        const size_t first = b->tiles.size();
        for (int y0 = 0; y0 < ny; y0 += lbmk::kBatchTileRows)
            for (int x0 = 0; x0 < nx; x0 += wb)
                b->tiles.push_back(
                    BatchItem{i, x0, std::min(wb, nx - x0), y0, std::min(y0 + lbmk::kBatchTileRows, ny)});
        b->order.push_back(make_int2(b->lat[i].nsteps, (int)(b->tiles.size() - first)));
    }
    const size_t tb = sizeof(BatchItem) * b->tiles.size(), ob = sizeof(int2) * b->order.size();
    BCK(cudaMalloc(&b->d_tiles, tb));
    BCK(cudaMemcpyAsync(b->d_tiles, b->tiles.data(), tb, cudaMemcpyHostToDevice, b->s_tile));
    BCK(cudaMalloc(&b->d_order, ob));
    BCK(cudaMemcpyAsync(b->d_order, b->order.data(), ob, cudaMemcpyHostToDevice, b->s_tile));
    return LBM_OK;
}

// Strip items of every tiled lattice for a given strip height, longest lattice first.
void build_items(lbm_batch* b, int rows) {
    b->items.clear();
    std::vector<int> order;
    for (int i = 0; i < b->n; ++i)
        if (!b->lat[i].resident) order.push_back(i);
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return b->lat[x].nsteps > b->lat[y].nsteps; });
    for (int i : order) {
        const int nx = b->lat[i].P.nx, ny = b->lat[i].P.ny;
        const int r = std::min(rows, ny);
        b->lat[i].P.rows = r;
        // pair strips: nx split into equal widths (multiples of 4, at most kBPTX columns)
        const int gx = (nx + kBPTX - 1) / kBPTX;
        const int wb = lbmk::warp_strip_width(nx, gx);
        for (int y0 = 0; y0 < ny; y0 += r)
            for (int x0 = 0; x0 < nx; x0 += wb)
                b->items.push_back(BatchItem{i, x0, std::min(wb, nx - x0), y0, std::min(y0 + r, ny)});
    }
}

int upload_tables(lbm_batch* b) {
    if (b->d_items) cudaFree(b->d_items);
    b->d_items = nullptr;
    BCK(cudaMemcpyAsync(b->d_lat, b->lat.data(), sizeof(BatchLattice) * b->n, cudaMemcpyHostToDevice, b->s_tile));
    if (!b->items.empty()) {
        BCK(cudaMalloc(&b->d_items, sizeof(BatchItem) * b->items.size()));
        BCK(cudaMemcpyAsync(b->d_items, b->items.data(), sizeof(BatchItem) * b->items.size(), cudaMemcpyHostToDevice,
                            b->s_tile));
    }
    return LBM_OK;
}

double time_ms(cudaStream_t s, const std::function<int()>& fn, int* rc) {
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    *rc = fn();
    cudaEventRecord(e1, s);
    cudaEventSynchronize(e1);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return ms;
}

// Autotuner: pairs of cells per thread of each resident group and tiled strip height.  Each
// candidate runs a short trial on the real initial state (restored afterwards); the choice is
// cached per shape class for the lifetime of the process.
int autotune(lbm_batch* b) {
    for (ResidentGroup& g : b->groups) {
        const TuneKey key{g.even ? 0 : 2, g.max_cells, (int)g.ids.size()};
        int choice = -1;
        {
            std::lock_guard<std::mutex> lk(g_tune_mu);
            auto it = g_tune_cache.find(key);
            if (it != g_tune_cache.end()) choice = it->second;
        }
        if (choice < 0) {
            double best = 1e30;
            for (int pairs : {1, 2, 4}) {
                const int threads = resident_threads(g.max_cells, pairs);
                if (threads > (pairs == 4 ? 576 : 512)) continue;
                g.pairs = pairs;
                g.threads = threads;
                int rc = launch_resident(b, g, 1);  // (loads the kernel)
                if (rc) return rc;
                const double ms = time_ms(g.stream, [&] { return launch_resident(b, g, 64); }, &rc);
                if (rc) return rc;
                if (ms < best) {
                    best = ms;
                    choice = pairs;
                }
            }
            std::lock_guard<std::mutex> lk(g_tune_mu);
            g_tune_cache[key] = choice;
        }
        g.pairs = choice;
        g.threads = resident_threads(g.max_cells, choice);
    }
    if (!b->items.empty() || b->max_tiled_steps > 0) {
        long long cells = 0;
        for (int i = 0; i < b->n; ++i)
            if (!b->lat[i].resident) cells += (long long)b->lat[i].P.nx * b->lat[i].P.ny;
        const TuneKey key{1, (int)std::min<long long>(cells >> 10, 1 << 30), b->n};
        int choice = -1;
        {
            std::lock_guard<std::mutex> g(g_tune_mu);
            auto it = g_tune_cache.find(key);
            if (it != g_tune_cache.end()) choice = it->second;
        }
        if (const char* e = std::getenv("LBM_BATCH_ROWS")) choice = std::max(1, std::atoi(e));  // tuning experiments
        if (choice < 0 && cells < kStripCells) choice = 32;  // the strips will not run
        if (choice < 0) {
            // two passes in opposite orders, 16 steps per trial, best time per candidate:
            // a single short pass in one order favoured whichever candidate ran last
            const int cand[3] = {16, 32, 64};
            double best_ms[3] = {1e30, 1e30, 1e30};
            for (int pass = 0; pass < 2; ++pass)
                for (int j = 0; j < 3; ++j) {
                    const int c = pass == 0 ? j : 2 - j;
                    build_items(b, cand[c]);
                    int rc = upload_tables(b);
                    if (rc) return rc;
                    const double ms = time_ms(b->s_tile, [&] {
                        for (int k = 0; k < 16; ++k) {
                            int r = launch_tiled_step(b, k, b->s_tile);
                            if (r) return r;
                        }
                        return (int)LBM_OK;
                    }, &rc);
                    if (rc) return rc;
                    best_ms[c] = std::min(best_ms[c], ms);
                }
            // the trial sees every lattice active; later, only the longest lattices remain and
            // more (shorter) strips keep the GPU busy: take the shortest strips within 5% of the
            // best trial time
            double best = 1e30;
            for (int c = 0; c < 3; ++c) best = std::min(best, best_ms[c]);
            for (int c = 0; c < 3; ++c)
                if (best_ms[c] <= 1.05 * best) {
                    choice = cand[c];
                    break;
                }
            std::lock_guard<std::mutex> g(g_tune_mu);
            g_tune_cache[key] = choice;
        }
        b->strip_rows = choice;
        build_items(b, choice);
        int rc = upload_tables(b);
        if (rc) return rc;
    }
    return batch_init_state(b);  // trials advanced the state: start again from f^eq(rho0)
}

// kChunk steps of the tiled lattices and the clock step as a graph.
int capture_chunk(lbm_batch* b, bool strips, cudaGraphExec_t* out) {
    cudaGraph_t g = nullptr;
    BCK(cudaStreamBeginCapture(b->s_tile, cudaStreamCaptureModeThreadLocal));
    int rc = LBM_OK;
    for (int k = 0; k < kChunk && rc == LBM_OK; ++k)
        rc = strips ? launch_tiled_step(b, k, b->s_tile) : launch_tile_step(b, k, b->s_tile);
    if (rc == LBM_OK)
        lbmk::batch_clock_kernel<<<1, 32, 0, b->s_tile>>>(b->d_step, kChunk, b->d_order, (int)b->order.size());
    cudaError_t e = cudaStreamEndCapture(b->s_tile, &g);
    if (rc) {
        if (g) cudaGraphDestroy(g);
        return rc;
    }
    if (e != cudaSuccess) return bfail(e, "cudaStreamEndCapture(batch)");
    e = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) return bfail(e, "cudaGraphInstantiate(batch)");
    return LBM_OK;
}

}  // namespace

extern "C" const char* lbm_batch_last_error(void) { return g_batch_msg; }

extern "C" void lbm_batch_destroy(lbm_batch* b) {
    if (!b) return;
    for (ResidentGroup& g : b->groups) {
        if (g.stream) cudaStreamSynchronize(g.stream);
        if (g.d_ids) cudaFree(g.d_ids);
        if (g.done) cudaEventDestroy(g.done);
        if (g.stream) cudaStreamDestroy(g.stream);
    }
    cudaStreamSynchronize(b->s_tile);
    for (cudaGraphExec_t g : b->chunk)
        if (g) cudaGraphExecDestroy(g);
    if (b->d_items) cudaFree(b->d_items);
    if (b->d_tiles) cudaFree(b->d_tiles);
    if (b->d_runs) cudaFree(b->d_runs);
    if (b->d_first) cudaFree(b->d_first);
    if (b->d_sums) cudaFree(b->d_sums);
    if (b->ready) cudaEventDestroy(b->ready);
    if (b->d_order) cudaFree(b->d_order);
    if (b->pool) cudaFree(b->pool);
    if (b->s_tile) cudaStreamDestroy(b->s_tile);
    delete b;
}

extern "C" int lbm_batch_create(int n, const lbm_batch_lattice* specs, const double* const* rho0, lbm_batch** out) {
    if (!out) return LBM_ERR_ARG;
    *out = nullptr;
    if (n < 1 || !specs || !rho0) return LBM_ERR_ARG;
    lbm_batch* b = new (std::nothrow) lbm_batch();
    if (!b) return LBM_ERR_ARG;
    b->n = n;
    b->spec.assign(specs, specs + n);
    b->lat.resize(n);
    // resolve parameters and validate on the host first
    std::vector<size_t> offs(n);
    b->max_tiled_steps = 0;
    std::vector<lbm_params> in_p(n), res_p(n);
    std::vector<lbm_thermo> res_t(n);
    std::vector<int> res_rc(n);
    for (int i = 0; i < n; ++i) in_p[i] = specs[i].params;
    lbm_resolve_params_many(n, in_p.data(), res_p.data(), res_t.data(), res_rc.data());
    for (int i = 0; i < n; ++i) {
        const lbm_batch_lattice& s = specs[i];
        if (s.nx < 1 || s.ny < 1 || s.nsteps < 0 || s.nsteps > (1LL << 30) || (s.geometry != 0 && s.geometry != 1) ||
            !rho0[i]) {
            delete b;
            return LBM_ERR_ARG;
        }
        if (s.params.model != LBM_PSEUDOPOTENTIAL || s.params.precision != LBM_F32) {
            delete b;
            return LBM_ERR_UNSUPPORTED;
        }
        const lbm_params& rp = res_p[i];
        const lbm_thermo& th = res_t[i];
        int rc = res_rc[i];
        if (rc) {
            delete b;
            return rc;
        }
        const size_t N = (size_t)s.nx * s.ny;
        for (size_t k = 0; k < N; ++k)
            if (!(rho0[i][k] > 0.0 && rho0[i][k] < 4.0 / rp.b)) {
                delete b;
                return LBM_ERR_ARG;
            }
        BatchLattice& L = b->lat[i];
        std::memset(&L, 0, sizeof(L));
        lbmk::StepParams<float>& P = L.P;
        P.nx = s.nx;
        P.ny = s.ny;
        P.pitch = ((long long)N + 63) / 64 * 64;
        P.rows = std::min(32, s.ny);
        const double G = -1.0, C1 = 5.0 / 6.0 * (rp.kappa_P - 1.0), C2 = 0.5 * (1.0 - rp.kappa_P);
        P.RT = (float)(rp.R * th.T);
        P.a = (float)rp.a;
        P.b4 = (float)(0.25 * rp.b);
        P.kA = (float)(G * (C1 - C2 / 3.0));
        P.kB = (float)(G * (C2 + 0.5 * rp.kappa_Li));
        P.li = (float)(12.0 * rp.kappa_P * rp.sigma_Li);
        P.s_e = (float)(1.0 / rp.tau_e);
        P.s_z = (float)(1.0 / rp.tau_zeta);
        P.s_q = (float)(1.0 / rp.tau_q);
        P.s_nu = (float)(1.0 / rp.tau_nu);
        P.fx = (float)rp.body_fx;
        P.fy = (float)rp.body_fy;
        P.rest_unit = (float)lbm_host::rest_unit(rp.b);
        P.rest_inv = (float)lbm_host::rest_inv(rp.b);
        P.h_e = (float)(1.0 - 0.5 / rp.tau_e);
        P.h_z = (float)(1.0 - 0.5 / rp.tau_zeta);
        P.h_q = (float)(1.0 - 0.5 / rp.tau_q);
        P.h_nu = (float)(1.0 - 0.5 / rp.tau_nu);
        P.h6_e = (float)(6.0 * (1.0 - 0.5 / rp.tau_e));
        P.h6_z = (float)(6.0 * (1.0 - 0.5 / rp.tau_zeta));
        L.RT = rp.R * th.T;
        L.a = rp.a;
        L.b4 = 0.25 * rp.b;
        L.nsteps = (int)s.nsteps;
        L.geometry = s.geometry;
        L.resident = resident_bytes(N) <= kResidentSmemMax;
        if (!L.resident && (s.nx % 4 != 0 || s.nx < 8 || s.ny < 4)) {
            delete b;
            return LBM_ERR_UNSUPPORTED;  // tiled lattices use the TMA strip kernels
        }
        if (!L.resident) b->max_tiled_steps = std::max(b->max_tiled_steps, L.nsteps);
    }
    // Two buffers, the scratch and the initial densities of every lattice; where the device has no room for
    // the last (8 of 96 bytes per cell), they stay on the host and go to the scratch before each run.
    size_t tail = 0;
    auto allocate = [&](bool keep_rho0) {
        size_t bytes = 0;
        for (int i = 0; i < n; ++i) {
            const size_t N = (size_t)specs[i].nx * specs[i].ny;
            offs[i] = bytes;
            bytes += 2 * buffer_bytes(b->lat[i].P.pitch) + a256(2 * N * 4 + (keep_rho0 ? 8 * N : 0));
        }
        tail = bytes;
        bytes += a256(sizeof(BatchLattice) * n) + 256 + 256 + a256(8 * sizeof(double) * n);
        return cudaMalloc(&b->pool, bytes);
    };
    cudaError_t e = allocate(true);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();  // (not an error of the calls below)
        try {
            for (int i = 0; i < n; ++i) b->rho0.emplace_back(rho0[i], rho0[i] + (size_t)specs[i].nx * specs[i].ny);
            e = allocate(false);
        } catch (const std::bad_alloc&) {  // no room on the host either: the device's error stands
        }
    }
    if (e != cudaSuccess) {
        delete b;
        return bfail(e, "cudaMalloc(batch pool)");
    }
    for (int i = 0; i < n; ++i) {
        BatchLattice& L = b->lat[i];
        const size_t fb = buffer_bytes(L.P.pitch);
        L.buf[0] = reinterpret_cast<float*>(b->pool + offs[i]);
        L.buf[1] = reinterpret_cast<float*>(b->pool + offs[i] + fb);
        L.scratch = reinterpret_cast<float*>(b->pool + offs[i] + 2 * fb);
        L.rho0 = reinterpret_cast<double*>(L.scratch + (b->rho0.empty() ? 2 * (size_t)L.P.nx * L.P.ny : 0));
    }
    b->d_lat = reinterpret_cast<BatchLattice*>(b->pool + tail);
    b->d_step = reinterpret_cast<int*>(b->pool + tail + a256(sizeof(BatchLattice) * n));
    b->d_err = reinterpret_cast<int*>(reinterpret_cast<char*>(b->d_step) + 256);
    b->d_obs = reinterpret_cast<double*>(reinterpret_cast<char*>(b->d_err) + 256);
    b->h_obs.assign(8 * (size_t)n, 0.0);
    int rc = LBM_OK;
    auto fail = [&](int code) {
        lbm_batch_destroy(b);
        return code;
    };
    if ((e = cudaStreamCreateWithFlags(&b->s_tile, cudaStreamNonBlocking)) != cudaSuccess ||
        (e = cudaEventCreateWithFlags(&b->ready, cudaEventDisableTiming)) != cudaSuccess)
        return fail(bfail(e, "stream/event create"));
    if ((rc = build_groups(b))) return fail(rc);
    if ((e = cudaFuncSetAttribute(strip_kernel(b), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(BPSmem))) != cudaSuccess)
        return fail(bfail(e, "cudaFuncSetAttribute(batch strip smem)"));
    if ((rc = build_tiles(b))) return fail(rc);
    build_items(b, 32);
    if ((rc = upload_tables(b))) return fail(rc);
    if ((rc = upload_state(b, rho0))) return fail(rc);
    if ((rc = batch_init_state(b))) return fail(rc);
    if ((rc = autotune(b))) return fail(rc);
    *out = b;
    return LBM_OK;
}

static int run_batch(lbm_batch* b) {
    if (b->ran) {
        int rc = batch_init_state(b);
        if (rc) return rc;
    }
    b->ran = true;
    // resident lattices: one persistent launch per group, concurrent with the tiled replays
    int rc = LBM_OK;
    for (const ResidentGroup& g : b->groups)
        if ((rc = launch_resident(b, g, -1))) return rc;
    // tiled lattices: replays of a captured chunk of single-step launches and a clock step; strips
    // while the unfinished lattices hold enough cells for them, then tiles
    for (int s = 0; s < b->max_tiled_steps; s += kChunk) {
        long long cells = 0;
        for (int i = 0; i < b->n; ++i)
            if (!b->lat[i].resident && b->lat[i].nsteps > s) cells += (long long)b->lat[i].P.nx * b->lat[i].P.ny;
        cudaGraphExec_t& g = b->chunk[cells >= kStripCells ? 0 : 1];
        if (!g && (rc = capture_chunk(b, cells >= kStripCells, &g))) return rc;
        BCK(cudaGraphLaunch(g, b->s_tile));
    }
    for (const ResidentGroup& g : b->groups) {
        BCK(cudaEventRecord(g.done, g.stream));
        BCK(cudaStreamWaitEvent(b->s_tile, g.done, 0));
    }
    return LBM_OK;
}

extern "C" int lbm_batch_run(lbm_batch* b) {
    if (!b) return LBM_ERR_ARG;
    const int rc = run_batch(b);
    // after a failure on the way the groups already launched are not joined to s_tile: a further run's initial
    // state must not be written before they have stored their last
    if (rc)
        for (const ResidentGroup& g : b->groups) cudaStreamSynchronize(g.stream);
    return rc;
}

extern "C" int lbm_batch_observables(lbm_batch* b, lbm_obs* out) {
    if (!b || !out) return LBM_ERR_ARG;
    if (!b->ran) return LBM_ERR_STATE;
    const unsigned runs = (unsigned)b->runs.size();
    lbmk::batch_fields_kernel<<<runs, 256, 0, b->s_tile>>>(b->d_lat, b->d_runs);
    lbmk::batch_sums_kernel<<<runs, 256, 0, b->s_tile>>>(b->d_lat, b->d_runs, b->d_sums);
    lbmk::batch_obs_kernel<<<b->n, 32, 0, b->s_tile>>>(b->d_lat, b->d_first, b->d_sums, b->d_obs);
    BCK(cudaGetLastError());
    BCK(cudaMemcpyAsync(b->h_obs.data(), b->d_obs, sizeof(double) * 8 * b->n, cudaMemcpyDeviceToHost, b->s_tile));
    int herr = 0;
    BCK(cudaMemcpyAsync(&herr, b->d_err, sizeof(int), cudaMemcpyDeviceToHost, b->s_tile));
    BCK(cudaStreamSynchronize(b->s_tile));
    for (int i = 0; i < b->n; ++i) {
        const double* h = &b->h_obs[8 * (size_t)i];
        lbm_obs& o = out[i];
        o.rho_l = h[0];
        o.rho_v = h[1];
        o.width = h[2];
        o.dp = h[3];
        o.u_max = h[4];
        o.mass = h[5];
        o.radius = h[6];
        o.step = b->ran ? b->lat[i].nsteps : 0;
        o.pad_ = 0;
        o.status = herr ? LBM_ERR_TIMEOUT : ((h[7] != 0.0 || !std::isfinite(h[5])) ? LBM_ERR_DIVERGED : LBM_OK);
    }
    return LBM_OK;
}

extern "C" int lbm_batch_populations(lbm_batch* b, int i, double* f) {
    if (!b || !f || i < 0 || i >= b->n) return LBM_ERR_ARG;
    if (!b->ran) return LBM_ERR_STATE;
    BCK(cudaStreamSynchronize(b->s_tile));  // (the resident groups have been joined to it)
    const BatchLattice& L = b->lat[i];
    const int nx = L.P.nx, ny = L.P.ny;
    const size_t n = (size_t)nx * ny;
    std::vector<float> plane(n);
    const float* src = L.buf[b->ran ? (L.nsteps & 1) : 0];
    static const int cxs[9] = {0, 1, 0, -1, 0, 1, -1, -1, 1}, cys[9] = {0, 0, 1, 0, -1, 1, 1, -1, -1};
    for (int q = 0; q < 9; ++q) {
        BCK(cudaMemcpy(plane.data(), src + q * L.P.pitch, n * sizeof(float), cudaMemcpyDeviceToHost));
        for (int y = 0; y < ny; ++y)
            for (int x = 0; x < nx; ++x) {
                const int xs = (x + cxs[q] + nx) % nx, ys = (y + cys[q] + ny) % ny;  // f_i(x + c_i) = S_i(x)
                f[q * n + (size_t)ys * nx + xs] = plane[(size_t)y * nx + x];
            }
    }
    std::vector<short> ext(n);  // the rest population's extension (plane 9)
    BCK(cudaMemcpy(ext.data(), reinterpret_cast<const char*>(src + 9 * L.P.pitch), n * sizeof(short),
                   cudaMemcpyDeviceToHost));
    for (size_t k = 0; k < n; ++k) f[k] = lbm_host::rest_decode((float)f[k], ext[k], (double)L.P.rest_unit);
    return LBM_OK;
}

extern "C" int lbm_batch_info(const lbm_batch* b, int* n_resident, int* n_items, int* resident_threads,
                              int* strip_rows) {
    if (!b) return LBM_ERR_ARG;
    int resident = 0, threads = 0;
    for (const ResidentGroup& g : b->groups) {
        resident += (int)g.ids.size();
        threads = g.threads;  // (of the largest lattices)
    }
    if (n_resident) *n_resident = resident;
    if (n_items) *n_items = (int)b->items.size();
    if (resident_threads) *resident_threads = threads;
    if (strip_rows) *strip_rows = b->strip_rows;
    return LBM_OK;
}

extern "C" void* lbm_batch_stream(const lbm_batch* b) { return b ? static_cast<void*>(b->s_tile) : nullptr; }
