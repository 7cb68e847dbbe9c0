// step_tile.cuh -- the step of every lattice that the TMA strip kernels do not serve: FP64, FP32
// lattices whose width is not a multiple of 4 or that are too small for strips, no-slip walls, the
// droplet-collision drive and the full free-energy model.
//
// A CTA updates a tile of a few rows and one warp's columns.  Each warp holds one row
// of the tile or of its halo; a lane holds two adjacent cells in FP32 (packed, F2) or one in FP64.
// A warp pulls its row's populations once and keeps them in registers; the neighbour fields (psi;
// rho and mu; rho, mu and u) go through shared memory between rows and through shuffles within a
// row, one CTA barrier per field.  So the chain from the first load to the last store is one row's
// work whatever the lattice, where a CTA that walks down a strip pays it once per row.
//
// What bounds it (GB300).  FP64: the FP64 pipe, 64 cycles per warp instruction on each of the 608
// sub-partitions whatever the number of active lanes, so the arithmetic below is written for few
// operations (step64.cuh) and the tile height spreads the rows over the sub-partitions
// (choose_tile_rows in lbm_api.cu).  FP32 on small lattices: the latency of one row's chain plus a
// launch; on lattices that fill the GPU: instruction issue.
//
// Per-cell FP32 arithmetic is that of the strip kernels (lbm_kernels.cuh, step_iwb_pair.cuh) on
// the same packed type, so both routes give the same bits.
//
// Walls (rows 0 and ny-1; see step_ext.cuh): halo rows beyond a wall are the mirrored rows; a wall
// row's populations get the first fill when they are pulled and the final fill (J = -F/2) before
// the collision (full model: before u).  band > 0 updates only the rows next to each wall (grid.y = 2).
#pragma once
#include <cuda_runtime.h>

#include "lbm_kernels.cuh"
#include "step64.cuh"
#include "step_ext.cuh"
#include "step_iwb_pair.cuh"
#include "step_pair.cuh"

namespace lbmk {

// Lane layout of a tile row: V the cells of a lane, kPer of them; HC halo columns on each side of
// the (at most) kCols columns a warp updates; kRows the most rows of a tile.  MODEL: 0 pseudopotential, 1
// free energy, 2 full free energy; LV is its number of halo rows.  kCtas: CTAs per SM that the registers
// have to allow (56 and 64 registers in FP32; with one CTA less a 2048^2 step, which streams from HBM,
// took 73.6 us instead of 66.6 and 99.0 instead of 85.4; 72 in FP64 for the full model's periodic step,
// 256 x 128 of which took 32 us with 76).
template <typename real, int MODEL>
struct Tile {
    using V = typename std::conditional<std::is_same<real, float>::value, F2, double>::type;
    static constexpr int kPer = std::is_same<real, float>::value ? 2 : 1;
    static constexpr int LV = MODEL + 1;
    static constexpr int HC = kPer == 1 ? LV : (MODEL == 2 ? 4 : 2);
    static constexpr int kCols = 32 * kPer - 2 * HC;
    static constexpr int kRows = kPer == 2 && MODEL < 2 ? 4 : 8;
    // FP64: a tile of at most kShared rows may have each row's collision done by two warps
    static constexpr int kShared = kPer == 1 && MODEL < 2 ? 2 : 0;
    static constexpr int kThreads = 32 * (kRows + 2 * LV + (kShared > LV ? kShared - LV : 0));
    static constexpr int kCtas = kPer == 1 ? (MODEL == 2 ? 2 : 1) : MODEL == 0 ? 6 : MODEL == 1 ? 4 : 2;
};

// The stored mass of driven steps: fixed-point numbers added atomically to kDriveParts 64-bit accumulators
// (FP64: pairs of them, the low 26 bits of every number to one and the rest to the other, so that a cell keeps
// its bits however many cells there are).  Integer sums are exact in any order and cost no FP64 instructions
// but the mean's (FP32: with FP64 sums per row a 1024^2 step took 38 us, with these 20 us; FP64: with sums per
// row that every CTA added up 200 x 100 took 12.0 us, with these 10.1).  Three sets of accumulators take turns:
// a step reads the set of the step before, adds to its own and zeroes the next one's.  With 2^e the power of
// two above the EOS packing limit, the range is 2^(e + 3) and the unit 2^(e - 55) in FP64, 2^(e - 39)
// (rest_unit) in FP32 up to 2^21 cells and 2^21 / N of the cells' precision beyond, where the total needs the
// bits.  So the mean is within half a unit and the roundings of its scaling of the mean of the densities as
// the step sums them, in flat phases too, whose cells all round alike; in FP32 up to 2^21 cells a density
// above 2^(e - 15) is exact.  A cell whose mass is not a number of that range (a diverged lattice) is counted
// in a third word and makes the mean NaN, as a sum in floating point would.
constexpr int kMassLow = 26;      // bits of the low accumulators' numbers
constexpr int kMassBits = 55;     // FP64: the unit is 2^(e - kMassBits)
constexpr int kMassHeadroom = 3;  // the range is 2^(e + kMassHeadroom): 2^31 cells' total >> kMassLow has 63 bits
constexpr int kDriveSet = 3 * kDriveParts;  // low (FP32: all), high, warps with a cell out of range
// s in units of 2^(base - 1075), rounded to nearest: the bits of s shifted as an integer; false out of range
__device__ __forceinline__ bool mass_fixed(double s, int base, long long& out) {
    const long long b = __double_as_longlong(s);
    const int r = 10 + base - ((__double2hiint(s) >> 20) & 0x7ff);
    const unsigned long long m = ((unsigned long long)b & 0xfffffffffffffull) | 0x10000000000000ull;
    const long long k = r > 63 ? 0ll : (long long)(((m << 10) + (1ull << max(r - 1, 0))) >> max(r, 0));
    out = b < 0 ? -k : k;
    return r >= 10 - (kMassBits + kMassHeadroom - 53);
}

// (hi 2^kMassLow + lo) unit: the total's leading 63 bits, one conversion and one product (each a rounding)
__device__ __forceinline__ double mass_mean(long long hi, unsigned long long lo, double unit) {
    hi += (long long)(lo >> kMassLow);
    const unsigned low = (unsigned)lo & ((1 << kMassLow) - 1);
    const int drop = max(0, kMassLow + 1 - __clzll(hi));  // bits beyond the 63
    const long long t = (long long)((unsigned long long)hi << (kMassLow - drop)) + (low >> drop);
    const double m = (double)t * unit;
    return t == 0 ? 0.0 : __hiloint2double(__double2hiint(m) + (drop << 20), __double2loint(m));
}

// What a tile step takes besides StepParams: the full model's terms, the walls' solved J_y, and the
// drive: the state's mass is the sum of D.parts or of the accumulators acc_in.
template <typename real>
struct TileArgs {
    int wb;    // columns per tile
    int rows;  // rows per tile (band: of the band)
    int band;  // > 0: only the rows next to each wall
    int share;  // two warps per row's collision (rows <= Tile::kShared)
    Ext<real> E;
    real fyg, dpg;  // fy + rho_g g (the force is fyg - rho g) and d_y p_g = rho_g g
    const real* wjy;
    bool driven;
    Drive<real> D;
    double mass_unit;  // the accumulators' unit as a mean density
    float mass_scale, mass_range;  // FP32: 1 / unit, and the range in units
    int mass_base;     // FP64: mass_fixed's
    const unsigned long long* acc_in;
    unsigned long long *acc_out, *acc_zero;
};

template <class V>
__device__ __forceinline__ V cst(double x) {
    if constexpr (std::is_same<V, double>::value)
        return x;
    else
        return V::c((float)x);
}
__device__ __forceinline__ F2 abs_v(F2 a) { return F2(fabsf(a.v.x), fabsf(a.v.y)); }

// FP32: the strip kernels' arithmetic (step64.cuh has the FP64 overloads)
__device__ __forceinline__ F2 tile_psi(F2 rho, const StepParams<float>& P) { return pseudo_psi_v(rho, P); }
__device__ __forceinline__ F2 tile_mu(F2 rho, const F2 n[9], const StepParams<float>& P, const LogTable&) {
    return fe_mu_v(rho, n, P);
}
template <int>
__device__ __forceinline__ void tile_collide_pp(F2 v[9], F2 rho, const F2 pn[9], F2 fx, F2, unsigned& qw,
                                                const StepParams<float>& P, const Exchange&) {
    F2 d0;
    pp_collide_fx_v<F2, true>(v, rho, pn[0], pn, fx, P, &d0);
    qw = rest_update_pair(v[0], qw, d0, P);
}
template <int>
__device__ __forceinline__ void tile_collide_fe(F2 v[9], F2 rho, const F2 mn[9], const F2 rn[9], F2 fx, F2 fy,
                                                unsigned& qw, const StepParams<float>& P, const Exchange&) {
    F2 d0;
    fe_collide_f_v<F2, true>(v, rho, mn, rn, fx, fy, P, &d0);
    qw = rest_update_pair(v[0], qw, d0, P);
}
__device__ __forceinline__ void tile_velocity(const F2 v[9], F2 rho, const F2 mn[9], F2 fx, F2 fy, F2& ux, F2& uy,
                                              F2& Fx, F2& Fy) {
    fe_velocity_v(v, rho, mn, fx, fy, ux, uy, Fx, Fy);
}
__device__ __forceinline__ void tile_collide_iwb(F2 v[9], F2 rho, const F2 rn[9], const F2 un[9], const F2 wn[9],
                                                 F2 ux, F2 uy, F2 Fx, F2 Fy, float pg, float dpg, float A,
                                                 unsigned& qw, const StepParams<float>& P) {
    F2 d0;
    fe_collide_iwb_u_v<F2, true>(v, rho, rn, strain_v(un, wn), ux, uy, Fx, Fy, F2::c(pg), dpg, A, P, &d0);
    qw = rest_update_pair(v[0], qw, d0, P);
}

// A row of a field with its x-shifted values (Row2 of step_pair.cuh, for either type).
template <class V>
struct Row {
    V c, xm, xp;
};
__device__ __forceinline__ Row<F2> shifted(F2 c) {
    const Row2 r = with_shifted(c);
    return {r.c, r.xm, r.xp};
}
__device__ __forceinline__ Row<double> shifted(double c) {
    return {c, __shfl_up_sync(0xffffffffu, c, 1), __shfl_down_sync(0xffffffffu, c, 1)};
}
template <class V>
__device__ __forceinline__ void neighbours(const Row<V>& ym, const Row<V>& y0, const Row<V>& yp, V n[9]) {
    n[0] = y0.c;
    n[1] = y0.xp;
    n[2] = yp.c;
    n[3] = y0.xm;
    n[4] = ym.c;
    n[5] = yp.xp;
    n[6] = yp.xm;
    n[7] = ym.xm;
    n[8] = ym.xp;
}

// Pulled populations of a lane's cells from global memory; om, o0, op: offsets of rows y-1, y, y+1;
// xl, xa, xb, xr: wrapped columns of the cell before, the lane's cells (one in FP64: xb unused) and
// the cell after.  EVEN: nx is even, so a lane's two cells are 8-byte aligned.
template <bool EVEN>
__device__ __forceinline__ void pull_tile(const float* __restrict__ f, long long pitch, int xl, int xa, int xb, int xr,
                                          long long om, long long o0, long long op, F2 v[9]) {
    auto pair = [](const float* p, int a, int b) {
        if constexpr (EVEN)
            return F2(__ldg(reinterpret_cast<const float2*>(p + a)));
        else
            return F2(__ldg(p + a), __ldg(p + b));
    };
    auto two = [](const float* p, int a, int b) { return F2(__ldg(p + a), __ldg(p + b)); };
    v[0] = pair(f + o0, xa, xb);
    v[1] = two(f + 1 * pitch + o0, xl, xa);
    v[2] = pair(f + 2 * pitch + om, xa, xb);
    v[3] = two(f + 3 * pitch + o0, xb, xr);
    v[4] = pair(f + 4 * pitch + op, xa, xb);
    v[5] = two(f + 5 * pitch + om, xl, xa);
    v[6] = two(f + 6 * pitch + om, xb, xr);
    v[7] = two(f + 7 * pitch + op, xb, xr);
    v[8] = two(f + 8 * pitch + op, xl, xa);
}
template <bool EVEN>
__device__ __forceinline__ void pull_tile(const double* __restrict__ f, long long pitch, int xl, int xa, int, int xr,
                                          long long om, long long o0, long long op, double v[9]) {
    pull9(f, pitch, xa, xl, xr, om, o0, op, v);
}

// The same for a buffer of less than 4 GB and even nx, by 32-bit byte offsets from its start: o0, om, op of
// column xa in rows y, y-1, y+1, l and r of the neighbours left and right of the pair (-4 and 8 away from the
// edges), pb the plane pitch.  One integer addition per plane instead of 64-bit address arithmetic per load.
__device__ __forceinline__ void pull_tile32(const float* __restrict__ f, unsigned pb, unsigned o0, unsigned om,
                                            unsigned op, int l, int r, F2 v[9]) {
    const char* b = reinterpret_cast<const char*>(f);
    auto one = [&](unsigned o) { return __ldg(reinterpret_cast<const float*>(b + o)); };
    auto pair = [&](unsigned o) { return F2(__ldg(reinterpret_cast<const float2*>(b + o))); };
    const unsigned a1 = o0 + pb, a3 = o0 + 3 * pb, a5 = om + 5 * pb, a6 = om + 6 * pb, a7 = op + 7 * pb,
                   a8 = op + 8 * pb;
    v[0] = pair(o0);
    v[2] = pair(om + 2 * pb);
    v[4] = pair(op + 4 * pb);
    v[1] = F2(one(a1 + l), one(a1));
    v[5] = F2(one(a5 + l), one(a5));
    v[8] = F2(one(a8 + l), one(a8));
    v[3] = F2(one(a3 + 4), one(a3 + r));
    v[6] = F2(one(a6 + 4), one(a6 + r));
    v[7] = F2(one(a7 + 4), one(a7 + r));
}

// Zou-He completion of a wall row's cells (wall_fill of step_ext.cuh).
template <class V>
__device__ __forceinline__ void tile_wall_fill(V v[9], bool top, V Jx, V Jy) {
    const V h = cst<V>(0.5) * (v[1] - v[3]);
    const V hx = cst<V>(0.5) * Jx, sy = Jy * cst<V>(1.0 / 6.0), ty = Jy * cst<V>(2.0 / 3.0);
    if (!top) {
        v[2] = v[4] + ty;
        v[5] = (v[7] - h) + (hx + sy);
        v[6] = (v[8] + h) - (hx - sy);
    } else {
        v[4] = v[2] - ty;
        v[7] = (v[5] + h) - (hx + sy);
        v[8] = (v[6] - h) + (hx - sy);
    }
}
// x component of the Eq. (24) gradient
template <class V>
__device__ __forceinline__ V tile_grad_x(const V n[9]) {
    return fmav(n[1] - n[3], cst<V>(1.0 / 3.0), ((n[5] - n[7]) + (n[8] - n[6])) * cst<V>(1.0 / 12.0));
}
// wall-normal gradient of the one-sided reading (wall_grad_y_onesided)
template <class V>
__device__ __forceinline__ V tile_grad_y_onesided(const V n[9], bool top) {
    const V a = cst<V>(2.0 / 3.0), d = cst<V>(1.0 / 6.0);
    if (!top) return fmav(a, n[2] - n[0], d * ((n[5] - n[1]) + (n[6] - n[3])));
    return -fmav(a, n[4] - n[0], d * ((n[8] - n[1]) + (n[7] - n[3])));
}

// EVEN: FP32 with even nx (cells of a lane 8-byte aligned); NEAR: and a buffer of less than 4 GB.  SHARE: FP64,
// a tile of at most kShared rows, two warps per row's collision.
template <typename real, int MODEL, bool WALLS, bool DRIVE, bool EVEN, bool NEAR, bool SHARE>
__global__ void __launch_bounds__(Tile<real, MODEL>::kThreads,
                                  std::is_same<real, double>::value && (WALLS || DRIVE) ? 1 : Tile<real, MODEL>::kCtas)
    tile_step(const real* __restrict__ fin, real* __restrict__ fout, const StepParams<real> P,
              const TileArgs<real> T) {
    using L = Tile<real, MODEL>;
    using V = typename L::V;
    constexpr int LV = L::LV, HC = L::HC, KP = L::kPer, RMAX = L::kRows + 2 * LV;
    __shared__ V s_a[RMAX][32];                        // psi or rho
    __shared__ V s_mu[MODEL > 0 ? RMAX : 1][32];       // mu
    __shared__ V s_u[MODEL > 1 ? 2 * RMAX : 1][32];    // u_x, then u_y
    __shared__ real s_rave;
    __shared__ double s_v[SHARE ? L::kShared : 1][10][32], s_x[SHARE ? L::kShared : 1][5][32];
    const int nx = P.nx, ny = P.ny;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows = SHARE ? T.rows : (int)(blockDim.x >> 5) - 2 * LV, nwarps = rows + 2 * LV;  // warps with a row
    const int by = blockIdx.y + gridDim.y * blockIdx.z;  // more than 65535 tiles in y use z
    const int y0 = WALLS && T.band > 0 ? (by == 0 ? 0 : ny - T.band) : by * rows;
    if (y0 >= ny) return;
    const int y1 = WALLS && T.band > 0 ? y0 + T.band : min(y0 + rows, ny);
    const int x0 = blockIdx.x * T.wb;
    const int w = min(T.wb, nx - x0);  // > 0 (the host's grid)
    int y = y0 - LV + warp;            // this warp's row (rows beyond the lattice mirrored or wrapped)
    const int yr = WALLS ? mirror_row(y, ny) : ny >= 16 ? wrap_once(y, ny) : wrap_idx(y, ny);
    bool wall = WALLS && (y == 0 || y == ny - 1);            // a wall row of the lattice or its image
    const bool wall_img = WALLS && (yr == 0 || yr == ny - 1);
    bool top = WALLS && yr != 0;
    const int c = KP * lane - HC;  // first column of the lane, from x0
    bool out_row = warp >= LV && y < y1;
    bool out_a = out_row && c >= 0 && c < w;
    const bool out_b = KP == 2 && out_row && c >= 0 && c + 1 < w;
    // the lane's place in a plane (out rows and lanes only), and with NEAR in bytes in the rest plane
    long long oc = NEAR ? 0 : (long long)y * nx + x0 + c;
    const unsigned oc32 = NEAR ? (unsigned)(y * nx + x0 + c) * 4u : 0u, qo = (unsigned)P.pitch * 36u + oc32 / 2;

    // the state's mean density: every CTA sums in the same order
    if constexpr (DRIVE) {
        if (warp == 0) {
            double m;
            if (T.acc_in) {
                unsigned long long lo = T.acc_in[lane], hi = KP == 1 ? T.acc_in[kDriveParts + lane] : 0ull;
                const bool bad = __any_sync(0xffffffffu, T.acc_in[2 * kDriveParts + lane] != 0);
                for (int o = 16; o > 0; o >>= 1) {
                    lo += __shfl_xor_sync(0xffffffffu, lo, o);
                    if (KP == 1) hi += __shfl_xor_sync(0xffffffffu, hi, o);
                }
                m = KP == 1 ? mass_mean((long long)hi, lo, T.mass_unit) : (double)(long long)lo * T.mass_unit;
                if (bad) m = __longlong_as_double(-1ll);  // NaN
            } else {
                m = drive_mean(T.D);
            }
            if (lane == 0) s_rave = (real)m;
        }
        if (blockIdx.x == 0 && by == 0 && warp == 1)
            T.acc_zero[lane] = T.acc_zero[kDriveParts + lane] = T.acc_zero[2 * kDriveParts + lane] = 0ull;
    }

    [[maybe_unused]] auto wrap_column = [nx](int x) {
        while (x < 0) x += nx;
        while (x >= nx) x -= nx;
        return x;
    };
    [[maybe_unused]] LogTable logs;
    if constexpr (KP == 1 && MODEL > 0) logs.load();
    V v[9], rho = cst<V>(1.0), f0 = cst<V>(0.0);  // f0: psi (MODEL 0)
    [[maybe_unused]] unsigned qw = 0;              // FP32: the cells' int16 rest extensions
    if ((!SHARE || warp < nwarps) && y < y1 + LV && c < w + HC) {
        int xl = x0 + c - 1, xa = x0 + c, xb = x0 + c + 1, xr = x0 + c + KP;
        const bool edge = x0 < HC + 1 || x0 + w + HC >= nx;  // (of the tile) some column wraps
        if (edge) {
            xl = wrap_column(xl);
            xa = wrap_column(xa);
            xb = wrap_column(xb);
            xr = wrap_column(xr);
        }
        if constexpr (NEAR) {
            const unsigned row = 4u * nx, o0 = yr * row + 4u * xa;
            const unsigned om = yr == 0 ? o0 + (ny - 1) * row : o0 - row, op = yr == ny - 1 ? o0 - yr * row : o0 + row;
            const unsigned pb = (unsigned)P.pitch * 4u;
            if (edge)
                pull_tile32(fin, pb, o0, om, op, 4 * (xl - xa), 4 * (xr - xa), v);
            else
                pull_tile32(fin, pb, o0, om, op, -4, 8, v);
        } else {
            const long long o0 = (long long)yr * nx, om = yr == 0 ? (long long)(ny - 1) * nx : o0 - nx,
                            op = yr == ny - 1 ? 0 : o0 + nx;
            pull_tile<EVEN>(fin, P.pitch, xl, xa, xb, xr, om, o0, op, v);
        }
        if constexpr (std::is_same<real, float>::value) {
            const short* q = rest_lo_plane(fin, P.pitch);
            if constexpr (NEAR) {
                if (out_a) qw = __ldg(reinterpret_cast<const unsigned*>(reinterpret_cast<const char*>(fin) + qo));
            } else if constexpr (EVEN) {
                if (out_a) qw = __ldg(reinterpret_cast<const unsigned*>(q + oc));
            } else {
                if (out_a) qw = (unsigned)(unsigned short)__ldg(q + oc);
                if (out_b) qw |= (unsigned)(unsigned short)__ldg(q + oc + 1) << 16;
            }
        }
        if (wall_img) {
            // first fill: J = (0, -fy/2), or the solved J_y of the one-sided reading
            V jy = cst<V>(real(-0.5) * P.fy);
            if (MODEL > 0 && T.wjy) {
                if constexpr (KP == 1)
                    jy = T.wjy[(top ? nx : 0) + xa];
                else
                    jy = F2(T.wjy[(top ? nx : 0) + xa], T.wjy[(top ? nx : 0) + xb]);
            }
            tile_wall_fill(v, top, cst<V>(0.0), jy);
            if (MODEL == 2 && !T.wjy && T.E.g != real(0)) {
                // gravity: the wall node's density solved in closed form (wall_gravity_refill)
                const real sg = top ? real(-0.5) : real(0.5);
                const V rw = (sum9_v(v) - cst<V>(sg * T.dpg)) * cst<V>(real(1) / (real(1) - sg * T.E.g));
                tile_wall_fill(v, top, cst<V>(0.0), cst<V>(-0.5) * fmav(cst<V>(-T.E.g), rw, cst<V>(T.fyg)));
            }
        }
        rho = sum9_v(v);
        if (MODEL == 0) f0 = tile_psi(rho, P);
    }
    // SHARE, a tile of n rows: warp LV + i collides row i (role 0) together with warp
    // LV + n + i (role 1), on another sub-partition.  The two take 80 and 88 operations in sequence
    // (pseudopotential, free energy) where one takes 125 and 120, each 64 cycles, or 76 with all four
    // sub-partitions busy (256 x 4: 6.1 us per step alone, 5.2 shared; 101 x 50 channel: 8.4, 7.9).
    [[maybe_unused]] int rw = warp, role = -1, sh = 0;
    if constexpr (SHARE) {
        const int n = y1 - y0, i = warp - LV;
        if (i >= 0 && i < 2 * n) {
            role = i < n ? 0 : 1;
            sh = i - role * n;
            rw = LV + sh;
        }
        if (role == 0) {
#pragma unroll
            for (int k = 0; k < 9; ++k) s_v[sh][k][lane] = v[k];
            s_v[sh][9][lane] = rho;
        }
    }
    if (!SHARE || warp < nwarps) s_a[warp][lane] = MODEL == 0 ? f0 : rho;
    __syncthreads();
    // the second warp of a row takes the row's place once the field of its own row is written
    auto join = [&]() {
        if constexpr (SHARE) {
            if (role != 1) return;
            y = y0 - LV + rw;
            wall = WALLS && (y == 0 || y == ny - 1);
            top = WALLS && y != 0;
            out_row = true;
            out_a = c >= 0 && c < w;
            oc = (long long)y * nx + x0 + c;
#pragma unroll
            for (int i = 0; i < 9; ++i) v[i] = s_v[sh][i][lane];
            rho = s_v[sh][9][lane];
        }
    };
    if (MODEL == 0) join();

    // external force of the lane's cells (body force, drive, buoyancy)
    V fx = cst<V>(P.fx), fy = cst<V>(P.fy);
    [[maybe_unused]] real rave = real(0);
    [[maybe_unused]] auto drive = [&]() {
        // the side is that of the lattice column: in the full model the halo lanes' velocities take the force too
        int ga = x0 + c, gb = ga + 1;
        if constexpr (MODEL == 2) {
            ga = wrap_column(ga);
            gb = wrap_column(gb);
        }
        const real al = ga <= T.D.x_split ? T.D.ax_lo : T.D.ax_hi, ah = gb <= T.D.x_split ? T.D.ax_lo : T.D.ax_hi;
        if constexpr (KP == 1)
            fx = fma(al, fabs(rho - rave), P.fx);
        else
            fx = fmav(F2(al, ah), abs_v(rho - F2::c(rave)), F2::c(P.fx));
    };
    if constexpr (DRIVE) {
        rave = s_rave;
        drive();
    }
    if (MODEL == 2) fy = fmav(cst<V>(-T.E.g), rho, cst<V>(T.fyg));

    if constexpr (MODEL == 0) {
        if (!out_row) return;
        V pn[9];
        neighbours(shifted(s_a[rw - 1][lane]), shifted(role == 1 ? s_a[rw][lane] : f0), shifted(s_a[rw + 1][lane]), pn);
        if (wall) {
            mirror_neighbours(pn, top);
            const V Fx = fmav(pn[0], tile_grad_x(pn), fx);  // Eq. (10) + external
            tile_wall_fill(v, top, cst<V>(-0.5) * Fx, cst<V>(-0.5) * fy);
        }
        const Exchange E{1 + sh, &s_x[sh][0][lane]};
        if (SHARE && role == 0)
            tile_collide_pp<0>(v, rho, pn, fx, fy, qw, P, E);
        else if (SHARE && role == 1)
            tile_collide_pp<1>(v, rho, pn, fx, fy, qw, P, E);
        else
            tile_collide_pp<-1>(v, rho, pn, fx, fy, qw, P, E);
    } else {
        Row<V> rm, r0 = shifted(rho), rp, m0;
        V mu = cst<V>(0.0);
        if (warp >= 1 && warp < nwarps - 1 && y < y1 + LV - 1) {
            rm = shifted(s_a[warp - 1][lane]);
            rp = shifted(s_a[warp + 1][lane]);
            V n[9];
            neighbours(rm, r0, rp, n);
            mu = tile_mu(rho, n, P, logs);
        }
        if (!SHARE || warp < nwarps) s_mu[warp][lane] = mu;
        __syncthreads();
        if constexpr (MODEL == 1) {
            join();
            if (!out_row) return;
            V mn[9], rn[9];
            if (SHARE && role == 1) {
                rm = shifted(s_a[rw - 1][lane]);
                r0 = shifted(rho);
                rp = shifted(s_a[rw + 1][lane]);
                mu = s_mu[rw][lane];
                if (DRIVE) drive();
            }
            neighbours(shifted(s_mu[rw - 1][lane]), shifted(mu), shifted(s_mu[rw + 1][lane]), mn);
            neighbours(rm, r0, rp, rn);
            if (wall) {
                // the one-sided reading's normal force -rho d_y mu enters through fy
                if (T.wjy) fy = fmav(-rho, tile_grad_y_onesided(mn, top), fy);
                mirror_neighbours(mn, top);
                mirror_neighbours(rn, top);
                const V Fx = fmav(-rho, tile_grad_x(mn), fx);
                tile_wall_fill(v, top, cst<V>(-0.5) * Fx, cst<V>(-0.5) * fy);
            }
            const Exchange E{1 + sh, &s_x[sh][0][lane]};
            if (SHARE && role == 0)
                tile_collide_fe<0>(v, rho, mn, rn, fx, fy, qw, P, E);
            else if (SHARE && role == 1)
                tile_collide_fe<1>(v, rho, mn, rn, fx, fy, qw, P, E);
            else
                tile_collide_fe<-1>(v, rho, mn, rn, fx, fy, qw, P, E);
        } else {
            V ux = cst<V>(0.0), uy = cst<V>(0.0), Fx = cst<V>(0.0), Fy = cst<V>(0.0);
            if (warp >= 2 && warp < nwarps - 2 && y < y1 + 1) {
                V mn[9];
                neighbours(shifted(s_mu[warp - 1][lane]), shifted(mu), shifted(s_mu[warp + 1][lane]), mn);
                if (wall) {
                    if (T.wjy) fy = fmav(-rho, tile_grad_y_onesided(mn, top), fy);
                    mirror_neighbours(mn, top);
                    const V Gx = fmav(-rho, tile_grad_x(mn), fx);
                    tile_wall_fill(v, top, cst<V>(-0.5) * Gx, cst<V>(-0.5) * fy);
                }
                tile_velocity(v, rho, mn, fx, fy, ux, uy, Fx, Fy);
            }
            s_u[warp][lane] = ux;
            s_u[RMAX + warp][lane] = uy;
            __syncthreads();
            if (!out_row) return;
            V rn[9], un[9], wn[9];
            neighbours(rm, r0, rp, rn);
            neighbours(shifted(s_u[warp - 1][lane]), shifted(ux), shifted(s_u[warp + 1][lane]), un);
            neighbours(shifted(s_u[RMAX + warp - 1][lane]), shifted(uy), shifted(s_u[RMAX + warp + 1][lane]), wn);
            if (wall) {
                mirror_neighbours(rn, top);
                // velocities beyond a no-slip wall: odd extension through u = 0 at the wall node
                mirror_neighbours(un, top);
                mirror_neighbours(wn, top);
                const int i0 = top ? 2 : 4, i1 = top ? 5 : 7, i2 = top ? 6 : 8;
#pragma unroll
                for (int i = 1; i < 9; ++i)
                    if (i == i0 || i == i1 || i == i2) {
                        un[i] = -un[i];
                        wn[i] = -wn[i];
                    }
            }
            tile_collide_iwb(v, rho, rn, un, wn, ux, uy, Fx, Fy, T.dpg * ((real)y - T.E.y_ref), T.dpg, T.E.A, qw, P);
        }
    }

    if constexpr (DRIVE) {
        // the mass this warp stored, summed in pieces of 26 bits
        constexpr unsigned kMask = (1u << kMassLow) - 1;
        bool bad;
        unsigned long long* acc = T.acc_out + (unsigned)(by * 8 + blockIdx.x * 3 + warp) % kDriveParts;
        if constexpr (KP == 1) {
            double s = (v[5] + v[7]) + (v[6] + v[8]);
            if (SHARE && role >= 0) {
                const Exchange E{1 + sh, &s_x[sh][0][lane]};
                if (role == 1) E.x[128] = s;
                E.meet();
                s = E.x[128];
            }
            s = v[0] + (((v[1] + v[3]) + (v[2] + v[4])) + s);
            long long k;
            bad = !mass_fixed(s, T.mass_base, k) && out_a;
            if (!out_a) k = 0;
            const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)k & kMask);
            const long long hi = (long long)__reduce_add_sync(0xffffffffu, (int)(k >> 2 * kMassLow)) * (1ll << kMassLow) +
                                 __reduce_add_sync(0xffffffffu, (unsigned)(k >> kMassLow) & kMask);
            if (lane == 0 && role != 1) {
                atomicAdd(acc, (unsigned long long)lo);
                atomicAdd(acc + kDriveParts, (unsigned long long)hi);
            }
        } else {
            const F2 m = sum9_v(v) * F2::c(T.mass_scale);
            bad = (out_a && !(fabsf(m.v.x) < T.mass_range)) || (out_b && !(fabsf(m.v.y) < T.mass_range));
            const long long k = (out_a ? __float2ll_rn(m.v.x) : 0ll) + (out_b ? __float2ll_rn(m.v.y) : 0ll);
            const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)k & kMask);
            const int hi = __reduce_add_sync(0xffffffffu, (int)(k >> kMassLow));
            if (lane == 0) atomicAdd(acc, (unsigned long long)((long long)hi * (1ll << kMassLow) + lo));
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicAdd(acc + 2 * kDriveParts, 1ull);
    }
    if constexpr (KP == 1) {
        if (out_a)
#pragma unroll
            for (int i = 0; i < 9; ++i)
                if (role < 0 || (i < 5) == (role == 0)) fout[i * P.pitch + oc] = v[i];
    } else if constexpr (NEAR) {
        if (out_a) {
            char* b = reinterpret_cast<char*>(fout);
#pragma unroll
            for (int i = 0; i < 9; ++i)
                *reinterpret_cast<float2*>(b + (oc32 + (unsigned)P.pitch * 4u * i)) = v[i].v;
            *reinterpret_cast<unsigned*>(b + qo) = qw;
        }
    } else if constexpr (EVEN) {
        if (out_a) {
#pragma unroll
            for (int i = 0; i < 9; ++i) *reinterpret_cast<float2*>(fout + i * P.pitch + oc) = v[i].v;
            *reinterpret_cast<unsigned*>(rest_lo_plane(fout, P.pitch) + oc) = qw;
        }
    } else {
        short* q = rest_lo_plane(fout, P.pitch);
        if (out_a) {
#pragma unroll
            for (int i = 0; i < 9; ++i) fout[i * P.pitch + oc] = v[i].v.x;
            q[oc] = (short)(qw & 0xffffu);
        }
        if (out_b) {
#pragma unroll
            for (int i = 0; i < 9; ++i) fout[i * P.pitch + oc + 1] = v[i].v.y;
            q[oc + 1] = (short)(qw >> 16);
        }
    }
}

}  // namespace lbmk
