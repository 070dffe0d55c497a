// Transposed step on the pre-scaled coefficient (FP64, equal spacings).
//
// With Cs = dt*lam*_d^2*Ci the forward step reads T2 = T + Cs*L(T) at interior
// nodes, L(A) = sum of the six neighbours of A minus six times the centre.
// Its transpose, for ybar = dL/dT2 and the state T the step read:
//   w[q]      = Cs[q]*ybar[q] at interior q, 0 elsewhere (and outside the grid),
//   Tbar[p]   = ybar[p] + L(w)[p]                      (every node p),
//   Csbar[q] += ybar[q]*L(T)[q]                         (interior q),
// and dL/dCi = dt*lam*_d^2 * Csbar (applied once by the caller).
//
// Layout as in the other z-march kernels: a CTA owns a 64 x BY x-y tile (one
// warp per row, two nodes per thread) and a chunk of z-planes of the whole
// grid.  For every plane one thread issues three TMA boxes (T, ybar, Cs with a
// one-node y halo and a 16-byte x halo) into one ring stage tracked by one
// mbarrier.  w of plane k+1 is built into one of three rotating shared tiles
// as 64-bit fixed point at a CTA-uniform, non-decreasing scale 2^(Esc-1079)
// (|value| < 2^57 units): each thread converts its own two nodes, and 144
// threads one halo node each.  A conversion that would not fit the current
// scale is flagged through the plane's single __syncthreads_or; only then does
// the CTA agree on a larger scale and shift what it already holds.
//
// Per node: Tbar = ybar + pack(S_w) with S_w the exact integer sum (one DADD);
// Csbar = fma(ybar, pack(S_T), Csbar) with S_T the exact bit-pattern sum of
// the same-binade fast path (one DFMA); w = Cs*ybar costs one DMUL per tile
// value.  Csbar of plane k is loaded at the top of iteration k so that its
// latency hides behind the w tile work.
//
// The same kernel takes Ci as given (kAx, kGiven below).  Measured at 256^3 against the
// z-march it replaced there (adjoint_zmarch.cu: w values spread over the threads, two
// barriers per plane, one pack and one FP64 product per axis): equal spacings 184 against
// 244 us, unequal 240 against 362; 512 x 384 x 256 unequal 693 against 1014.
#include <cudaTypedefs.h>


#include "emu64.cuh"
#include "internal.h"
#include "pdl.cuh"
#include "tma.cuh"
#include "waves.h"
#include "zmarch.h"

namespace psd {

__device__ unsigned g_adjs_error;  // set when an mbarrier wait times out

struct AdjSParams {
    int64_t nx, ny, nz;
    int kchunk, ntx;
    EmuCoef ek;  // AX_COMMON, AX_SPREAD: dt*lam*_d^2 of the axes at one exponent
};

// Fixed-point value of FP64 bits v at scale 2^(E-1079) (E >= the exponent of v).
__device__ __forceinline__ long long adjs_fixed(unsigned long long v, int E) {
    return emu_fixed(v, E);
}

// Exact-when-possible FP64 of the integer S at scale 2^sc.
__device__ __forceinline__ double adjs_pack(long long S, int sc) { return emu_pack(S, sc); }

// The same for a scale at which every packed sum is normal (or zero): |S| < 2^61 at
// scale 2^(E-1079) has an exponent between E - 57 and E + 3, so for E in [57, 2042] the
// range checks can go (the CTA-uniform scale picks this form for the whole plane).
__device__ __forceinline__ double adjs_pack_normal(long long S, int sc) {
    unsigned long long sg;
    const unsigned long long a = emu_abs(S, &sg);
    return bitsd(emu_pack_mag_normal(a, sc) | sg);
}

template <int kAx>
static __device__ __noinline__ double adjs_lap_general(unsigned long long c, unsigned long long xm,
                                                       unsigned long long xp, unsigned long long ym,
                                                       unsigned long long yp, unsigned long long zm,
                                                       unsigned long long zp, const EmuCoef &k) {
    long long sx, sy, sz;
    int sc;
    const double cc = bitsd(c);
    if (emu_sums_general(c, xm, xp, ym, yp, zm, zp, sx, sy, sz, sc)) {
        if constexpr (kAx != AX_ISO) return emu_L_signed<kAx>(sx, sy, sz, sc, c, k);
        return emu_pack(sx + sy + sz, sc);
    }
    // Inf / NaN: plain FP64 propagates it
    if constexpr (kAx != AX_ISO) {
        const double d2x = (bitsd(xp) - cc) - (cc - bitsd(xm)), d2y = (bitsd(yp) - cc) - (cc - bitsd(ym)),
                     d2z = (bitsd(zp) - cc) - (cc - bitsd(zm));
        return k.dtlam * ((d2x * k.ax + d2y * k.ay) + d2z * k.az);
    }
    return (((bitsd(xm) + bitsd(xp)) + (bitsd(ym) + bitsd(yp))) + (bitsd(zm) + bitsd(zp))) - 6.0 * cc;
}

// Odd rows whose march meets an infinite or NaN w, which no fixed point holds: plain FP64 from the fields
// themselves (the plain column kernels' arithmetic, adjoint.cu).  kGiven: Ci as given, else the pre-scaled
// coefficient.
struct AdjsFields {
    const double *ybar, *Ci;
    int nx, ny, nz;
    double dtlam, ax, ay, az;
};
template <bool kGiven>
__device__ __forceinline__ double adjs_plain_lap(const AdjsFields &f, double c, double xm, double xp, double ym,
                                                 double yp, double zm, double zp) {
    if (!kGiven) return ((xm + xp) + (ym + yp)) + (zm + zp) - 6.0 * c;
    const double d2x = (xp - c) - (c - xm), d2y = (yp - c) - (c - ym), d2z = (zp - c) - (c - zm);
    return (d2x * f.ax + d2y * f.ay) + d2z * f.az;
}
// Tbar of one node.
template <bool kGiven>
__device__ __noinline__ double adjs_plain(const AdjsFields f, int x, int y, int z) {
    auto w = [&](int i, int j, int k) -> double {
        if (i < 1 || i > f.nx - 2 || j < 1 || j > f.ny - 2 || k < 1 || k > f.nz - 2) return 0.0;
        const int64_t q = i + (int64_t)f.nx * (j + (int64_t)f.ny * k);
        return kGiven ? f.dtlam * (f.Ci[q] * f.ybar[q]) : f.Ci[q] * f.ybar[q];
    };
    return f.ybar[x + (int64_t)f.nx * (y + (int64_t)f.ny * z)] +
           adjs_plain_lap<kGiven>(f, w(x, y, z), w(x - 1, y, z), w(x + 1, y, z), w(x, y - 1, z), w(x, y + 1, z),
                                  w(x, y, z - 1), w(x, y, z + 1));
}
// Planes [k0, k1) at nodes x0 and x1 of row y: the rest of a march.
template <bool kGiven>
__device__ __noinline__ void adjs_plain_march(const AdjsFields f, double *Tbar, double *Cbar, const double *T, int x0,
                                              int x1, int y, int k0, int k1) {
    if (y > f.ny - 1) return;
    const int64_t sy = f.nx, sz = sy * f.ny;
    for (int k = k0; k < k1; ++k)
        for (int x = x0; x <= x1 && x <= f.nx - 1; x += x1 - x0) {
            const int64_t q = x + sy * y + sz * k;
            Tbar[q] = adjs_plain<kGiven>(f, x, y, k);
            if (x < 1 || x > f.nx - 2 || y < 1 || y > f.ny - 2 || k < 1 || k > f.nz - 2) continue;
            const double L = adjs_plain_lap<kGiven>(f, T[q], T[q - 1], T[q + 1], T[q - sy], T[q + sy], T[q - sz], T[q + sz]);
            Cbar[q] = kGiven ? Cbar[q] + f.dtlam * (f.ybar[q] * L) : fma(f.ybar[q], L, Cbar[q]);
        }
}

// kAx, kGiven: AX_ISO on the pre-scaled coefficient; AX_ISO and kGiven, Ci as given on equal
// spacings: w = Ci*ybar, the one dt*lam*_d^2 multiplied in last (Tbar by the DFMA that
// replaces the DADD, Cibar by one more DMUL); AX_COMMON and AX_SPREAD, Ci as given on unequal spacings: w =
// Ci*ybar, Tbar = ybar + L(w) and Cibar += ybar*L(T) with L = sum_d dt*lam*_d^2 * (second
// difference along d), the axes' exact sums combined as integers (emu_L_common).
// kRag: odd nx.  A plane of a field arrives as two boxes, its even and its odd tile rows, over
// the field mapped as rows of 2*nx (zrag_tile.cuh); a row's data then starts at its slot's
// first or second element, and lanes own nodes lane and lane + 32 of their row.  Measured
// against the plain column kernel: 161 x 128 x 96 unequal 49 against 204 us, 257^3 pre-scaled
// 248 against 735 (a fifth of that in the tiles of the one column past 256).
template <int BY, int NST, int kAx, bool kGiven, bool kRag>
__global__ void __launch_bounds__(32 * BY, 3)
k_adjoint_scaled(const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmY,
                 const __grid_constant__ CUtensorMap tmC, double *__restrict__ Tbar,
                 double *__restrict__ Csbar, const double *__restrict__ ybar, const double *__restrict__ T,
                 const double *__restrict__ Ci, const AdjSParams p) {
    constexpr int PX = 2, HX = 2, BX = 64, W = BX + 2 * HX, H = BY + 2;
    constexpr int NHALO = 2 * BX + 2 * BY;  // y-halo rows and x-halo columns (no corners)
    static_assert(NHALO <= 32 * BY, "one halo value per thread at most");
    constexpr unsigned TB = W * H * 8;
    constexpr unsigned WBA = (TB + 127) / 128 * 128, WS = WBA / 8;  // w tile stride
    constexpr unsigned HBX = (TB / 2 + 127) / 128 * 128;             // box of even or odd rows
    constexpr unsigned TBA = kRag ? 2 * HBX : WBA, SS = TBA / 8;     // field stride in elements
    constexpr int XS = kRag ? 32 : 1;                                // between a lane's two nodes
    extern __shared__ __align__(128) unsigned char smem[];
    double *ring = (double *)smem;                       // NST stages x {T, ybar, Cs}
    long long *wtile = (long long *)(smem + 3 * NST * TBA);  // 3 rotating w tiles
    uint64_t *bar = (uint64_t *)(smem + 3 * NST * TBA + 3 * WBA);
    __shared__ int s_abort, s_E;
    grid_dep_wait();  // the previous launch's writes (and its reads of Tbar) are complete
    grid_dep_launch();

    const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int X0 = (int)(blockIdx.x % p.ntx) * BX, Y0 = (int)(blockIdx.x / p.ntx) * BY;
    const int k0 = (int)blockIdx.y * p.kchunk;
    const int k1 = (int)min((int64_t)k0 + p.kchunk, p.nz);  // output planes [k0, k1)
    const int nx = (int)p.nx, ny = (int)p.ny, nz = (int)p.nz;

    auto issue = [&](int s, int q) {
        mbar_expect_tx(&bar[s], 3 * TB);
        if constexpr (kRag) {
            // tile row h is field row r + h; o: the residue of row r, boxes of rows h = 0, 2, ..
            // and h = 1, 3, ..; x from column -1 rounded down to an even element
            const int64_t r = (int64_t)q * ny + Y0 - 1;
            const int o = (int)(r & 1), g0 = (int)(r >> 1), g1 = (int)((r + 1) >> 1);
            const int x0 = (o * nx + X0 - 1) & ~1, x1 = ((o ^ 1) * nx + X0 - 1) & ~1;
            const CUtensorMap *tm[3] = {&tmT, &tmY, &tmC};
#pragma unroll
            for (int f = 0; f < 3; ++f) {
                unsigned char *dst = (unsigned char *)(ring + (3 * s + f) * SS);
                tma_load_2d(dst, tm[f], &bar[s], x0, g0);
                tma_load_2d(dst + HBX, tm[f], &bar[s], x1, g1);
            }
            return;
        }
        tma_load_3d(ring + (3 * s + 0) * SS, &tmT, &bar[s], X0 - HX, Y0 - 1, q);
        tma_load_3d(ring + (3 * s + 1) * SS, &tmY, &bar[s], X0 - HX, Y0 - 1, q);
        tma_load_3d(ring + (3 * s + 2) * SS, &tmC, &bar[s], X0 - HX, Y0 - 1, q);
    };
    if (threadIdx.x == 0) {
        s_abort = 0;
        s_E = 1;
        for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int s = 0; s < NST; ++s)
            if (k0 - 1 + s <= k1) issue(s, k0 - 1 + s);  // planes k0-1 .. (-1 and nz read zeros)

    unsigned par = 0u;
    auto nexts = [](int s) { return s + 1 == NST ? 0 : s + 1; };
    // After a timed-out wait: bounded waits for the copies of the last NST planes
    // issued (up to plane q_iss), so that no TMA write lands after the CTA exits.
    auto drain = [&](int q_iss) {
        for (int q = max(k0 - 1, q_iss - NST + 1); q <= q_iss; ++q) {
            const int i = q - (k0 - 1);
            mbar_wait(&bar[i % NST], (unsigned)(i / NST) & 1u);
        }
    };
    auto acquire = [&](int s) -> bool {
        const unsigned ph = (par >> s) & 1u;
        par ^= 1u << s;
        return mbar_wait(&bar[s], ph);
    };

    // this thread's own nodes (row, col and col + XS of the tile) and halo node
    const int row = ty + 1, col = HX + (kRag ? lane : lane * PX);
    const int gy = Y0 + ty, gx0 = X0 + (kRag ? lane : lane * PX);
    const bool iny = gy >= 1 && gy <= ny - 2;
    const bool m0 = iny && gx0 >= 1 && gx0 <= nx - 2;
    const bool m1 = iny && gx0 + XS >= 1 && gx0 + XS <= nx - 2;
    // position of tile row r, column c (the w tile's columns, node x = X0 - HX + c) in a field
    // of plane q.  kRag: row r of the field's even or odd box, shifted by the row's offset
    // d = (row * nx + X0 - 1) mod 2 = (row + 1) mod 2 (odd nx, even X0)
    auto at = [&](int r, int c, int q) -> int {
        if (!kRag) return r * W + c;
        const int d = (q * ny + Y0 + r) & 1;
        return (r & 1) * (int)(HBX / 8) + (r >> 1) * W + c - 1 + d;
    };
    // values at the lane's two nodes of a field row at position o (and of a w tile row)
    auto two = [&](const double *f, int o) -> double2 {
        return kRag ? make_double2(f[o], f[o + XS]) : *(const double2 *)(f + o);
    };
    // a last single row is outside the row-pair map (N rows, N odd): its ybar, which Tbar
    // copies there, is read from the field itself
    const bool lone = kRag && gy == ny - 1 && (((int64_t)ny * nz) & 1);
    const int t = threadIdx.x;
    const bool has_h = t < NHALO;
    int hr, hc;
    if (t < 2 * BX) {
        hr = t < BX ? 0 : H - 1;
        hc = HX + (t & (BX - 1));
    } else {
        const int u = t - 2 * BX;
        hr = 1 + (u >> 1);
        hc = (u & 1) ? HX + BX : HX - 1;
    }
    const int hidx = has_h ? hr * W + hc : 0;
    if (!has_h) hr = 0, hc = 1;
    const int hx = X0 - HX + hc, hy = Y0 - 1 + hr;
    const bool hm = has_h && hx >= 1 && hx <= nx - 2 && hy >= 1 && hy <= ny - 2;

    auto put2 = [&](long long *o, long long a, long long b) {
        if (kRag) {
            o[0] = a;
            o[XS] = b;
        } else {
            *(longlong2 *)o = make_longlong2(a, b);
        }
    };
    // w of plane q from a stage: own two nodes and the halo node, as doubles
    double w0, w1, wh;
    double2 ynext;  // ybar at the own nodes of plane q (the next iteration's centre)
    auto w_compute = [&](int s, int q) -> int {
        const double *Ys = ring + (3 * s + 1) * SS, *Cs = ring + (3 * s + 2) * SS;
        const bool zin = q >= 1 && q <= nz - 2;
        const int o = at(row, col, q);
        ynext = two(Ys, o);
        const double2 c2 = two(Cs, o);
        if (lone && q == nz - 1) {
            const double *yl = ybar + (int64_t)nx * ((int64_t)ny * nz - 1) + gx0;
            if (gx0 <= nx - 1) ynext.x = yl[0];
            if (gx0 + XS <= nx - 1) ynext.y = yl[XS];
        }
        w0 = (zin && m0) ? c2.x * ynext.x : 0.0;
        w1 = (zin && m1) ? c2.y * ynext.y : 0.0;
        const int oh = at(hr, hc, q);
        wh = (zin && hm) ? Cs[oh] * Ys[oh] : 0.0;
        return max(max(emu_exp(dbits(w0)), emu_exp(dbits(w1))), emu_exp(dbits(wh)));
    };
    auto w_store = [&](long long *wt, int E, long long &f0, long long &f1) {
        f0 = adjs_fixed(dbits(w0), E);
        f1 = adjs_fixed(dbits(w1), E);
        put2(wt + row * W + col, f0, f1);
        if (has_h) wt[hidx] = adjs_fixed(dbits(wh), E);
    };

    // ---- prologue: planes k0-1 (own w, T centre) and k0 (w tile, T and ybar centres)
    int s_m = 0, s_c = 1 % NST;
    bool ok = acquire(s_m);
    ok = acquire(s_c) && ok;
    double2 tm = two(ring + (3 * s_m) * SS, at(row, col, k0 - 1));
    double2 tc = two(ring + (3 * s_c) * SS, at(row, col, k0));
    int em = w_compute(s_m, k0 - 1);  // includes both own w of plane k0-1
    const double wm0d = w0, wm1d = w1;  // (its halo value is not needed)
    em = max(em, w_compute(s_c, k0));
    double2 yc = ynext;
    em = (int)__reduce_max_sync(0xffffffffu, (unsigned)em);
    if (lane == 0) atomicMax(&s_E, em);
    if (!ok) {
        s_abort = 1;
        atomicOr(&g_adjs_error, 1u);
    }
    __syncthreads();
    if (s_abort) {
        drain(min(k0 + 1, k1));
        return;
    }
    int Esc = s_E;  // CTA-uniform
    // A non-finite w (Esc 0x7ff) makes the CTA's Tbar NaN from there on; on odd rows it stays with the nodes
    // that meet it: with equal spacings the march ends and plain FP64 takes its rest, else the march goes on
    // and forms every Tbar so (either form costs the other kernel 3 to 5% in registers; this way 257^3
    // pre-scaled 251 us, 249.5 without, 257 x 200 x 180 unequal 212 and 212).
    auto fields = [&]() {
        return AdjsFields{ybar, Ci, nx, ny, nz, p.ek.dtlam, p.ek.ax, p.ek.ay, p.ek.az};
    };
    constexpr bool kEnds = kRag && kAx == AX_ISO;
    auto plain_rest = [&](int k) {
        drain(min(k + 1, k1));
        adjs_plain_march<kGiven>(fields(), Tbar, Csbar, T, gx0, gx0 + XS, gy, k, k1);
    };
    if (kEnds && Esc == 0x7ff) {
        plain_rest(k0);
        return;
    }
    int wcur = 0;
    long long wc0, wc1;
    w_store(wtile, Esc, wc0, wc1);
    long long wm0 = adjs_fixed(dbits(wm0d), Esc), wm1 = adjs_fixed(dbits(wm1d), Esc);

    const bool row_out = gy <= ny - 1;
    const bool all_x = !kRag && gx0 + PX - 1 <= nx - 1;
    const bool all_in = m0 && m1;
    const bool vec = !kRag && all_in;  // 16-byte accesses to Csbar

    for (int k = k0; k < k1; ++k) {
        const int s_n = nexts(s_c);  // stage of plane k+1
        const bool plane_in = k >= 1 && k <= nz - 2;
        const bool do_ci = iny && plane_in;
        const int64_t base = (int64_t)gx0 + p.nx * ((int64_t)gy + p.ny * (int64_t)k);
        // Csbar of plane k: issued early, used at the end of the iteration
        double2 cb = make_double2(0.0, 0.0);
        if (do_ci) {
            if (vec) {
                cb = *(const double2 *)(Csbar + base);
            } else {
                if (m0) cb.x = Csbar[base];
                if (m1) cb.y = Csbar[base + XS];
            }
        }
        ok = acquire(s_n);
        const int wnxt = wcur == 2 ? 0 : wcur + 1;
        const int emn = w_compute(s_n, k + 1);
        long long wp0, wp1;
        w_store(wtile + wnxt * WS, Esc, wp0, wp1);
        if (!ok) {
            s_abort = 1;
            atomicOr(&g_adjs_error, 1u);
        }
        // tile k+1 complete; every thread has left iteration k-1 (its stage is free)
        if (__syncthreads_or(emn > Esc || !ok)) {
            if (s_abort) {
                drain(min(k + 1, k1));
                return;
            }
            // a w of plane k+1 needs a larger scale: agree on it, shift what is held
            const int e = (int)__reduce_max_sync(0xffffffffu, (unsigned)emn);
            if (lane == 0) atomicMax(&s_E, e);
            __syncthreads();
            const int E2 = s_E;
            if (kEnds && E2 == 0x7ff) {
                plain_rest(k);
                return;
            }
            const int d = E2 - Esc;  // > 0
            long long *wk = wtile + wcur * WS;
            auto shr = [d](long long v) { return d >= 64 ? 0ll : (v >> d); };
            wc0 = shr(wc0);
            wc1 = shr(wc1);
            wm0 = shr(wm0);
            wm1 = shr(wm1);
            put2(wk + row * W + col, wc0, wc1);
            if (has_h) wk[hidx] = shr(wk[hidx]);
            Esc = E2;
            w_store(wtile + wnxt * WS, Esc, wp0, wp1);
            __syncthreads();
        }
        if (threadIdx.x == 0 && k - 1 + NST <= k1) issue(s_m, k - 1 + NST);  // plane k-1's stage

        if (row_out) {
            // ---- Tbar = ybar + L(w), exact integer sums, one DADD per node
            const long long *wk = wtile + wcur * WS + row * W + col;
            // x-neighbours: of node 0 (wl, wr0) and of node 1 (wl1, wr); side by side where the
            // lane's nodes are neighbours
            const long long wl = wk[-1], wr = wk[kRag ? XS + 1 : PX];
            const long long wr0 = kRag ? wk[1] : wc1, wl1 = kRag ? wk[XS - 1] : wc0;
            longlong2 wu, wd;
            if constexpr (kRag) {
                wu = make_longlong2(wk[-W], wk[XS - W]);
                wd = make_longlong2(wk[W], wk[XS + W]);
            } else {
                wu = *(const longlong2 *)(wk - W);
                wd = *(const longlong2 *)(wk + W);
            }
            const int sc = Esc - 1079;
            double2 tb;
            const long long S0 = ((wl + wr0) + (wu.x + wd.x)) + (wm0 + wp0) - 6 * wc0;
            const long long S1 = ((wl1 + wr) + (wu.y + wd.y)) + (wm1 + wp1) - 6 * wc1;
            if constexpr (kAx != AX_ISO) {
                if (Esc == 0x7ff) {  // a non-finite w in this CTA's march
                    tb.x = tb.y = __longlong_as_double(0x7ff8000000000000ll);
                    if constexpr (kRag) {
                        if (gx0 <= nx - 1) tb.x = adjs_plain<kGiven>(fields(), gx0, gy, k);
                        if (gx0 + XS <= nx - 1) tb.y = adjs_plain<kGiven>(fields(), gx0 + XS, gy, k);
                    }
                } else {
                    const long long a2 = 2 * wc0, b2 = 2 * wc1;
                    tb.x = yc.x + emu_L_common<3, kAx == AX_SPREAD, false>(wl + wr0 - a2, wu.x + wd.x - a2, wm0 + wp0 - a2, sc, 0ull, p.ek);
                    tb.y = yc.y + emu_L_common<3, kAx == AX_SPREAD, false>(wl1 + wr - b2, wu.y + wd.y - b2, wm1 + wp1 - b2, sc, 0ull, p.ek);
                }
            } else if (Esc >= 57 && Esc <= 2042) {  // CTA-uniform: the packed sums are normal
                tb.x = kGiven ? fma(p.ek.Kx, adjs_pack_normal(S0, sc), yc.x) : yc.x + adjs_pack_normal(S0, sc);
                tb.y = kGiven ? fma(p.ek.Kx, adjs_pack_normal(S1, sc), yc.y) : yc.y + adjs_pack_normal(S1, sc);
            } else if (!kRag && Esc == 0x7ff) {  // a non-finite w in this CTA's march
                tb.x = tb.y = __longlong_as_double(0x7ff8000000000000ll);
            } else {
                tb.x = kGiven ? fma(p.ek.Kx, adjs_pack(S0, sc), yc.x) : yc.x + adjs_pack(S0, sc);
                tb.y = kGiven ? fma(p.ek.Kx, adjs_pack(S1, sc), yc.y) : yc.y + adjs_pack(S1, sc);
            }
            if (all_x) {
                *(double2 *)(Tbar + base) = tb;
            } else {
                if (gx0 <= nx - 1) Tbar[base] = tb.x;
                if (gx0 + XS <= nx - 1) Tbar[base + XS] = tb.y;
            }

            // ---- Csbar += ybar * L(T), bit-pattern sums on the same-binade fast path
            if (do_ci) {
                const double *Tk = ring + (3 * s_c) * SS;
                const double2 tp = two(ring + (3 * s_n) * SS, at(row, col, k + 1));
                const double2 tu = two(Tk, at(row - 1, col, k));
                const double2 td = two(Tk, at(row + 1, col, k));
                const double *To = Tk + at(row, col, k);
                const double tl = To[-1], tr = To[kRag ? XS + 1 : PX];
                const unsigned long long c0 = dbits(tc.x), c1 = dbits(tc.y);
                const unsigned long long xl = dbits(tl), xr = dbits(tr);
                const unsigned long long xr0 = kRag ? dbits(To[1]) : c1, xl1 = kRag ? dbits(To[XS - 1]) : c0;
                const unsigned long long u0 = dbits(tu.x), u1 = dbits(tu.y), d0 = dbits(td.x),
                                         d1 = dbits(td.y), m0b = dbits(tm.x), m1b = dbits(tm.y),
                                         p0 = dbits(tp.x), p1 = dbits(tp.y);
                unsigned hc0 = (unsigned)(c0 >> 32);
                unsigned hw[kRag ? 13 : 11] = {(unsigned)(xl >> 32), (unsigned)(xr >> 32), (unsigned)(u0 >> 32),
                                   (unsigned)(d0 >> 32), (unsigned)(m0b >> 32), (unsigned)(p0 >> 32),
                                   (unsigned)(u1 >> 32), (unsigned)(d1 >> 32), (unsigned)(m1b >> 32),
                                   (unsigned)(p1 >> 32), (unsigned)(c1 >> 32)};
                if constexpr (kRag) {
                    hw[11] = (unsigned)(xr0 >> 32);
                    hw[12] = (unsigned)(xl1 >> 32);
                }
                if (!all_in) {  // values of unstored nodes must not force the general path
                    // a lane that stores neither node (past the grid: zeros) votes for the fast
                    // path: its reference is 1.0's word (its outputs are never stored)
                    if (!m0 && !m1) hc0 = 0x3ff00000u;
                    if (!m0) hw[0] = hw[2] = hw[3] = hw[4] = hw[5] = hc0;
                    if (!m1) hw[1] = hw[6] = hw[7] = hw[8] = hw[9] = hc0;
                    if constexpr (kRag) {  // the nodes are no neighbours: each has its own six
                        if (!m0) hc0 = m1 ? (unsigned)(c1 >> 32) : 0x3ff00000u;
                        if (!m0) hw[0] = hw[2] = hw[3] = hw[4] = hw[5] = hw[11] = hc0;
                        if (!m1) hw[1] = hw[6] = hw[7] = hw[8] = hw[9] = hw[10] = hw[12] = hc0;
                    }
                    if (!m0 && !m1) hw[10] = hc0;
                }
                const bool fast = emu_same_binade_hi(hw, hc0);
                double L0, L1;
                if (kAx != AX_ISO && __all_sync(0xffffffffu, fast)) {
                    const unsigned long long a2 = 2ull * c0, b2 = 2ull * c1;
                    const int sct = (int)((hc0 >> 20) & 0x7ffu) - 1075;
                    const unsigned long long flip = (unsigned long long)(hc0 & 0x80000000u) << 32;  // negative: minus
                    L0 = emu_L_common<3, kAx == AX_SPREAD, true>((long long)(xl + xr0 - a2), (long long)(u0 + d0 - a2),
                                         (long long)(m0b + p0 - a2), sct, flip, p.ek);
                    L1 = emu_L_common<3, kAx == AX_SPREAD, true>((long long)(xl1 + xr - b2), (long long)(u1 + d1 - b2),
                                         (long long)(m1b + p1 - b2), sct, flip, p.ek);
                } else if (kAx == AX_ISO && __all_sync(0xffffffffu, fast)) {
                    const long long S0t = (long long)(((xl + xr0) + (u0 + d0)) + (m0b + p0) - 6ull * c0);
                    const long long S1t = (long long)(((xl1 + xr) + (u1 + d1)) + (m1b + p1) - 6ull * c1);
                    const int sct = (int)((hc0 >> 20) & 0x7ffu) - 1075;
                    const unsigned long long flip = (unsigned long long)(hc0 & 0x80000000u) << 32;  // negative: minus
                    unsigned long long g0, g1;
                    const unsigned long long a0 = emu_abs(S0t, &g0), a1 = emu_abs(S1t, &g1);
                    L0 = bitsd(emu_pack_mag_normal(a0, sct) | (g0 ^ flip));
                    L1 = bitsd(emu_pack_mag_normal(a1, sct) | (g1 ^ flip));
                } else {
                    L0 = m0 ? adjs_lap_general<kAx>(c0, xl, xr0, u0, d0, m0b, p0, p.ek) : 0.0;
                    L1 = m1 ? adjs_lap_general<kAx>(c1, xl1, xr, u1, d1, m1b, p1, p.ek) : 0.0;
                }
                cb.x = fma(kAx == AX_ISO && kGiven ? p.ek.Kx * yc.x : yc.x, L0, cb.x);
                cb.y = fma(kAx == AX_ISO && kGiven ? p.ek.Kx * yc.y : yc.y, L1, cb.y);
                if (vec) {
                    *(double2 *)(Csbar + base) = cb;
                } else {
                    if (m0) Csbar[base] = cb.x;
                    if (m1) Csbar[base + XS] = cb.y;
                }
            }
        }
        // rotate: plane k becomes the minus neighbour, plane k+1 the centre
        tm = tc;
        tc = two(ring + (3 * s_n) * SS, at(row, col, k + 1));
        yc = ynext;
        wm0 = wc0;
        wm1 = wc1;
        wc0 = wp0;
        wc1 = wp1;
        s_m = s_c;
        s_c = s_n;
        wcur = wnxt;
    }
}

template <int kAx, bool kGiven, bool kRag>
static cudaError_t launch_adjs_t(double *Tbar, double *Csbar, const double *ybar, const double *T,
                               const double *Cs, const EmuCoef &ek, Grid3 g, cudaStream_t s) {
    constexpr int BY = 8, NST = 3, PX = 2, BX = 32 * PX, W = BX + 2 * PX, H = BY + 2;
    constexpr unsigned WBA = (W * H * 8 + 127) / 128 * 128;
    constexpr unsigned TBA = kRag ? 2 * ((W * H / 2 * 8 + 127) / 128 * 128) : WBA;
    constexpr size_t smem = 3 * NST * TBA + 3 * WBA + NST * 8;
    static unsigned attr_gen[64] = {0};
    cudaError_t ae;
    if (!set_smem_attr_once((const void *)k_adjoint_scaled<BY, NST, kAx, kGiven, kRag>, (int)smem, attr_gen, &ae)) return ae;
    CUtensorMap mT, mY, mC;
    auto map = [&](CUtensorMap *m, const double *f) {
        return kRag ? make_tensor_map_rows(m, f, 8, g.n(), 2 * g.nx, W, H / 2) : make_tensor_map_3d(m, f, 8, g, W, H);
    };
    if (!map(&mT, T) || !map(&mY, ybar) || !map(&mC, Cs)) return cudaErrorInvalidValue;
    const int64_t ntx = (g.nx + BX - 1) / BX, nty = (g.ny + BY - 1) / BY, tiles = ntx * nty;
    int kchunk = launch_override(PS_OVERRIDE_ADJ_KCHUNK);
    if (kchunk <= 0) {
        // long z-chunks amortise the two prologue planes; keep at least ~3 waves of CTAs
        // (3 per SM).  Where chunks of 16 planes or more keep that many, take the chunk
        // of 16-24 planes whose last wave is fullest: measured 256^3 at 19 planes
        // (3.93 waves) 0.1734 ms against 0.1777 at 16 (4.49 waves); 512^3 at 22-24
        // planes 1.5% ahead of 16.
        const int64_t slots = 3LL * sm_count();
        if (g.nz * tiles / (3 * slots) < 16) {
            // (chunks below 4 planes only where 4 leave most of the chip idle: 32^3 4.1 us at
            // 1 plane against 7.6, 48^3 5.2 at 2 against 7.7, 64^3 7.6 at 4 against 8.4 at 2).
            // A few waves: fitted to sweeps of 40 shapes (us against chunks for about three waves:
            // 100^3 21.1 / 23.7, 160^3 58.4 / 62.3, 161^3 69.9 / 77.6, 128 x 150 x 200 45.5 / 53.2), but
            // not where the last tile of a row is nearly empty: its CTAs end early, and what
            // the others gain by long chunks is lost (129 x 400 x 96 139 us, 130 in short ones)
            const int64_t at4 = tiles * ((g.nz + 3) / 4), kc = g.nz * tiles / (3 * slots);
            const bool thin = g.nx % BX >= 1 && g.nx % BX <= BX / 4;
            kchunk = at4 * 8 < slots ? 1
                     : at4 * 4 < slots ? 2
                     : thin            ? (int)(kc < 4 ? 4 : kc)
                                       : wave_chunk(g.nz, tiles, sm_count(), 3, WaveCost{0.5, 0.6, 0.05, 3, 40});
        } else {
            kchunk = 16;
            int64_t best = -1;
            for (int c = 16; c <= 24; ++c) {
                const int64_t ctas = tiles * ((g.nz + c - 1) / c);
                const int64_t last = ctas % slots == 0 ? slots : ctas % slots;  // CTAs in the last wave
                if (last > best) {
                    best = last;
                    kchunk = c;
                }
            }
        }
    }
    kchunk = grid_chunk(g.nz, kchunk);
    const int64_t gz = (g.nz + kchunk - 1) / kchunk;
    if (tiles > 0x7fffffffLL || gz > 65535) return cudaErrorInvalidConfiguration;
    AdjSParams p{g.nx, g.ny, g.nz, kchunk, (int)ntx, ek};
    return launch_pdl(k_adjoint_scaled<BY, NST, kAx, kGiven, kRag>, dim3((unsigned)tiles, (unsigned)gz, 1), dim3(32 * BY), smem, s,
                      mT, mY, mC, Tbar, Csbar, ybar, T, Cs, p);
}

template <int kAx, bool kGiven>
static cudaError_t launch_adjs(double *Tbar, double *Csbar, const double *ybar, const double *T,
                               const double *Cs, const EmuCoef &ek, Grid3 g, cudaStream_t s) {
    if (g.nx % 2) return launch_adjs_t<kAx, kGiven, true>(Tbar, Csbar, ybar, T, Cs, ek, g, s);
    return launch_adjs_t<kAx, kGiven, false>(Tbar, Csbar, ybar, T, Cs, ek, g, s);
}

cudaError_t launch_adjoint_scaled(double *Tbar, double *Csbar, const double *ybar, const double *T,
                                  const double *Cs, Grid3 g, cudaStream_t s) {
    return launch_adjs<AX_ISO, false>(Tbar, Csbar, ybar, T, Cs, EmuCoef{}, g, s);
}

cudaError_t launch_adjoint_given(double *Tbar, double *Cibar, const double *ybar, const double *T,
                                 const double *Ci, const EmuCoef &ek, Grid3 g, cudaStream_t s) {
    if (ek.ax == ek.ay && ek.ay == ek.az)
        return launch_adjs<AX_ISO, true>(Tbar, Cibar, ybar, T, Ci, ek, g, s);
    if (ek.axes == AX_COMMON) return launch_adjs<AX_COMMON, true>(Tbar, Cibar, ybar, T, Ci, ek, g, s);
    return launch_adjs<AX_SPREAD, true>(Tbar, Cibar, ybar, T, Ci, ek, g, s);
}

unsigned adjoint_scaled_device_error(bool clear) {
    unsigned v = 0;
    cudaMemcpyFromSymbol(&v, g_adjs_error, sizeof(v));
    if (clear) {
        const unsigned z = 0;
        cudaMemcpyToSymbol(g_adjs_error, &z, sizeof(z));
    }
    return v;
}

}  // namespace psd
