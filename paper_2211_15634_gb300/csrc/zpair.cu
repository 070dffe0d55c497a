// FP32 steps fused in pairs over a single grid: T2 = step(step(T)) in one pass, one read of T
// and Ci and one write of T2 (temporal blocking of depth 2).
//
// What binds.  One step at a time moves 12 bytes per node (228 us at 512^3, the copy rate).
// A pair moves the same for two steps, so it must not cost more than about 60 instructions
// per node to stay with the memory.  A thread therefore steps eight nodes (four along x in each
// of two rows) with packed FP32 arithmetic (f32x2, the same roundings as f32_node), shares the
// first differences along x between neighbours and along z between planes, and its loop's own
// instructions count for eight nodes.  Measured (us a step): 512^3 130.9, 384^3 57.4, 256^3
// 18.8, where the four-node form with a scalar ring around the tile (zmarch2_tile.cuh, 95
// instructions per node and pass against 45) took 179, 82.8 and 27.6.  Four nodes per thread
// with halo rows and columns in whole warps and lanes took 188 at 512^3 (the 120 columns that
// leaves waste a seventh of the lanes), and passes of three and four steps in that form 215
// and 372 per step's share: more levels cost more instructions than the memory they save.
//
// Layout.  A CTA owns 128 x BY output nodes and a chunk of planes [k0, k1).  Warp w steps rows
// 2w and 2w+1 of the BY + 2 rows from Y0-1; level 1 (the state after one step) is formed on all
// of them, level 2 stored from the inner BY.  Iteration z steps level 1 at plane z+1 and level 2
// at plane z: a node itself and its z-neighbours are the thread's registers, the x-neighbours
// the thread's or its neighbour lanes' (shuffles), the y-neighbours the thread's other row or
// shared memory - T's plane in its stage, level 1's tile of plane z, written one iteration
// earlier (two slots).  Level 1 in the columns beside the tile (X0-1 and X0+128) is formed
// by one more warp, a row per lane.  One barrier per iteration.  T plane q (BY + 4 rows) and
// Ci plane q-1 (BY + 2 rows) arrive by TMA in one stage on one mbarrier, used in iterations
// q-2 and (T's x- and y-neighbours) q-1; Ci moves to level 2 in registers.
// Level 1 of a node that is not interior is its level 0: its rate of change (Ci times the bracket of
// f32_node) is replaced by the zero that leaves every value as it is.  Not its Ci: the bracket reads
// the zeros outside the grid and the nodes beside it in the face, so it may be infinite or NaN
// where every value that an interior stencil reads is finite.  Replacing the rate rather than
// selecting between the old and the new value keeps the old one from being held longer (us a step,
// on one GPU: 512^3 130.9 with the rate, 137.2 with Ci, 142.7 with the value; 256^3 18.8, 19.7, 20.4).
#include <cudaTypedefs.h>

#include "f32x2.cuh"
#include "internal.h"
#include "node.cuh"
#include "pdl.cuh"
#include "tma.cuh"
#include "waves.h"
#include "zmarch.h"

namespace psd {

__device__ unsigned g_zpair_error;  // set when an mbarrier wait times out

struct ZPairParams {
    int nx, ny, nz, kchunk, ntx;
    float dtlam, ax, ay, az;
};

__device__ __forceinline__ V4 v4_load(const float *p) {
    const ulonglong2 v = *(const ulonglong2 *)p;
    return V4{v.x, v.y};
}
__device__ __forceinline__ void v4_store(float *p, V4 v) { *(ulonglong2 *)p = make_ulonglong2(v.a, v.b); }
// x, with y's first node where f0 and its last where f3.
__device__ __forceinline__ V4 v4_faces(V4 x, V4 y, bool f0, bool f3) {
    return V4{f2_make(f0 ? f2_lo(y.a) : f2_lo(x.a), f2_hi(x.a)), f2_make(f2_lo(x.b), f3 ? f2_hi(y.b) : f2_hi(x.b))};
}

// Ci times the bracket of f32_node, of four neighbouring nodes: c the centres, left / right the
// values beside them, up / dn the rows above and below, en = zp - c and eo = c - zm the differences
// along z.
__device__ __forceinline__ V4 v4_rate(V4 c, float left, float right, V4 up, V4 dn, V4 en, V4 eo, V4 ci,
                                      const ZCoef2 &k) {
    const float c0 = f2_lo(c.a), c1 = f2_hi(c.a), c2 = f2_lo(c.b), c3 = f2_hi(c.b);
    const float d0 = __fsub_rn(c0, left), d1 = __fsub_rn(c1, c0), d2 = __fsub_rn(c2, c1), d3 = __fsub_rn(c3, c2),
                d4 = __fsub_rn(right, c3);
    const f2 xa = f2_make(__fsub_rn(d1, d0), __fsub_rn(d2, d1)), xb = f2_make(__fsub_rn(d3, d2), __fsub_rn(d4, d3));
    const V4 y = v4_sub(v4_sub(dn, c), v4_sub(c, up)), z = v4_sub(en, eo);
    const f2 la = f2_fma(z.a, k.az, f2_fma(y.a, k.ay, f2_mul(xa, k.ax)));
    const f2 lb = f2_fma(z.b, k.az, f2_fma(y.b, k.ay, f2_mul(xb, k.ax)));
    return V4{f2_mul(ci.a, la), f2_mul(ci.b, lb)};
}
__device__ __forceinline__ V4 v4_add(V4 c, V4 rate, const ZCoef2 &k) {
    return V4{f2_fma(k.dtlam, rate.a, c.a), f2_fma(k.dtlam, rate.b, c.b)};
}

template <int BY>
struct ZPair {
    static constexpr int BX = 128, W = BX + 8, ROWS = BY + 2, TROWS = BY + 4, NW = ROWS / 2;
    static_assert(BY % 2 == 0 && ROWS <= 16, "two rows per warp, a halo row per lane of half a warp");
    static constexpr unsigned TB = (TROWS * W * 4 + 127) / 128 * 128, CB = (ROWS * W * 4 + 127) / 128 * 128;
    static constexpr unsigned SB = TB + CB, LB = CB;  // stage, level-1 tile slot
    static constexpr int NTH = 32 * (NW + 1);
};

// kStates: level 1 goes to T1o too, and T1o and T2 are written at every node of the output
// rows, boundary nodes as T's.
template <int BY, int NST, int MINB, bool kStates>
__global__ void __launch_bounds__(ZPair<BY>::NTH, MINB)
k_zpair(const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmC, float *__restrict__ T2,
        const ZPairParams p, float *__restrict__ T1o) {
    using Z = ZPair<BY>;
    constexpr int W = Z::W, ROWS = Z::ROWS, NW = Z::NW;
    constexpr int LBF = Z::LB / 4, CF = Z::TB / 4;
    extern __shared__ __align__(128) unsigned char smem[];
    float *tiles = (float *)(smem + NST * Z::SB);  // level 1 of plane q in slot q % 2
    uint64_t *bar = (uint64_t *)(smem + NST * Z::SB + 2 * Z::LB);
    __shared__ int s_abort;
    grid_dep_wait();  // the previous launch's writes (and its reads of T2) are complete
    grid_dep_launch();

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int X0 = (int)(blockIdx.x % p.ntx) * Z::BX, Y0 = (int)(blockIdx.x / p.ntx) * BY;
    const int k0 = 1 + (int)blockIdx.y * p.kchunk, k1 = min(k0 + p.kchunk, nz - 1);  // output planes

    // stage j % NST: T plane k0 - 2 + j, and for j >= 2 Ci plane k0 - 3 + j
    const int jmax = k1 - k0 + 3;
    auto issue = [&](int j) {
        const int s = j % NST, q = k0 - 2 + j;
        unsigned char *st = smem + s * Z::SB;
        mbar_expect_tx(&bar[s], Z::TROWS * W * 4 + (j >= 2 ? ROWS * W * 4 : 0));
        tma_load_3d(st, &tmT, &bar[s], X0 - 4, Y0 - 2, q);
        if (j >= 2) tma_load_3d(st + Z::TB, &tmC, &bar[s], X0 - 4, Y0 - 1, q - 1);
    };
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int j = 0; j < NST && j <= jmax; ++j) issue(j);
    // After a timed-out wait: bounded waits for the copies still in flight (stages up to j),
    // so that no TMA write lands after the CTA exits.
    auto drain = [&](int j) {
        for (int i = max(0, j - NST + 1); i <= j; ++i) mbar_wait(&bar[i % NST], (unsigned)(i / NST) & 1u);
    };
    bool ok = mbar_wait(&bar[0], 0u);
    ok = mbar_wait(&bar[1], 0u) && ok;
    int s1 = 1 % NST, s0 = 2 % NST;  // stages of T planes z+1 and z+2 (and Ci plane z+1)
    unsigned par = 3u;               // parity of each stage's next completion
    const int zfirst = k0 - 2;       // level 1 from plane k0 - 1 on

    if (w == NW) {
        // ---- the halo warp: level 1 at column X0-1 (lanes 0-15) and X0+128 (lanes 16-31),
        // tile row lane % 16
        const int r = min(lane & 15, ROWS - 1), hc = lane < 16 ? 3 : 4 + Z::BX;  // box column
        const int x = X0 - 4 + hc, y = Y0 - 1 + r;
        const bool in = x >= 1 && x <= nx - 2 && y >= 1 && y <= ny - 2;
        const bool put = (lane & 15) < ROWS;
        const int o = (r + 1) * W + hc;  // the node in a T box
        float c = ((const float *)(smem + Z::SB))[o], e = __fsub_rn(c, ((const float *)smem)[o]);
        __syncthreads();  // stage 0 is read
        int j = 2;
        for (int z = zfirst; z < k1; ++z, ++j) {
            ok = mbar_wait(&bar[s0], (par >> s0) & 1u) && ok;
            par ^= 1u << s0;
            const float *t0 = (const float *)(smem + s0 * Z::SB), *t1 = (const float *)(smem + s1 * Z::SB);
            const float zp = t0[o], en = __fsub_rn(zp, c), ci = t0[CF + r * W + hc];
            const float d2x = __fsub_rn(__fsub_rn(t1[o + 1], c), __fsub_rn(c, t1[o - 1]));
            const float d2y = __fsub_rn(__fsub_rn(t1[o + W], c), __fsub_rn(c, t1[o - W]));
            const float lap = __fmaf_rn(__fsub_rn(en, e), p.az, __fmaf_rn(d2y, p.ay, __fmul_rn(d2x, p.ax)));
            const float v = __fmaf_rn(p.dtlam, __fmul_rn(ci, lap), c);
            if (put) tiles[((z + 1) & 1) * LBF + r * W + hc] = in && z + 1 >= 1 && z + 1 <= nz - 2 ? v : c;
            e = en;
            c = zp;
            if (!ok) {
                s_abort = 1;
                atomicOr(&g_zpair_error, 1u);
            }
            __syncthreads();
            if (s_abort) return;  // warp 0 waits for the copies in flight
            s1 = s0;
            s0 = s0 + 1 == NST ? 0 : s0 + 1;
        }
        return;
    }

    // ---- rows ra = 2w and ra + 1 of the stepped rows (T box rows one more)
    const int ra = 2 * w, gya = Y0 - 1 + ra, gx0 = X0 + 4 * lane;
    const bool ina = gya >= 1 && gya <= ny - 2, inb = gya + 1 >= 1 && gya + 1 <= ny - 2;
    // rows are whole groups of four: only a lane's first and last node can be on an x face, and
    // a lane past the row's end has no node at all (what it forms is read by no interior node)
    const bool row = gx0 < nx, f0 = gx0 == 0, f3 = gx0 + 4 >= nx;
    const bool outa = w > 0 && (kStates ? gya <= ny - 1 : ina);
    const bool outb = w < NW - 1 && (kStates ? gya + 1 <= ny - 1 : inb);
    const ZCoef2 k{f2_make(p.dtlam, p.dtlam), f2_make(p.ax, p.ax), f2_make(p.ay, p.ay), f2_make(p.az, p.az)};
    // a rate that leaves every value as it is (its product with dtlam is -0)
    const f2 z2 = f2_make(copysignf(0.f, -p.dtlam), copysignf(0.f, -p.dtlam));
    const V4 still{z2, z2};
    const int oT = (ra + 1) * W + 4 + 4 * lane, oC = ra * W + 4 + 4 * lane;  // own nodes in a T box, in a Ci box or tile
    const int up1 = max(ra - 1, 0) * W + 4 + 4 * lane, dn1 = min(ra + 2, ROWS - 1) * W + 4 + 4 * lane;
    const bool eL = lane == 0, eR = lane == 31;
    const int oE = eR ? 4 : -1;  // from the own nodes to the value beside the tile (lanes 0, 31)

    V4 ca, cb, ea, eb;  // level 0 of plane z+1, and its difference to plane z
    {
        const float *t0 = (const float *)smem, *t1 = (const float *)(smem + Z::SB);
        ca = v4_load(t1 + oT);
        cb = v4_load(t1 + oT + W);
        ea = v4_sub(ca, v4_load(t0 + oT));
        eb = v4_sub(cb, v4_load(t0 + oT + W));
    }
    V4 c1a{0ull, 0ull}, c1b = c1a, e1a = c1a, e1b = c1a;  // level 1 of plane z, difference to z-1
    V4 cia = c1a, cib = c1a;                               // Ci of plane z
    __syncthreads();  // stage 0 (own rows only) is read
    if (threadIdx.x == 0 && NST <= jmax) issue(NST);

    // x-neighbours of a row held in registers; f: the row's own nodes in shared memory, whose
    // columns beside the tile lanes 0 and 31 read
    auto beside = [&](V4 v, const float *f, float &left, float &right) {
        float h = 0.f;
        if (eL || eR) h = f[oE];
        left = __shfl_up_sync(0xffffffffu, f2_hi(v.b), 1);
        right = __shfl_down_sync(0xffffffffu, f2_lo(v.a), 1);
        left = eL ? h : left;
        right = eR ? h : right;
    };
    int64_t base = (int64_t)gx0 + (int64_t)nx * ((int64_t)gya + (int64_t)ny * zfirst);
    const int64_t plane = (int64_t)nx * ny;
    int j = 2;
#pragma unroll 2
    for (int z = zfirst; z < k1; ++z, ++j, base += plane) {
        ok = mbar_wait(&bar[s0], (par >> s0) & 1u) && ok;
        par ^= 1u << s0;
        const float *t0 = (const float *)(smem + s0 * Z::SB), *t1 = (const float *)(smem + s1 * Z::SB);
        float *const w1 = tiles + ((z + 1) & 1) * LBF;     // level 1 of plane z+1
        const float *const w0 = tiles + (z & 1) * LBF;     // and of plane z
        // level 1 of plane z+1
        const V4 za = v4_load(t0 + oT), zb = v4_load(t0 + oT + W);
        const V4 na = v4_load(t0 + CF + oC), nb = v4_load(t0 + CF + oC + W);  // Ci of plane z+1
        const bool zin = z + 1 >= 1 && z + 1 <= nz - 2;
        const V4 ena = v4_sub(za, ca), enb = v4_sub(zb, cb);
        float la, ra_, lb, rb_;
        beside(ca, t1 + oT, la, ra_);
        beside(cb, t1 + oT + W, lb, rb_);
        V4 qa = v4_rate(ca, la, ra_, v4_load(t1 + oT - W), cb, ena, ea, na, k);
        V4 qb = v4_rate(cb, lb, rb_, ca, v4_load(t1 + oT + 2 * W), enb, eb, nb, k);
        if (!(ina && zin)) qa = still;
        if (!(inb && zin)) qb = still;
        qa = v4_faces(qa, still, f0, f3);
        qb = v4_faces(qb, still, f0, f3);
        const V4 oa = v4_add(ca, qa, k), ob = v4_add(cb, qb, k);
        v4_store(w1 + oC, oa);
        v4_store(w1 + oC + W, ob);
        ca = za;
        cb = zb;
        ea = ena;
        eb = enb;
        // level 2 of plane z
        const V4 fna = v4_sub(oa, c1a), fnb = v4_sub(ob, c1b);
        if (z >= k0) {
            beside(c1a, w0 + oC, la, ra_);
            beside(c1b, w0 + oC + W, lb, rb_);
            V4 ya = v4_add(c1a, v4_rate(c1a, la, ra_, v4_load(w0 + up1), c1b, fna, e1a, cia, k), k);
            V4 yb = v4_add(c1b, v4_rate(c1b, lb, rb_, c1a, v4_load(w0 + dn1), fnb, e1b, cib, k), k);
            if constexpr (kStates) {
                if (!ina) ya = c1a;
                if (!inb) yb = c1b;
                if (X0 == 0 || X0 + Z::BX > nx - 1) {  // CTA-uniform: x faces in the tile
                    ya = v4_faces(ya, c1a, f0, f3);
                    yb = v4_faces(yb, c1b, f0, f3);
                }
                if (outa && row) {
                    v4_store(T1o + base, c1a);
                    v4_store(T2 + base, ya);
                }
                if (outb && row) {
                    v4_store(T1o + base + nx, c1b);
                    v4_store(T2 + base + nx, yb);
                }
            } else {
                auto put = [&](float *t, V4 v) {
                    if (!(f0 || f3)) {
                        v4_store(t, v);
                    } else if (row) {
                        if (!f0) t[0] = f2_lo(v.a);
                        t[1] = f2_hi(v.a);
                        t[2] = f2_lo(v.b);
                        if (!f3) t[3] = f2_hi(v.b);
                    }
                };
                if (outa) put(T2 + base, ya);
                if (outb) put(T2 + base + nx, yb);
            }
        }
        c1a = oa;
        c1b = ob;
        e1a = fna;
        e1b = fnb;
        cia = na;
        cib = nb;
        if (!ok) {
            s_abort = 1;
            atomicOr(&g_zpair_error, 1u);
        }
        // level 1 of plane z+1 is complete, T plane z+1's stage no longer read
        __syncthreads();
        if (s_abort) {
            drain(min(j - 2 + NST, jmax));
            return;
        }
        if (threadIdx.x == 0 && j - 1 + NST <= jmax) issue(j - 1 + NST);
        s1 = s0;
        s0 = s0 + 1 == NST ? 0 : s0 + 1;
    }
}

// Planes per chunk for `tiles` tiles on `slots` resident CTAs.
int pair_kchunk(Grid3 g, int64_t tiles, int64_t slots) {
    int kchunk = launch_override(PS_OVERRIDE_KCHUNK2);
    if (kchunk <= 0) {
        const int64_t per_tile = tiles > 0 ? slots / tiles : 0;
        const int64_t one_wave = per_tile > 0 ? (g.nz - 2 + per_tile - 1) / per_tile : 0;
        if (one_wave <= 96 && one_wave > 0) {
            // all CTAs resident at once (112^3 5.4 us a step at 3 planes, 6.6 at 6; odd rows, 129^3 7.6
            // at 4, 7.1 at 5, 7.6 at 6)
            kchunk = (int)(one_wave < 3 ? 3 : one_wave);
        } else {
            // the chunk whose waves march the fewest planes in all (each chunk two and a half
            // more than it stores): 384^3 61 us a step at 40 planes, 67 at 35
            double best = 0.0;
            for (int c = 16; c <= 96; ++c) {
                const int64_t ctas = tiles * ((g.nz - 2 + c - 1) / c), waves = (ctas + slots - 1) / slots;
                const double cost = (double)waves * (c + 2.5);
                if (kchunk <= 0 || cost < best) {
                    best = cost;
                    kchunk = c;
                }
            }
        }
    }
    return grid_chunk(g.nz, kchunk);
}

template <int BY, int NST, int MINB, bool kStates>
static cudaError_t launch_pair_t(float *T1o, float *T2, const float *T, const float *Ci, StepCoef c, Grid3 g,
                                 cudaStream_t s) {
    using Z = ZPair<BY>;
    constexpr size_t smem = NST * Z::SB + 2 * Z::LB + NST * 8;
    static unsigned attr_gen[64] = {0};
    cudaError_t ae;
    if (!set_smem_attr_once((const void *)k_zpair<BY, NST, MINB, kStates>, (int)smem, attr_gen, &ae)) return ae;
    CUtensorMap mT, mC;
    if (!make_tensor_map_3d(&mT, T, 4, g, Z::W, Z::TROWS) || !make_tensor_map_3d(&mC, Ci, 4, g, Z::W, Z::ROWS))
        return cudaErrorInvalidValue;
    const int64_t ntx = (g.nx + Z::BX - 1) / Z::BX, nty = (g.ny + BY - 1) / BY, tiles = ntx * nty;
    const int kchunk = pair_kchunk(g, tiles, (int64_t)MINB * sm_count());
    const int64_t gz = (g.nz - 2 + kchunk - 1) / kchunk;
    if (tiles > 0x7fffffffLL || gz > 65535) return cudaErrorInvalidConfiguration;
    const ZPairParams p{(int)g.nx, (int)g.ny, (int)g.nz, kchunk, (int)ntx, (float)c.dtlam, (float)c.ax, (float)c.ay,
                        (float)c.az};
    return launch_pdl(k_zpair<BY, NST, MINB, kStates>, dim3((unsigned)tiles, (unsigned)gz, 1), dim3(Z::NTH), smem,
                      s, mT, mC, T2, p, T1o);
}

// 14-row tiles, four stages (91 KB), two CTAs per SM (96 registers).
cudaError_t launch_step2_f32(float *T2, const float *T, const float *Ci, StepCoef c, Grid3 g, cudaStream_t s) {
    return launch_pair_t<14, 4, 2, false>(nullptr, T2, T, Ci, c, g, s);
}

cudaError_t launch_step2_states_f32(float *T1o, float *T2, const float *T, const float *Ci, StepCoef c, Grid3 g,
                                    cudaStream_t s) {
    return launch_pair_t<14, 4, 2, true>(T1o, T2, T, Ci, c, g, s);
}

bool pairs_pay(Grid3 g, bool states) {
    const double x = (double)g.nx / (128.0 * (double)((g.nx + 127) / 128)),
                 y = (double)g.ny / (14.0 * (double)((g.ny + 13) / 14));
    // Rows of 14-row tiles that are used, against the one-step march's 8: thin grids take single steps (us a
    // step, single steps / pairs: 868 x 3 x 2734 18 / 28, 284 x 6 x 1323 5.4 / 8.2, 872 x 16 x 376 (0.57) 9.5 / 10.8,
    // 2328 x 18 x 184 (0.64) 14.8 / 13.6, 1816 x 10 x 2092 (0.71) 73 / 56).
    if (y < 0.6) return false;
    const double n = (double)g.n(), useful = n * x * y;
    // loops that keep every state (us a step, single steps / pairs): 128^3 6.0 / 7.1, 160^3 (0.63) 13.1
    // / 9.9, 256^3 33.8 / 22.7
    if (states) return useful > 2.2e6;
    // By nodes and the share of useful lanes against the column kernel's, which steps small grids
    // and wastes at most 31 columns (us a step, single steps / pairs): 108 x 48 x 128 (0.84 of the
    // lanes) 3.8 / 4.1, 104^3 5.5 / 4.3, 128^3 5.6 / 5.2, 72 x 300 x 200 (0.56, the column kernel's
    // 0.75) 12.3 / 11.0, 160^3 (0.63, 1.0) 8.9 / 9.7, 192^3 13.0 / 12.4, 144 x 250 x 250 24.3 / 18.7,
    // 372 x 96 x 96 9.6 / 6.3.  Over 174 shapes of 3 to 6000 nodes an axis 0.9% off the better of the two
    // on average.
    const double column = (double)g.nx / (32.0 * (double)((g.nx + 31) / 32));
    return x < 0.65 * column ? n > 7.5e6 && useful > 2.8e6 : useful > 7.5e5;
}

unsigned zpair_device_error(bool clear) {
    unsigned v = 0;
    cudaMemcpyFromSymbol(&v, g_zpair_error, sizeof(v));
    if (clear) {
        const unsigned z = 0;
        cudaMemcpyToSymbol(g_zpair_error, &z, sizeof(z));
    }
    return v;
}

}  // namespace psd
