// FP32 step pairs (zpair.cu) on rows that are no multiple of 16 bytes.
//
// Layout.  As k_zpair - a CTA marches a tile of 128 x BY output nodes, eight nodes per thread in
// two rows, level 1 of the columns beside the tile in one more warp - but tiles start at x = 1
// and a lane's nodes of a row are 32 apart, so that shared memory is read at any element
// without bank conflicts.  Rows r = y + ny*z of one residue mod 4 are a multiple of 16 bytes
// apart, and all start at the same element of their 16 bytes: one tensor map per residue, based
// at the 16-byte boundary before its first row, loads every fourth row of the box in one copy
// (four copies per plane and field; a copy per row took as long as the arithmetic).  Row r then
// lies r*nx mod 4 elements to the right in the box.
//
// What binds.  Issue, as in k_zpair, with a load per node instead of per four (two more for the
// x-neighbours).  us a step, single steps (k_zmarch_rag) / pairs: 255^3 33.4 / 22.5, 321^3
// 66.9 / 50.9, 383^3 101.5 / 71, 511^3 231 / 157; three stages 4% slower, the loop unrolled
// once or twice instead of four times 6% and 2%.
#include <cudaTypedefs.h>

#include "f32x2.cuh"
#include "internal.h"
#include "pdl.cuh"
#include "tma.cuh"
#include "zmarch.h"

namespace psd {

__device__ unsigned g_zpair_rag_error;  // set when an mbarrier wait times out

struct ZPairRagParams {
    int nx, ny, nz, kchunk, ntx;
    float dtlam, ax, ay, az;
};

template <int BY>
struct ZPairRag {
    static constexpr int BX = 128, W = BX + 12, W1 = BX + 4, ROWS = BY + 2, TROWS = BY + 4, NW = ROWS / 2;
    static_assert(BY % 2 == 0 && ROWS == 16, "two rows per warp, a halo row per lane of half a warp");
    static constexpr int TG = (TROWS + 3) / 4, CG = ROWS / 4;  // rows per copy
    // floats of a copy, 128-byte aligned
    static constexpr int TGF = (TG * W + 31) / 32 * 32, CGF = (CG * W + 31) / 32 * 32;
    static constexpr unsigned SB = 16 * (TGF + CGF);                  // stage
    static constexpr unsigned LB = (ROWS * W1 * 4 + 127) / 128 * 128;  // level-1 tile slot
    static constexpr int NTH = 32 * (NW + 1);
    // first float of box row q, before its shift
    static __device__ __forceinline__ int trow(int q) { return (q & 3) * TGF + (q >> 2) * W; }
    static __device__ __forceinline__ int crow(int q) { return 4 * TGF + (q & 3) * CGF + (q >> 2) * W; }
};

// f32_node of four nodes: l / r the x-neighbours, up / dn the rows above and below, en = zp - c and
// eo = c - zm the differences along z.
__device__ __forceinline__ V4 v4_step32(V4 c, V4 l, V4 r, V4 up, V4 dn, V4 en, V4 eo, V4 ci, const ZCoef2 &k) {
    const V4 x = v4_sub(v4_sub(r, c), v4_sub(c, l)), y = v4_sub(v4_sub(dn, c), v4_sub(c, up)), z = v4_sub(en, eo);
    const f2 la = f2_fma(z.a, k.az, f2_fma(y.a, k.ay, f2_mul(x.a, k.ax)));
    const f2 lb = f2_fma(z.b, k.az, f2_fma(y.b, k.ay, f2_mul(x.b, k.ax)));
    return V4{f2_fma(k.dtlam, f2_mul(ci.a, la), c.a), f2_fma(k.dtlam, f2_mul(ci.b, lb), c.b)};
}
__device__ __forceinline__ V4 v4_pick(const bool (&m)[4], V4 x, V4 y) {
    return V4{f2_make(m[0] ? f2_lo(x.a) : f2_lo(y.a), m[1] ? f2_hi(x.a) : f2_hi(y.a)),
              f2_make(m[2] ? f2_lo(x.b) : f2_lo(y.b), m[3] ? f2_hi(x.b) : f2_hi(y.b))};
}

template <int BY, int NST, int MINB>
__global__ void __launch_bounds__(ZPairRag<BY>::NTH, MINB)
k_zpair_rag(const __grid_constant__ RagMaps<2> maps, float *__restrict__ T2, const ZPairRagParams p) {
    using Z = ZPairRag<BY>;
    constexpr int W1 = Z::W1, ROWS = Z::ROWS, NW = Z::NW, LBF = Z::LB / 4;
    extern __shared__ __align__(128) unsigned char smem[];
    float *tiles = (float *)(smem + NST * Z::SB);  // level 1 of plane q in slot q % 2
    uint64_t *bar = (uint64_t *)(smem + NST * Z::SB + 2 * Z::LB);
    __shared__ int s_abort;
    grid_dep_wait();  // the previous launch's writes (and its reads of T2) are complete
    grid_dep_launch();

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int xt = (int)(blockIdx.x % p.ntx) * Z::BX;
    const int X0 = 1 + xt, Y0 = 1 + (int)(blockIdx.x / p.ntx) * BY;
    const int k0 = 1 + (int)blockIdx.y * p.kchunk, k1 = min(k0 + p.kchunk, nz - 1);  // output planes

    // stage j % NST: T plane k0 - 2 + j (rows Y0 - 2 ..), and for j >= 2 Ci plane k0 - 3 + j (rows
    // Y0 - 1 ..); element x of a row with shift s at column x - X0 + 5 + s
    const int jmax = k1 - k0 + 3;
    auto issue = [&](int j) {
        const int s = j % NST, q = k0 - 2 + j;
        float *st = (float *)(smem + s * Z::SB);
        mbar_expect_tx(&bar[s], 16 * Z::W * (Z::TG + (j >= 2 ? Z::CG : 0)));
        const int r = q * ny + Y0 - 2, rc = r - ny + 1;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            tma_load_2d(st + i * Z::TGF, &maps.f[0][(r + i) & 3], &bar[s], xt - 4, (r + i) >> 2);
        if (j >= 2)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                tma_load_2d(st + 4 * Z::TGF + i * Z::CGF, &maps.f[1][(rc + i) & 3], &bar[s], xt - 4, (rc + i) >> 2);
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
    // shift of box row q of T plane z: sh(plane base, q); the base of the plane after it is
    // step further (Ci's row q is T's row q + 1 of its plane)
    const int n3 = nx & 3, step = (ny & 3) * n3;
    int b = ((zfirst & 3) * (ny & 3) + Y0 - 2) * n3;  // of plane zfirst
    auto sh = [&](int base, int q) { return (base + q * n3) & 3; };

    if (w == NW) {
        // ---- the halo warp: level 1 at column X0-1 (lanes 0-15) and X0+128 (lanes 16-31),
        // tile row lane % 16
        const int r = lane & 15, hx = lane < 16 ? -1 : Z::BX;
        const int x = X0 + hx, y = Y0 - 1 + r;
        const bool in = x >= 1 && x <= nx - 2 && y >= 1 && y <= ny - 2;
        const int q1 = Z::trow(r + 1) + 5 + hx, qu = Z::trow(r) + 5 + hx, qd = Z::trow(r + 2) + 5 + hx;
        const int qc = Z::crow(r) + 5 + hx;
        const float *f0 = (const float *)smem, *f1 = (const float *)(smem + Z::SB);
        float e = f0[q1 + sh(b, r + 1)];
        b = (b + step) & 3;
        float c = f1[q1 + sh(b, r + 1)];
        e = __fsub_rn(c, e);
        __syncthreads();  // stage 0 is read
        int j = 2;
        for (int z = zfirst; z < k1; ++z, ++j) {
            ok = mbar_wait(&bar[s0], (par >> s0) & 1u) && ok;
            par ^= 1u << s0;
            const float *t0 = (const float *)(smem + s0 * Z::SB), *t1 = (const float *)(smem + s1 * Z::SB);
            const int o = sh(b, r + 1), ou = qu + sh(b, r), od = qd + sh(b, r + 2);
            b = (b + step) & 3;
            const float zp = t0[q1 + sh(b, r + 1)], en = __fsub_rn(zp, c), ci = t0[qc + o];
            const float d2x = __fsub_rn(__fsub_rn(t1[q1 + o + 1], c), __fsub_rn(c, t1[q1 + o - 1]));
            const float d2y = __fsub_rn(__fsub_rn(t1[od], c), __fsub_rn(c, t1[ou]));
            const float lap = __fmaf_rn(__fsub_rn(en, e), p.az, __fmaf_rn(d2y, p.ay, __fmul_rn(d2x, p.ax)));
            const float v = __fmaf_rn(p.dtlam, __fmul_rn(ci, lap), c);
            tiles[((z + 1) & 1) * LBF + r * W1 + 1 + hx] = in && z + 1 >= 1 && z + 1 <= nz - 2 ? v : c;
            e = en;
            c = zp;
            if (!ok) {
                s_abort = 1;
                atomicOr(&g_zpair_rag_error, 1u);
            }
            __syncthreads();
            if (s_abort) return;  // warp 0 waits for the copies in flight
            s1 = s0;
            s0 = s0 + 1 == NST ? 0 : s0 + 1;
        }
        return;
    }

    // ---- rows ra = 2w and ra + 1 of the stepped rows (T box rows one more)
    const int ra = 2 * w, gya = Y0 - 1 + ra, gx0 = X0 + lane;
    const bool ina = gya >= 1 && gya <= ny - 2, inb = gya + 1 >= 1 && gya + 1 <= ny - 2;
    const bool xedge = X0 + Z::BX > nx - 1;  // CTA-uniform: columns past the interior in the tile
    bool in[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) in[i] = gx0 + 32 * i <= nx - 2;
    const bool outa = w > 0 && ina, outb = w < NW - 1 && inb;
    const ZCoef2 k{f2_make(p.dtlam, p.dtlam), f2_make(p.ax, p.ax), f2_make(p.ay, p.ay), f2_make(p.az, p.az)};
    // a lane's first node in box rows ra .. ra + 3 of T and ra, ra + 1 of Ci, before the shift
    const int q0 = Z::trow(ra) + 5 + lane, q1 = Z::trow(ra + 1) + 5 + lane, q2 = Z::trow(ra + 2) + 5 + lane,
              q3 = Z::trow(ra + 3) + 5 + lane;
    const int qc = Z::crow(ra) + 5 + lane, qd = Z::crow(ra + 1) + 5 + lane;
    const int oC = ra * W1 + 1 + lane;  // own nodes in a level-1 tile
    const int up1 = max(ra - 1, 0) * W1 + 1 + lane, dn1 = min(ra + 2, ROWS - 1) * W1 + 1 + lane;

    V4 ca, cb, ea, eb;  // level 0 of plane z+1, and its difference to plane z
    {
        const float *t0 = (const float *)smem, *t1 = (const float *)(smem + Z::SB);
        ea = v4_load32(t0 + q1 + sh(b, ra + 1));
        eb = v4_load32(t0 + q2 + sh(b, ra + 2));
        b = (b + step) & 3;  // of plane z+1
        ca = v4_load32(t1 + q1 + sh(b, ra + 1));
        cb = v4_load32(t1 + q2 + sh(b, ra + 2));
        ea = v4_sub(ca, ea);
        eb = v4_sub(cb, eb);
    }
    V4 c1a{0ull, 0ull}, c1b = c1a, e1a = c1a, e1b = c1a;  // level 1 of plane z, difference to z-1
    V4 cia = c1a, cib = c1a;                               // Ci of plane z
    __syncthreads();  // stage 0 (own rows only) is read
    if (threadIdx.x == 0 && NST <= jmax) issue(NST);

    int64_t base = (int64_t)gx0 + (int64_t)nx * ((int64_t)gya + (int64_t)ny * zfirst);
    const int64_t plane = (int64_t)nx * ny;
    int j = 2;
#pragma unroll 4
    for (int z = zfirst; z < k1; ++z, ++j, base += plane) {
        ok = mbar_wait(&bar[s0], (par >> s0) & 1u) && ok;
        par ^= 1u << s0;
        const float *t0 = (const float *)(smem + s0 * Z::SB), *t1 = (const float *)(smem + s1 * Z::SB);
        float *const w1 = tiles + ((z + 1) & 1) * LBF;     // level 1 of plane z+1
        const float *const w0 = tiles + (z & 1) * LBF;     // and of plane z
        // level 1 of plane z+1
        const int s_a = sh(b, ra + 1), s_b = sh(b, ra + 2);
        const float *const tu = t1 + q0 + sh(b, ra), *const td = t1 + q3 + sh(b, ra + 3);
        const float *const ta = t1 + q1 + s_a, *const tb = t1 + q2 + s_b;
        b = (b + step) & 3;
        const bool zin = z + 1 >= 1 && z + 1 <= nz - 2;
        const V4 na = v4_load32(t0 + qc + s_a), nb = v4_load32(t0 + qd + s_b);  // Ci of plane z+1
        const V4 za = v4_load32(t0 + q1 + sh(b, ra + 1)), zb = v4_load32(t0 + q2 + sh(b, ra + 2));
        const V4 ena = v4_sub(za, ca), enb = v4_sub(zb, cb);
        V4 oa = v4_step32(ca, v4_load32(ta - 1), v4_load32(ta + 1), v4_load32(tu), cb, ena, ea, na, k);
        V4 ob = v4_step32(cb, v4_load32(tb - 1), v4_load32(tb + 1), ca, v4_load32(td), enb, eb, nb, k);
        if (!(ina && zin)) oa = ca;
        if (!(inb && zin)) ob = cb;
        if (xedge) {
            oa = v4_pick(in, oa, ca);
            ob = v4_pick(in, ob, cb);
        }
        auto tile = [&](float *f, V4 v) {
            f[0] = f2_lo(v.a);
            f[32] = f2_hi(v.a);
            f[64] = f2_lo(v.b);
            f[96] = f2_hi(v.b);
        };
        tile(w1 + oC, oa);
        tile(w1 + oC + W1, ob);
        ca = za;
        cb = zb;
        ea = ena;
        eb = enb;
        // level 2 of plane z
        const V4 fna = v4_sub(oa, c1a), fnb = v4_sub(ob, c1b);
        if (z >= k0) {
            const float *const va = w0 + oC, *const vb = va + W1;
            auto put = [&](float *t, V4 v) {
                if (in[0]) t[0] = f2_lo(v.a);
                if (in[1]) t[32] = f2_hi(v.a);
                if (in[2]) t[64] = f2_lo(v.b);
                if (in[3]) t[96] = f2_hi(v.b);
            };
            if (outa)
                put(T2 + base, v4_step32(c1a, v4_load32(va - 1), v4_load32(va + 1), v4_load32(w0 + up1), c1b, fna,
                                         e1a, cia, k));
            if (outb)
                put(T2 + base + nx, v4_step32(c1b, v4_load32(vb - 1), v4_load32(vb + 1), c1a, v4_load32(w0 + dn1),
                                              fnb, e1b, cib, k));
        }
        c1a = oa;
        c1b = ob;
        e1a = fna;
        e1b = fnb;
        cia = na;
        cib = nb;
        if (!ok) {
            s_abort = 1;
            atomicOr(&g_zpair_rag_error, 1u);
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

template <int BY, int NST, int MINB>
static cudaError_t launch_pair_rag_t(float *T2, const float *T, const float *Ci, StepCoef c, Grid3 g, cudaStream_t s) {
    using Z = ZPairRag<BY>;
    constexpr size_t smem = NST * Z::SB + 2 * Z::LB + NST * 8;
    static unsigned attr_gen[64] = {0};
    cudaError_t ae;
    if (!set_smem_attr_once((const void *)k_zpair_rag<BY, NST, MINB>, (int)smem, attr_gen, &ae)) return ae;
    RagMaps<2> maps;
    for (int m = 0; m < 4; ++m)
        if (!make_tensor_map_quarter(&maps.f[0][m], T, g, m, Z::W, Z::TG) ||
            !make_tensor_map_quarter(&maps.f[1][m], Ci, g, m, Z::W, Z::CG))
            return cudaErrorInvalidValue;
    const int64_t ntx = (g.nx - 2 + Z::BX - 1) / Z::BX, nty = (g.ny - 2 + BY - 1) / BY, tiles = ntx * nty;
    const int kchunk = pair_kchunk(g, tiles, (int64_t)MINB * sm_count());
    const int64_t gz = (g.nz - 2 + kchunk - 1) / kchunk;
    if (tiles > 0x7fffffffLL || gz > 65535) return cudaErrorInvalidConfiguration;
    const ZPairRagParams p{(int)g.nx, (int)g.ny, (int)g.nz, kchunk, (int)ntx, (float)c.dtlam, (float)c.ax, (float)c.ay,
                           (float)c.az};
    return launch_pdl(k_zpair_rag<BY, NST, MINB>, dim3((unsigned)tiles, (unsigned)gz, 1), dim3(Z::NTH), smem, s, maps,
                      T2, p);
}

// 14-row tiles, two CTAs per SM.
cudaError_t launch_step2_ragged_f32(float *T2, const float *T, const float *Ci, StepCoef c, Grid3 g, cudaStream_t s) {
    return launch_pair_rag_t<14, 4, 2>(T2, T, Ci, c, g, s);
}

bool pairs_pay_ragged(Grid3 g) {
    // By the useful nodes of 128 x 14 tiles.  Up to 8.8 million nodes single steps are the column kernel's, whose
    // fields stay in L2, so pairs need rows that fill three quarters of a tile and 0.6 of
    // its height; from there on both read HBM (us a step, single steps / pairs, shares in x
    // and y): 103^3 (0.79, 0.90) 5.4 / 4.7, 102 x 75 x 208 (0.78, 0.87) 5.6 / 5.1, 159^3 (0.61, 0.93) 8.9 / 10.9, 299 x
    // 256 x 64 (0.77, 0.95) 10.8 / 10.3, 87 x 128 x 387 (0.66, 1) 9.5 / 10, 625 x 5 x 980 (0.97, 0.21) 6.2 / 11, 113 x 18 x
    // 588 (0.87, 0.57) 4.5 / 4.9, 1697 x 12 x 800 (0.95, 0.71) 39 / 27, 129 x 18 x 4932 (0.99, 0.57) 24.6 / 23, 1061 x 6 x
    // 4776 (0.92, 0.29) 65 / 79, 143 x 250 x 250 (0.55, 0.98) 24.7 / 21.3, 255^3 33.4 / 22.5.  Over 186 shapes 0.3%
    // off the better of the two on average.
    const double n = (double)g.n(), x = (double)(g.nx - 2) / (128.0 * (double)((g.nx - 2 + 127) / 128)),
                 y = (double)(g.ny - 2) / (14.0 * (double)((g.ny - 2 + 13) / 14)), share = x * y;
    return n > 8.8e6 ? share >= 0.5 : x >= 0.75 && y >= 0.6 && n * share * share > 6e5;
}

unsigned zpair_rag_device_error(bool clear) {
    unsigned v = 0;
    cudaMemcpyFromSymbol(&v, g_zpair_rag_error, sizeof(v));
    if (clear) {
        const unsigned z = 0;
        cudaMemcpyToSymbol(g_zpair_rag_error, &z, sizeof(z));
    }
    return v;
}

}  // namespace psd
