// FP32 step of the two-float state (comp32_node) on rows that are no multiple of 16 bytes.
//
// Layout.  A CTA marches a tile of 128 x 16 nodes from x = 1, y = 1 on, eight nodes per thread: two
// rows, a lane's nodes of a row 32 apart, so that shared memory is read at any element without bank
// conflicts.  The state's two fields (18 rows) and Ci (16) arrive by TMA, four copies each, every
// fourth row of a box by one map (zpair_rag.cu says why).  Packed FP32 arithmetic, comp32_node's
// roundings.
//
// What binds: memory from 40 million nodes on, 20 bytes a node (511^3 400 us, 6.7 TB/s), latency and
// the last wave below.  us a step, plain column kernel / this: 511^3 557 / 400, 383^3 268 / 177, 255^3
// 103 / 58, 193^3 41 / 31, 129^3 11.3 / 9.9.
#include <cudaTypedefs.h>

#include "f32x2.cuh"
#include "internal.h"
#include "pdl.cuh"
#include "tma.cuh"
#include "waves.h"
#include "zmarch.h"

namespace psd {

__device__ unsigned g_comp_rag_error;  // set when an mbarrier wait times out

struct CompRagParams {
    int nx, ny, nz, kchunk, ntx;
    int eb;  // first element of E in its 16 bytes (T and Ci start there)
    float dtlam, ax, ay, az;
};

struct CompRag {
    static constexpr int BX = 128, BY = 16, H = BY + 2, W = BX + 12, NST = 3, MINB = 2;
    static constexpr int TG = (H + 3) / 4, CG = BY / 4;  // rows per copy
    // floats of a copy, 128-byte aligned; T's four, E's, Ci's
    static constexpr int TGF = (TG * W + 31) / 32 * 32, CGF = (CG * W + 31) / 32 * 32;
    static constexpr int EO = 4 * TGF, CO = 8 * TGF;
    static constexpr unsigned SB = 4 * (8 * TGF + 4 * CGF);  // stage
    // first float of box row q, before its shift
    static __device__ __forceinline__ int trow(int q) { return (q & 3) * TGF + (q >> 2) * W; }
    static __device__ __forceinline__ int crow(int q) { return CO + (q & 3) * CGF + (q >> 2) * W; }
};

__device__ __forceinline__ V4 v4_lap(V4 c, V4 l, V4 r, V4 up, V4 dn, V4 en, V4 eo, const ZCoef2 &k) {
    const V4 x = v4_sub(v4_sub(r, c), v4_sub(c, l)), y = v4_sub(v4_sub(dn, c), v4_sub(c, up)), z = v4_sub(en, eo);
    return V4{f2_fma(z.a, k.az, f2_fma(y.a, k.ay, f2_mul(x.a, k.ax))),
              f2_fma(z.b, k.az, f2_fma(y.b, k.ay, f2_mul(x.b, k.ax)))};
}
// comp32_node's update of two nodes: the new D, and the new correction to *e2.
__device__ __forceinline__ f2 comp_update(f2 c, f2 ec, f2 lapD, f2 lapE, f2 ci, f2 dtlam, f2 *e2) {
    const f2 q = f2_mul(ci, f2_add(lapD, lapE));
    // (scalar: the packed product would be fused with the sum)
    const f2 s = f2_add(ec, f2_make(__fmul_rn(f2_lo(dtlam), f2_lo(q)), __fmul_rn(f2_hi(dtlam), f2_hi(q))));
    const f2 t = f2_add(c, s), bp = f2_sub(t, c), ap = f2_sub(t, bp);
    *e2 = f2_add(f2_sub(c, ap), f2_sub(s, bp));
    return t;
}

__global__ void __launch_bounds__(16 * CompRag::BY, CompRag::MINB)
k_comp_rag(const __grid_constant__ RagMaps<3> maps, float *__restrict__ T2, float *__restrict__ E2,
           const CompRagParams p) {
    using Z = CompRag;
    constexpr int NST = Z::NST;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = (uint64_t *)(smem + NST * Z::SB);
    __shared__ int s_abort;
    grid_dep_wait();  // the previous step's writes (and its reads of T2 and E2) are complete
    grid_dep_launch();

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int xt = (int)(blockIdx.x % p.ntx) * Z::BX;
    const int X0 = 1 + xt, Y0 = 1 + (int)(blockIdx.x / p.ntx) * Z::BY;
    const int k0 = 1 + (int)blockIdx.y * p.kchunk, k1 = min(k0 + p.kchunk, nz - 1);  // output planes

    // plane q (k0-1 .. k1) in stage s: rows Y0 - 1 .. of T and E, and of an output plane rows Y0 ..
    // of Ci; element x of a row with shift d at column x - X0 + 5 + d
    auto issue = [&](int s, int q) {
        const bool ci = q >= k0 && q < k1;
        float *st = (float *)(smem + s * Z::SB);
        mbar_expect_tx(&bar[s], 16 * Z::W * (2 * Z::TG + (ci ? Z::CG : 0)));
        const int r = q * ny + Y0 - 1;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            tma_load_2d(st + i * Z::TGF, &maps.f[0][(r + i) & 3], &bar[s], xt - 4, (r + i) >> 2);
            tma_load_2d(st + Z::EO + i * Z::TGF, &maps.f[1][(r + i) & 3], &bar[s], xt - 4, (r + i) >> 2);
        }
        if (ci)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                tma_load_2d(st + Z::CO + i * Z::CGF, &maps.f[2][(r + 1 + i) & 3], &bar[s], xt - 4, (r + 1 + i) >> 2);
    };
    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int s = 0; s < NST; ++s)
            if (k0 - 1 + s <= k1) issue(s, k0 - 1 + s);
    unsigned par = 0u;  // bit s: parity of the next completion of stage s
    auto acquire = [&](int s) -> bool {
        const unsigned ph = (par >> s) & 1u;
        par ^= 1u << s;
        return mbar_wait(&bar[s], ph);
    };
    // After a timed-out wait: bounded waits for the copies of the last NST planes issued
    // (up to plane q_iss), so that no TMA write lands after the CTA exits.
    auto drain = [&](int q_iss) {
        for (int q = max(k0 - 1, q_iss - NST + 1); q <= q_iss; ++q) {
            const int i = q - (k0 - 1);
            mbar_wait(&bar[i % NST], (unsigned)(i / NST) & 1u);
        }
    };
    auto stage = [&](int s) { return (const float *)(smem + s * Z::SB); };

    // shift of box row q of a plane: (b + q * n3) mod 4, b that of its first row
    const int n3 = nx & 3, step = (ny & 3) * n3;
    int b = (((k0 - 1) & 3) * (ny & 3) + Y0 - 1) * n3;
    auto sh = [&](int base, int q) { return (base + q * n3) & 3; };
    const int eb = p.eb;  // E's rows lie eb further (mod 4)
    const int ra = 2 * w;  // rows ra and ra + 1 of the tile, ra + 1 and ra + 2 of a T box
    const int q0 = Z::trow(ra) + 5 + lane, q1 = Z::trow(ra + 1) + 5 + lane, q2 = Z::trow(ra + 2) + 5 + lane,
              q3 = Z::trow(ra + 3) + 5 + lane;
    const int qc = Z::crow(ra) + 5 + lane, qd = Z::crow(ra + 1) + 5 + lane;
    const int gy = Y0 + ra, gx0 = X0 + lane;
    bool in[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) in[i] = gx0 + 32 * i <= nx - 2;
    const bool outa = gy <= ny - 2, outb = gy + 1 <= ny - 2;
    const ZCoef2 k{f2_make(p.dtlam, p.dtlam), f2_make(p.ax, p.ax), f2_make(p.ay, p.ay), f2_make(p.az, p.az)};

    // [0] row ra, [1] row ra + 1: D and E of plane k, and their differences to plane k - 1
    V4 dc[2], ec[2], dd[2], ed[2];
    bool ok = acquire(0);
    {
        const float *t = stage(0);
        const int o0 = q1 + sh(b, ra + 1), o1 = q2 + sh(b, ra + 2);
        dd[0] = v4_load32(t + o0);
        dd[1] = v4_load32(t + o1);
        ed[0] = v4_load32(t + Z::EO + q1 + sh(b + eb, ra + 1));
        ed[1] = v4_load32(t + Z::EO + q2 + sh(b + eb, ra + 2));
    }
    ok = acquire(1) && ok;
    b = (b + step) & 3;
    {
        const float *t = stage(1);
        const int o0 = q1 + sh(b, ra + 1), o1 = q2 + sh(b, ra + 2);
        dc[0] = v4_load32(t + o0);
        dc[1] = v4_load32(t + o1);
        ec[0] = v4_load32(t + Z::EO + q1 + sh(b + eb, ra + 1));
        ec[1] = v4_load32(t + Z::EO + q2 + sh(b + eb, ra + 2));
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        dd[i] = v4_sub(dc[i], dd[i]);
        ed[i] = v4_sub(ec[i], ed[i]);
    }
    if (!ok) {
        s_abort = 1;
        atomicOr(&g_comp_rag_error, 1u);
    }
    __syncthreads();
    if (s_abort) {
        drain(min(k0 - 2 + NST, k1));
        return;
    }
    if (threadIdx.x == 0 && k0 - 1 + NST <= k1) issue(0, k0 - 1 + NST);  // stage 0 held plane k0-1
    int sk = 1;  // stage of plane k
    int64_t base = (int64_t)gx0 + (int64_t)nx * ((int64_t)gy + (int64_t)ny * k0);
    const int64_t plane = (int64_t)nx * ny;
    for (int kz = k0; kz < k1; ++kz, base += plane) {
        const int sn = sk + 1 == NST ? 0 : sk + 1;
        ok = acquire(sn);
        const float *tk = stage(sk), *tn = stage(sn);
        const int s0 = sh(b, ra + 1), s1 = sh(b, ra + 2), up = q0 + sh(b, ra), dn = q3 + sh(b, ra + 3);
        const int own[2] = {q1 + s0, q2 + s1}, co[2] = {qc + s0, qd + s1};
        const int eown[2] = {Z::EO + q1 + sh(b + eb, ra + 1), Z::EO + q2 + sh(b + eb, ra + 2)};
        const int eup = Z::EO + q0 + sh(b + eb, ra), edn = Z::EO + q3 + sh(b + eb, ra + 3);
        b = (b + step) & 3;
        const int nxt[2] = {q1 + sh(b, ra + 1), q2 + sh(b, ra + 2)};
        const int enxt[2] = {Z::EO + q1 + sh(b + eb, ra + 1), Z::EO + q2 + sh(b + eb, ra + 2)};
        V4 dz[2], ez[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            dz[i] = v4_load32(tn + nxt[i]);
            ez[i] = v4_load32(tn + enxt[i]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const float *t = tk + own[i], *e = tk + eown[i];
            const V4 dn_d = i == 0 ? dc[1] : v4_load32(tk + dn), up_d = i == 0 ? v4_load32(tk + up) : dc[0];
            const V4 dn_e = i == 0 ? ec[1] : v4_load32(tk + edn), up_e = i == 0 ? v4_load32(tk + eup) : ec[0];
            const V4 nd = v4_sub(dz[i], dc[i]), ne = v4_sub(ez[i], ec[i]);
            const V4 ld = v4_lap(dc[i], v4_load32(t - 1), v4_load32(t + 1), up_d, dn_d, nd, dd[i], k);
            const V4 le = v4_lap(ec[i], v4_load32(e - 1), v4_load32(e + 1), up_e, dn_e, ne, ed[i], k);
            const V4 ci = v4_load32(tk + co[i]);
            dd[i] = nd;
            ed[i] = ne;
            if (i == 0 ? outa : outb) {
                V4 e2;
                const f2 ta = comp_update(dc[i].a, ec[i].a, ld.a, le.a, ci.a, k.dtlam, &e2.a);
                const f2 tb = comp_update(dc[i].b, ec[i].b, ld.b, le.b, ci.b, k.dtlam, &e2.b);
                float *o = T2 + base + (i ? nx : 0), *oe = E2 + base + (i ? nx : 0);
                if (in[0]) o[0] = f2_lo(ta), oe[0] = f2_lo(e2.a);
                if (in[1]) o[32] = f2_hi(ta), oe[32] = f2_hi(e2.a);
                if (in[2]) o[64] = f2_lo(tb), oe[64] = f2_lo(e2.b);
                if (in[3]) o[96] = f2_hi(tb), oe[96] = f2_hi(e2.b);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            dc[i] = dz[i];
            ec[i] = ez[i];
        }
        if (!ok) {
            s_abort = 1;
            atomicOr(&g_comp_rag_error, 1u);
        }
        __syncthreads();  // every thread is done with plane k's stage
        if (s_abort) {
            drain(min(kz - 1 + NST, k1));
            return;
        }
        if (threadIdx.x == 0 && kz + NST <= k1) issue(sk, kz + NST);
        sk = sn;
    }
}

cudaError_t launch_comp_ragged(float *T2, const float *T, float *E2, const float *E, const float *Ci, StepCoef c,
                               Grid3 g, cudaStream_t s) {
    using Z = CompRag;
    constexpr size_t smem = Z::NST * Z::SB + Z::NST * 8;
    static unsigned attr_gen[64] = {0};
    cudaError_t ae;
    if (!set_smem_attr_once((const void *)k_comp_rag, (int)smem, attr_gen, &ae)) return ae;
    RagMaps<3> maps;
    for (int m = 0; m < 4; ++m)
        if (!make_tensor_map_quarter(&maps.f[0][m], T, g, m, Z::W, Z::TG) ||
            !make_tensor_map_quarter(&maps.f[1][m], E, g, m, Z::W, Z::TG) ||
            !make_tensor_map_quarter(&maps.f[2][m], Ci, g, m, Z::W, Z::CG))
            return cudaErrorInvalidValue;
    const int64_t ntx = (g.nx - 2 + Z::BX - 1) / Z::BX, nty = (g.ny - 2 + Z::BY - 1) / Z::BY, tiles = ntx * nty;
    int kchunk = launch_override(PS_OVERRIDE_KCHUNK);
    if (kchunk <= 0) kchunk = wave_chunk(g.nz - 2, tiles, sm_count(), Z::MINB, WaveCost{1.5, 0.6, 0.0, 3, 48});
    kchunk = grid_chunk(g.nz, kchunk);
    const int64_t gz = (g.nz - 2 + kchunk - 1) / kchunk;
    if (tiles > 0x7fffffffLL || gz > 65535) return cudaErrorInvalidConfiguration;
    const CompRagParams p{(int)g.nx, (int)g.ny, (int)g.nz, kchunk, (int)ntx, (int)(((uintptr_t)E >> 2) & 3), (float)c.dtlam, (float)c.ax, (float)c.ay,
                          (float)c.az};
    return launch_pdl(k_comp_rag, dim3((unsigned)tiles, (unsigned)gz, 1), dim3(16 * Z::BY), smem, s, maps, T2, E2, p);
}

unsigned comp_rag_device_error(bool clear) {
    unsigned v = 0;
    cudaMemcpyFromSymbol(&v, g_comp_rag_error, sizeof(v));
    if (clear) {
        const unsigned z = 0;
        cudaMemcpyToSymbol(g_comp_rag_error, &z, sizeof(z));
    }
    return v;
}

}  // namespace psd
