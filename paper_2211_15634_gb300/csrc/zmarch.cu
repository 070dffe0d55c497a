// Tiled z-march step kernels fed by TMA over a single grid: CTA (tile, chunk)
// runs the z-march tile body of zmarch_tile.cuh on its x-y tile and z-chunk.
//
// Preconditions (checked by the host launcher, else the plain kernel runs):
// nx*sizeof(elem) is a multiple of 16 (TMA row pitch) and all base pointers
// are 16-byte aligned.
#include <cudaTypedefs.h>


#include <map>
#include <mutex>
#include <tuple>

#include "emu64.cuh"
#include "internal.h"
#include "node.cuh"
#include "pdl.cuh"
#include "tma.cuh"
#include "waves.h"
#include "zmarch.h"
#include "zmarch_tile.cuh"
#include "zrag_tile.cuh"

namespace psd {

__device__ unsigned g_zmarch_error;  // set when an mbarrier wait times out

template <int MODE, int BY, int NST, bool kBnd>
__global__ void __launch_bounds__(32 * BY, 1)
k_zmarch(const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmC,
         const __grid_constant__ CUtensorMap tmE, void *__restrict__ T2v, void *__restrict__ E2v,
         const ZParams p) {
    grid_dep_wait();  // the previous step's writes (and its reads of T2) are complete
    grid_dep_launch();
    const int X0 = (int)(blockIdx.x % p.ntx) * (32 * ZTraits<MODE>::PX);
    const int Y0 = (int)(blockIdx.x / p.ntx) * BY;
    const int k0 = 1 + (int)blockIdx.y * p.kchunk;
    const int k1 = (int)min((int64_t)k0 + p.kchunk, p.nz - 1);  // output planes [k0, k1)
    zmarch_tile<MODE, BY, NST, 32, kBnd>(&tmT, &tmC, T2v, E2v, p, X0, Y0, k0, k1, &g_zmarch_error, &tmE);
}

// The same on ragged rows (zrag_tile.cuh).
template <int MODE, int PX, int BY, int NST, int MINB, bool kBnd>
__global__ void __launch_bounds__(32 * BY, MINB)
k_zmarch_rag(const __grid_constant__ CUtensorMap tmT, const __grid_constant__ CUtensorMap tmC,
             void *__restrict__ T2v, const ZParams p) {
    grid_dep_wait();
    grid_dep_launch();
    const int X0 = 1 + (int)(blockIdx.x % p.ntx) * (32 * PX);
    const int Y0 = 1 + (int)(blockIdx.x / p.ntx) * BY;
    const int k0 = 1 + (int)blockIdx.y * p.kchunk;
    const int k1 = (int)min((int64_t)k0 + p.kchunk, p.nz - 1);
    zrag_tile<MODE, PX, BY, NST, kBnd>(&tmT, &tmC, T2v, p, X0, Y0, k0, k1, &g_zmarch_error);
}

// Failure-path self-test: one CTA waits on an mbarrier that nothing ever arrives on.
// The bounded wait gives up after `polls` polls of at most `ns` nanoseconds each and
// reports through the same device flag as a pipelined kernel's time-out.
__global__ void k_selftest_wait(unsigned polls, unsigned ns) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    bool done = false;
    for (unsigned i = 0; i < polls && !done; ++i) done = mbar_try_wait_hint(&bar, 0u, ns);
    if (!done && threadIdx.x == 0) atomicOr(&g_zmarch_error, 1u);
}

cudaError_t launch_selftest_wait(unsigned polls, unsigned ns, cudaStream_t s) {
    k_selftest_wait<<<1, 32, 0, s>>>(polls, ns);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ host
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                             &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (PFN_cuTensorMapEncodeTiled_v12000)ptr;
    });
    return fn;
}

bool make_tensor_map_3d(CUtensorMap *m, const void *ptr, int esz, Grid3 g, unsigned bx, unsigned by) {
    return make_tensor_map_3d_pitch(m, ptr, esz, g, g.nx, bx, by);
}

bool make_tensor_map_3d_pitch(CUtensorMap *m, const void *ptr, int esz, Grid3 g, int64_t pitch,
                              unsigned bx, unsigned by) {
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz};
    const cuuint64_t strides[2] = {(cuuint64_t)(pitch * esz), (cuuint64_t)(pitch * g.ny * esz)};
    const cuuint32_t box[3] = {bx, by, 1};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = fn(m, esz == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                          3, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_tensor_map_rows(CUtensorMap *m, const void *ptr, int esz, int64_t n, int64_t rowlen, unsigned bx,
                          unsigned by) {
    auto fn = encode_fn();
    if (!fn) return false;
    const bool line = by == 0;  // one line of n elements
    const cuuint64_t dims[2] = {(cuuint64_t)(line ? n : rowlen), (cuuint64_t)(line ? 1 : n / (rowlen > 0 ? rowlen : 1))};
    const cuuint64_t strides[1] = {line ? 0 : (cuuint64_t)(rowlen * esz)};
    const cuuint32_t box[2] = {bx, line ? 1u : by}, estr[2] = {1, 1};
    const CUresult r = fn(m, esz == 8 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT64 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                          line ? 1 : 2, const_cast<void *>(ptr), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

bool make_tensor_map_quarter(CUtensorMap *m, const float *ptr, Grid3 g, int64_t r, unsigned bx, unsigned by) {
    auto fn = encode_fn();
    if (!fn) return false;
    const int64_t shift = (r * g.nx + (int64_t)((uintptr_t)ptr >> 2)) & 3;
    const cuuint64_t dims[2] = {(cuuint64_t)(g.nx + shift), (cuuint64_t)((g.ny * g.nz - r + 3) / 4)};
    const cuuint64_t strides[1] = {(cuuint64_t)(16 * g.nx)};
    const cuuint32_t box[2] = {bx, by}, estr[2] = {1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(ptr + (r * g.nx - shift)), dims, strides, box,
              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool ragged_supported(Grid3 g, const void *a, const void *b, const void *c) {
    if (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c) & 15u) return false;
    // element coordinates of planes -1 .. nz, tiles past the grid included, fit 32 bits
    // (FP32; FP64's row-pair coordinates then do)
    if (g.nx > (1LL << 30) || g.ny > (1LL << 30)) return false;
    const double plane = (double)g.nx * ((double)g.ny + 64.0);
    if (plane * ((double)g.nz + 2.0) + 4096.0 >= 2147483647.0) return false;
    return encode_fn() != nullptr;
}

bool zmarch_supported(Grid3 g, int esz, const void *a, const void *b, const void *c) {
    if ((g.nx * esz) % 16 != 0) return false;
    if (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c) & 15u) return false;
    if (g.nx > (1LL << 31) - 256 || g.ny > (1LL << 31) - 64 || g.nz > (1LL << 31) - 2) return false;
    return encode_fn() != nullptr;
}

// Share of n items' tiles of t that is used.
static double fill(int64_t n, int64_t t) { return (double)n / (double)((n + t - 1) / t * t); }

bool step_small(Grid3 g, int mode, bool in_loop) {
    // a set z-chunk or nodes-per-thread override asks for the march
    if (launch_override(PS_OVERRIDE_KCHUNK) > 0 || launch_override(PS_OVERRIDE_F64_PX2) == 1) return false;
    const bool fp32 = mode == Z_F32 || mode == Z_F32_COMP;
    const bool aligned = (g.nx * (fp32 ? 4 : 8)) % 16 == 0;
    // on aligned rows a single step keeps the march, and so does Ci as given on equal spacings, whose one-binade
    // form multiplies Ci by K first, which rounds another way than the column kernel's K*S
    if (aligned && (!in_loop || mode == Z_F64_EMU_ISO)) return false;
    const double n = (double)g.nx * (double)g.ny * (double)g.nz;
    // The line lies where the march catches up (us a step, column / march).
    // rows that fill the march's 128-node tiles by 77% or more favour it
    const bool full = fill(g.nx, 128) >= 0.77;
    switch (mode) {
        case Z_F32:  // full rows 5e5 nodes 3.0 / 2.9, 1e6 4.1 / 3.7; 192^3 13.1 / 14.3, 200^3 16 / 16;
                     // ragged 205^3 20.8 / 21.7, 211^3 25.5 / 23.8
            return n <= (aligned ? (full ? 6e5 : 7.5e6) : 8.8e6);
        case Z_F32_COMP:  // 160^3 14 / 19, 176^3 25 / 25; full rows 128^3 9.4 / 10.9, 368 x 112 x 72
                          // 12.0 / 10.8
            if (!aligned) {
                // odd rows (zcomp_rag.cu), by the useful lanes of its 128 x 16 tiles against the column
                // kernel's 32 x 8: 113 x 18 x 588 (0.9) 7.2 / 6.2, 2717 x 48 x 20 (1) 11.2 / 10.7, 225 x 205 x 80
                // (0.87) 13.3 / 14.7, 437 x 734 x 16 (0.87) 22 / 18.5, 1079 x 8 x 408 (0.5) 12 / 19
                return n <= (comp_ragged_share(g) >= 0.9 ? 2e6 : 5.2e6);
            }
            return n <= (full ? 2.2e6 : 4.3e6);
        case Z_F64_EMU_ANISO:  // 192^3 37 / 41, 200^3 53 / 49; ragged 219^3 61 / 64, 227^3 71 / 69, 93 x 512 x
                               // 257 (0.75 of the column kernel's useful lanes) 80 / 117
            return n <= (aligned ? 7.5e6 : (fill(g.nx - 2, 64) >= 0.8 * fill(g.nx - 2, 32) ? 1.05e7 : 1.3e7));
        case Z_F64_EMU_ISO:  // odd rows (aligned ones above): 369 x 160 x 112 (1) 38 / 41, 303 x 250 x 160 (1) 74 / 71,
                             // 213 x 407 x 192 (0.88) 95 / 107, 797 x 20 x 1559 (0.96) 168 / 141
            return n <= (fill(g.nx - 2, 64) >= 0.94 * fill(g.nx - 2, 32) ? 7.5e6 : 2e7);
        default: {
            // by the share of useful lanes in the march's 64-node tiles (four nodes per thread:
            // where as good): 128 x 321 x 75 (1) 23 / 21, 128^3 (1) 10 / 15; 160^3 (0.83) 21 / 24,
            // 176^3 (0.92) 32 / 29; 200^3 (0.78) 50 / 45
            if (aligned) {
                const double lanes = fill(g.nx, 64);
                return n <= (lanes >= 0.87 ? 2.2e6 : (lanes >= 0.8 ? 4.3e6 : 7.5e6));
            }
            // odd rows, whose march is slower, by that share against the column kernel's (32 nodes wide):
            // 191 x 8 x 1793 (1) 12 / 15, 919 x 15 x 261 (0.97) 17 / 22, 125 x 128 x 352 (1) 33 / 32; 225 x 205 x 80
            // (0.87) 17 / 23, 199 x 104 x 353 (0.82) 45 / 45; 75 x 148 x 320 (0.76) 21 / 31, 93 x 512 x 257 (0.75) 69 / 77
            const double share = fill(g.nx - 2, 64) / fill(g.nx - 2, 32);
            return n <= (share >= 0.9 ? 4.5e6 : (share >= 0.8 ? 7.5e6 : 1.3e7));
        }
    }
}

bool step_ragged_ok(Grid3 g, int esz, const void *a, const void *b, const void *c) {
    if (launch_override(PS_OVERRIDE_STEP_PLAIN) == 1 || (g.nx * esz) % 16 == 0) return false;
    // FP32 grids that leave more than 40% of its 128 x 8 tiles idle: the column kernel is as
    // fast (151 x 367 x 271, 0.58 in use: 44.5 us a step here, 43.6 there; 391 x 8 x 3059, 0.57: 24 and 18)
    if (esz == 4 && fill(g.nx - 2, 128) * fill(g.ny - 2, 8) < 0.6 && launch_override(PS_OVERRIDE_KCHUNK) <= 0)
        return false;
    return ragged_supported(g, a, b, c);
}

double comp_ragged_share(Grid3 g) {
    return fill(g.nx - 2, 128) * fill(g.ny - 2, 16) / (fill(g.nx - 2, 32) * fill(g.ny - 2, 8));
}

bool comp_ragged_ok(Grid3 g, const void *a, const void *b, const void *c) {
    if (launch_override(PS_OVERRIDE_STEP_PLAIN) == 1 || g.nx % 4 == 0) return false;
    // less than 0.45 of the column kernel's useful lanes: that kernel (us a step, column / here: 391 x 8 x 3059
    // (0.4) 41 / 55, 1061 x 6 x 4776 (0.47) 228 / 184, 67 x 400 x 400 (0.75) 86 / 55)
    if (comp_ragged_share(g) < 0.45 && launch_override(PS_OVERRIDE_KCHUNK) <= 0) return false;
    return ragged_supported(g, a, b, c);
}

bool step_tma_ok(Grid3 g, int esz, const void *a, const void *b, const void *c) {
    return launch_override(PS_OVERRIDE_STEP_PLAIN) != 1 && zmarch_supported(g, esz, a, b, c);
}

// Planes per CTA of the one-step march.
// per_sm: CTAs that an SM holds; waves: their cost, or null.
static int step_kchunk(int esz, Grid3 g, int64_t tiles, int per_sm, const WaveCost *waves, bool comp = false) {
    // Short chunks keep many CTAs in flight (no wave tail) while consecutive
    // CTAs - neighbouring tiles of one chunk - share their halo planes in L2;
    // each chunk pays two extra planes.  Measured (sweeps at 256^3 and 512^3):
    // FP32 is fastest at 8 planes; FP64 at 8 planes on small grids, at 13-18 at 320^3 and at 24
    // at 448^3 to 640^3 (1% ahead of 32), so about 32 CTAs per SM between 8 and 24 planes (with
    // 64: 320^3 134 us a step / 130, 321^3 150 / 144, 384^3 216 / 212).
    // FP32 grids up to 3 million nodes (a few CTAs per SM): 3 planes (128^3 5.1 against 5.6 us, 192 x 67 x 184
    // 8.6 and 11.4).  The two-float state up to 2.5 million in whole tiles (384 x 96 x 64 10.4 against 11.5, but
    // 400 x 140 x 52 13.7 against 11.5 and 52 x 197 x 141 13.2 against 10.5).
    if (esz == 4 && (comp ? (double)tiles * 1024.0 * (double)g.nz <= 2.5e6 : (double)g.n() <= 3e6)) return 3;
    const int64_t target = 32LL * sm_count();
    const int64_t kmax = esz == 8 ? 24 : 8;
    const int64_t kc = (g.nz - 2) * tiles / target;
    // FP64 grids of a few waves: the chunk whose waves end soonest, fitted to sweeps of 13 to 18
    // shapes each (us a step against 8 planes: 128 x 150 x 200 20.8 / 23.9, 400 x 100 x 60 15.2 /
    // 16.8, 128^3 12.9 / 16.2, 256 x 40 x 400 22.4 / 24.2)
    if (waves && kc <= 8) return wave_chunk(g.nz - 2, tiles, sm_count(), per_sm, *waves);
    return (int)(kc < 8 ? 8 : (kc > kmax ? kmax : kc));
}

template <int MODE, int BY, int NST, bool kBnd = false>
static cudaError_t launch_zmarch_t(void *T2, const void *T, void *E2, const void *Ein, const void *Ci,
                                   Grid3 g, ZParams p, int kchunk, cudaStream_t s) {
    using E = typename ZTraits<MODE>::E;
    constexpr int PX = ZTraits<MODE>::PX, BX = 32 * PX, W = BX + 2 * PX, H = BY + 2;
    constexpr unsigned TBA = (W * H * sizeof(E) + 127) / 128 * 128;
    constexpr unsigned CBA = (BX * BY * sizeof(E) + 127) / 128 * 128;
    constexpr unsigned EBA = MODE == Z_F32_COMP ? TBA : 0u;
    constexpr size_t smem = NST * (TBA + CBA + EBA) + NST * 8;
    static unsigned attr_gen[64] = {0};
    cudaError_t ae;
    if (!set_smem_attr_once((const void *)k_zmarch<MODE, BY, NST, kBnd>, (int)smem, attr_gen, &ae)) return ae;
    CUtensorMap mT, mC, mE;
    if (!make_tensor_map_3d(&mT, T, sizeof(E), g, W, H) ||
        !make_tensor_map_3d(&mC, Ci, sizeof(E), g, BX, BY))
        return cudaErrorInvalidValue;
    if (MODE == Z_F32_COMP) {
        if (!make_tensor_map_3d(&mE, Ein, sizeof(E), g, W, H)) return cudaErrorInvalidValue;
    } else {
        mE = mT;  // not read
    }
    const int64_t ntx = (g.nx + BX - 1) / BX, nty = (g.ny + BY - 1) / BY;
    const int64_t tiles = ntx * nty;
    if (kchunk <= 0) {
        constexpr WaveCost wide{2.0, 0.6, 0.2, 3, 12}, narrow{1.0, 0.4, 0.2, 3, 8};
        constexpr bool kWide = MODE == Z_F64_SCALED4;
        // (from two waves of 8 planes on, 8 stay as fast or faster: 128 x 144 x 496 45 us a step, 46 at
        // 12; 208 x 361 x 79, a field of both signs, 61 and 62.5)
        const bool few = tiles * ((g.nz + 5) / 8) < 2 * 5LL * sm_count();
        kchunk = step_kchunk(sizeof(E), g, tiles, kWide ? 5 : 4,
                             kWide ? (few ? &wide : nullptr)
                             : MODE == Z_F64_SCALED || MODE == Z_F64_EMU_ISO_DMUL ? &narrow : nullptr,
                             MODE == Z_F32_COMP);
    }
    kchunk = grid_chunk(g.nz, kchunk);
    const int64_t gz = (g.nz - 2 + kchunk - 1) / kchunk;
    if (tiles > 0x7fffffffLL || gz > 65535) return cudaErrorInvalidConfiguration;
    p.nx = g.nx;
    p.ny = g.ny;
    p.nz = g.nz;
    p.pitch = g.nx;
    p.ntx = (int)ntx;
    p.kchunk = kchunk;
    return launch_pdl(k_zmarch<MODE, BY, NST, kBnd>, dim3((unsigned)tiles, (unsigned)gz, 1), dim3(32 * BY), smem,
                      s, mT, mC, mE, T2, E2, p);
}

static ZParams make_params(StepCoef c) {
    ZParams p{};
    p.ek = emu_coef(c.dtlam, c.ax, c.ay, c.az);
    p.fdtlam = (float)c.dtlam;
    p.fax = (float)c.ax;
    p.fay = (float)c.ay;
    p.faz = (float)c.az;
    return p;
}

bool tma_encoder_available() { return encode_fn() != nullptr; }

bool f64_scaled_wide(Grid3 g, const void *T2, const void *T, const void *Ci) {
    if (launch_override(PS_OVERRIDE_F64_PX2) == 1) return false;
    // 128 x 4 tiles, unless 64 x 8 ones leave fewer lanes past the grid's edges (us a step, four
    // / two per thread: 192^3 41 / 34, 320^3 150 / 132, 448^3 357 / 330, 3000 x 3 x 300 14 / 18; equal
    // widths 256^3 71 / 71, 384^3 212 / 216).  Below a million nodes the launch counts, not the lanes.
    if (fill(g.nx, 64) * fill(g.ny, 8) > fill(g.nx, 128) * fill(g.ny, 4) && (double)g.n() >= 1e6) return false;
    return g.nx % 4 == 0 && ((((uintptr_t)T2 | (uintptr_t)T | (uintptr_t)Ci) & 31u) == 0);
}

ZParams zparams_for(StepCoef c, Grid3 g, int64_t pitch) {
    ZParams p = make_params(c);
    p.nx = g.nx;
    p.ny = g.ny;
    p.nz = g.nz;
    p.pitch = pitch;
    return p;
}

// One mode's launch, with the boundary-writing instantiation where asked (the forms
// that state-keeping time loops use; never the two-float step).
template <int MODE, int BY, int NST>
static cudaError_t launch_zmarch_b(void *T2, const void *T, void *E2, const void *Ein, const void *Ci, Grid3 g,
                                   ZParams p, int kchunk, cudaStream_t s, bool write_bnd) {
    if (MODE != Z_F32_COMP && write_bnd)
        return launch_zmarch_t<MODE, BY, NST, MODE != Z_F32_COMP>(T2, T, E2, Ein, Ci, g, p, kchunk, s);
    return launch_zmarch_t<MODE, BY, NST, false>(T2, T, E2, Ein, Ci, g, p, kchunk, s);
}

template <int MODE, int PX, int BY, int MINB, bool kBnd>
static cudaError_t launch_rag_t(void *T2, const void *T, const void *Ci, Grid3 g, ZParams p, cudaStream_t s) {
    constexpr int NST = 4;
    using R = ZRag<MODE, PX, BY>;
    using E = typename R::E;
    constexpr size_t smem = NST * R::SB + NST * 8;
    static unsigned attr_gen[64] = {0};
    cudaError_t ae;
    if (!set_smem_attr_once((const void *)k_zmarch_rag<MODE, PX, BY, NST, MINB, kBnd>, (int)smem, attr_gen, &ae))
        return ae;
    CUtensorMap mT, mC;
    if (!make_tensor_map_rows(&mT, T, sizeof(E), g.n(), 2 * g.nx, R::W, R::kPairs ? R::H / 2 : 0) ||
        !make_tensor_map_rows(&mC, Ci, sizeof(E), g.n(), 2 * g.nx, R::W, R::kPairs ? BY / 2 : 0))
        return cudaErrorInvalidValue;
    const int64_t ntx = (g.nx - 2 + R::BX - 1) / R::BX, nty = (g.ny - 2 + BY - 1) / BY, tiles = ntx * nty;
    int kchunk = launch_override(PS_OVERRIDE_KCHUNK);
    if (kchunk <= 0) {
        constexpr WaveCost ragged{0.5, 0.4, 0.1, 3, 12};
        kchunk = step_kchunk(sizeof(E), g, tiles, 3,
                             MODE == Z_F64_SCALED || MODE == Z_F64_EMU_ISO ? &ragged : nullptr);
    }
    kchunk = grid_chunk(g.nz, kchunk);
    const int64_t gz = (g.nz - 2 + kchunk - 1) / kchunk;
    if (tiles > 0x7fffffffLL || gz > 65535) return cudaErrorInvalidConfiguration;
    p.nx = g.nx;
    p.ny = g.ny;
    p.nz = g.nz;
    p.pitch = g.nx;
    p.ntx = (int)ntx;
    p.kchunk = kchunk;
    return launch_pdl(k_zmarch_rag<MODE, PX, BY, NST, MINB, kBnd>, dim3((unsigned)tiles, (unsigned)gz, 1),
                      dim3(32 * BY), smem, s, mT, mC, T2, p);
}

template <int MODE, int PX, int BY, int MINB>
static cudaError_t launch_rag_b(void *T2, const void *T, const void *Ci, Grid3 g, ZParams p, cudaStream_t s,
                                bool write_bnd) {
    if (write_bnd) return launch_rag_t<MODE, PX, BY, MINB, true>(T2, T, Ci, g, p, s);
    return launch_rag_t<MODE, PX, BY, MINB, false>(T2, T, Ci, g, p, s);
}

cudaError_t launch_zmarch_ragged(int mode, void *T2, const void *T, const void *Ci, StepCoef c, Grid3 g,
                                 cudaStream_t s, bool write_bnd) {
    const ZParams p = make_params(c);
    switch (mode) {
        // K*S, bit for bit the column kernel's, which takes smaller grids (257^3 91 us a step, 85 with Ci*K
        // multiplied first, whose last bit depends on which nodes share a warp; column kernel 99)
        case Z_F64_EMU_ISO:
            return launch_rag_b<Z_F64_EMU_ISO, 2, 8, 3>(T2, T, Ci, g, p, s, write_bnd);
        case Z_F64_EMU_ANISO:
            if (p.ek.axes == AX_SPREAD)
                return launch_rag_b<Z_F64_EMU_ANISO_SPREAD, 2, 8, 3>(T2, T, Ci, g, p, s, write_bnd);
            return launch_rag_b<Z_F64_EMU_ANISO, 2, 8, 3>(T2, T, Ci, g, p, s, write_bnd);
        case Z_F64_SCALED:
            return launch_rag_b<Z_F64_SCALED, 2, 8, 3>(T2, T, Ci, g, p, s, write_bnd);
        case Z_F32:
            return launch_rag_b<Z_F32, 4, 8, 4>(T2, T, Ci, g, p, s, write_bnd);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_zmarch(int mode, void *T2, const void *T, void *E2, const void *Ein, const void *Ci,
                          StepCoef c, Grid3 g, cudaStream_t s, bool write_bnd) {
    const ZParams p = make_params(c);
    const int kchunk = launch_override(PS_OVERRIDE_KCHUNK);
    const bool positive = c.dtlam * c.ax > 0 && c.dtlam * c.ay > 0 && c.dtlam * c.az > 0;
    const bool wb = write_bnd;
    switch (mode) {
        case Z_F64_EMU_ISO:
        case Z_F64_EMU_ANISO:
            if (!positive) return launch_zmarch_b<Z_F64_NATIVE, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
            // isotropic grids: fma(Ci*K, S, T), two FP64 ops and the fewest integer ops
            // (measured faster than one DFMA after a 64 x 64-bit high multiply by K)
            if (mode == Z_F64_EMU_ISO)
                return launch_zmarch_b<Z_F64_EMU_ISO_DMUL, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
            // spacings 2 to 16 apart: the sums at the lowest exponent instead of the K at the highest (256^3 115 us a
            // step against 101, but every axis keeps its bits)
            if (p.ek.axes == AX_SPREAD)
                return launch_zmarch_b<Z_F64_EMU_ANISO_SPREAD, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
            // more than 16 apart: the shifted sums would not fit 64 bits, so each axis has its own
            // rounded product (443 us)
            if (p.ek.axes == AX_FAR)
                return launch_zmarch_b<Z_F64_EMU_ANISO_FAR, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
            // four nodes per thread on large grids (us a step, two / four: 512 x 384 x 256 280 / 273, 512^3
            // 731 / 711, 256^3 103 / 103, 240 x 200 x 300 100 / 103)
            if ((double)g.n() >= 3e7 && f64_scaled_wide(g, T2, T, Ci))
                return launch_zmarch_b<Z_F64_EMU_ANISO4, 4, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
            return launch_zmarch_b<Z_F64_EMU_ANISO, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
        case Z_F64_NATIVE:
            return launch_zmarch_b<Z_F64_NATIVE, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
        case Z_F64_SCALED:
            // four nodes per thread (4-row tiles, 128 threads) where rows allow 32-byte
            // accesses and fill its tiles (f64_scaled_wide): measured 2-3% faster at 512^3 and 768^3 than two per thread
            // (8-row tiles of four per thread, at two CTAs per SM, were 15% slower)
            if (f64_scaled_wide(g, T2, T, Ci))
                return launch_zmarch_b<Z_F64_SCALED4, 4, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
            return launch_zmarch_b<Z_F64_SCALED, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
        case Z_F32:
            return launch_zmarch_b<Z_F32, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s, wb);
        case Z_F32_COMP:
            return launch_zmarch_t<Z_F32_COMP, 8, 4>(T2, T, E2, Ein, Ci, g, p, kchunk, s);
    }
    return cudaErrorInvalidValue;
}

unsigned zmarch_device_error(bool clear) {
    unsigned v = 0;
    cudaMemcpyFromSymbol(&v, g_zmarch_error, sizeof(v));
    if (clear) {
        const unsigned z = 0;
        cudaMemcpyToSymbol(g_zmarch_error, &z, sizeof(z));
    }
    return v;
}

}  // namespace psd
