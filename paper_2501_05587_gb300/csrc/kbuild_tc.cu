// Tensor-core (tcgen05) build of the kernel matrix K = kappa(P P^T).
//
// Sec. 3.2 forms B = P P^T with GEMM or SYRK and then applies the kernel
// function elementwise (Gaussian through Eq. 12 from B and the row norms).
// Here one persistent kernel walks the tiles (i, q) of the upper triangle,
// where a tile is a 128-row block i against a pair of 128-column blocks
// (2q, 2q + 1), 2q + 1 >= i:
//
//   warp 0  (one lane)  TMA loads, per k-block, of the 128 rows of the row block
//                       and the 256 rows of the column pair (swizzled) into a ring
//                       of stages;
//   warp 1  (one lane)  tcgen05.mma kind::f16 (M = 128, N = 256, FP32 accumulator
//                       in TMEM), double-buffered (512 columns);
//   warps 2-9           epilogue, one warpgroup a column block: tcgen05.ld the
//                       accumulator, apply kappa with FP32 row norms, stage a chunk
//                       and its transpose in shared memory and TMA-store both into
//                       K -- or, for the block-packed upper triangle the symmetric
//                       pass reads, bulk-copy the swizzled chunk alone to its place
//                       in the packed tile (each value stored once).
//
// Why column pairs: an SM takes in about 36 bytes per clock from L2 whichever path
// it uses (TMA, bulk copy, cp.async or vector loads), and a 128 x 128 tile moves
// 32 KB per k-block for 4 MMAs -- three times what that allows at the MMA rate.
// Sharing each row block between two column blocks cuts the bytes per MMA by a
// quarter, and one N = 256 MMA reads 12 KB of shared memory where two of N = 128
// read 16 (at 128 bytes a clock those alone take 64 of an N = 128 MMA's 68 clocks,
// before the operand ring's own writes): the images FP32 build 13.3 -> 11.8 ms.
// Block (2q + 1, 2q), below the diagonal, is computed and not stored.
//
// Precision modes (operand matrix W, one row per point; where there are two parts, 32 columns of hi and
// the same 32 of lo follow one another, so that a stage's rows are 128 bytes in every mode.  With the
// parts in two halves of W, read as 64-byte pieces by twice as many loads, BF16X3 took 23.8 ms at
// n = 10,000, d = 100,000 where it takes 20.0, and 650 at n = 50,000 where 554; FP32 n = 20,001, d = 1,000
// 1.37 and 1.33):
//   BF16    W = bf16(P);  norms of the rounded rows, so the Gaussian distance
//           r_i + r_j - 2 B_ij is the distance of the rounded points.
//   BF16X3  W = [hi | lo] with hi = bf16(p), lo = bf16(p - hi); each stage
//           holds the hi and lo parts of both operands once and the MMAs form
//           hi.hi + hi.lo + lo.hi (~16 significant bits of the cross term that
//           the Gaussian's cancellation needs) -- 2 d loaded instead of the 3 d
//           a [hi|hi|lo] x [hi|lo|hi] GEMM would stream.
//   FP32    (SPLIT) W = [hi | lo] in FP16 of the points times a power of two s:
//           hi = fp16(s p), lo = fp16(s p - hi), which represent p to 2^-23 of itself
//           (hi and lo carry 11 bits each and lo's sign one more: 1 + 2^-12 + 2^-23 is 2^-23 off), or
//           to 2^-27 of its row's and column's largest value (see split_decide).
//           The products are exact in FP32, but the tensor core adds them with
//           truncation: left in TMEM over a long row the sum drifts low by half an ulp an
//           MMA (measured at d = 784 on uniform points: relative error 6.1e-6 against
//           4.2e-7 for FP32 FMAs).  So a TMEM accumulator holds only 32 columns of the
//           rows: the small products lo.lo, hi.lo, lo.hi first, then the two hi.hi MMAs, and
//           the epilogue warps add each such chunk into FP32 registers, round to nearest, the
//           last two away from zero.  Why two, for any d: a chunk is truncated where its two
//           hi.hi MMAs add, at half its size and at its size, 3/4 ulp on average, and the ulps
//           of C chunks of a sum are together about one ulp of the sum, whatever C is; an
//           addition rounded away adds half an ulp of its partial sum on average where it
//           rounds at all, and the last two partial sums are about the sum.  (An exact sum stays exact,
//           which a factor above 1 on the chunks would not leave so.  Two chunks, d <= 64, have one
//           addition that rounds, and only every other time.)  Mean signed error, in 2^-24 |x| |y|,
//           linear, n = 2,000 (C = 2, 2, 3, 4, 8, 16, 25, 47):
//             d                              48     64     96    128    256    512    784   1500
//             uniform (0, 1), nearest     -0.86  -1.02  -1.01  -1.01  -1.01  -1.01  -1.00  -1.01
//                             so          -0.53  -0.69  -0.47  -0.35  -0.21  -0.14  -0.05  -0.01
//             |x|^2 of normal, nearest    -1.24  -1.44  -1.46  -1.46  -1.46  -1.46  -1.41  -1.48
//                             so          -0.77  -1.01  -0.72  -0.57  -0.40  -0.21  -0.18  -0.15
//             normal (mixed sign), nearest -0.10 -0.09  -0.08  -0.07  -0.05  -0.03  -0.03  -0.02
//                             so          -0.04  -0.05  -0.01  -0.01   0.00   0.01   0.01   0.01
//           J = trace K - ... of tight clusters sees it as a bias: uniform points -6e-8 to -9e-8
//           with nearest, 6e-8 at most so.  The root mean square is below the FMAs' throughout
//           (uniform: 0.6 to 1.3 here, 1.3 to 7.4 there).
//           lo.lo is below an ulp, but on the diagonal it is a sum of squares: left out, J =
//           trace K - ... of tight clusters is off by ten times that.
//           Images, n = 70,000, d = 784: 10.5 ms (64.7 on CUDA cores); the operand loads allow
//           8.4 (36 bytes a clock an SM), the MMAs 6.7, and the epilogue's stores (about 2 ms)
//           are not overlapped: the next tile's MMAs run two chunks ahead.  n = 20,001,
//           d = 1,000: 6.87 -> 1.33 ms a call.
//           Measured on those points: 7.8e-8 (and 5.0e-8 at d = 128, where FMAs give 1.6e-7).
//
// Every mbarrier wait is bounded (about 2 s by %globaltimer).  A wait that
// runs out sets *err, raises a shared abort flag that ends every role's loop,
// waits (bounded again) for the CTA's own TMA copies and MMAs in flight,
// frees TMEM and returns; the host reports POPCORN_ERR_TIMEOUT.
#include <cstdlib>
#include <cstring>

#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "popcorn_internal.cuh"
#include "tc_common.cuh"

namespace popcorn {
namespace {

using namespace tc;

constexpr uint32_t kIdescBf16 = idesc_bf16(128, 256);
constexpr uint32_t kIdescF16 = idesc_f16(128, 256);

constexpr int kModeBf16 = 0, kModeX3 = 1, kModeSplit = 2;
constexpr int BM = 128;                      // block rows / columns
// depth of a k-block, in 16-bit elements: a stage is 48 KB in every mode (SPLIT: also what a TMEM
// accumulator holds before it is drained)
constexpr int kbuild_dk(int mode) { return mode == kModeBf16 ? 64 : 32; }
constexpr int kRowElems = 64;                // a stage's row: 64 columns, or 32 of hi and the same 32 of lo: 128 bytes
constexpr int STG_BYTES = 16 * 1024;         // staging of one epilogue warpgroup: a 128 x 32 FP32 chunk, a
                                             // 128 x 64 half box, or a 128 x 16 chunk and its transpose
constexpr int NTHREADS = 320;                // 10 warps
constexpr int kStageBytes = 48 * 1024;       // a k-block of the row block and the column pair
constexpr int kStages = 3;                   // operand ring
constexpr int kStg = 2;                      // staging buffers per warpgroup
constexpr int NBARS = 2 * kStages + 5;
// shared memory: ring, staging of both warpgroups, their copies of the column norms, barriers
constexpr int kOffStg = kStages * kStageBytes, kOffRj = kOffStg + 2 * kStg * STG_BYTES, kOffBar = kOffRj + 2 * BM * 4,
              kOffMisc = kOffBar + NBARS * 8, kSmemBytes = kOffMisc + 16 + 1024;   // (slack: 1024-byte alignment)
constexpr uint32_t kTmemCols = 512;          // 2 buffers x 256 columns

struct TcArgs {
    int n, T, T2, nkb;        // rows, 128-blocks, column pairs, k-blocks per part
    long long tiles;
    float* K;                 // row-major square (SPLIT: the diagonal blocks are stored with plain stores)
    int64_t ldk;
    float* Kp;                // block-packed K (tile (I, J), I <= J, at its row-by-row triangle index
                              // times 16384 floats, four 128 x 32 boxes; FP16 / BF16: times 32 KB,
                              // two 128 x 64 boxes), or null
    int full;                 // 1: every tile of the square (the GEMM form), each stored once; 0: the
                              // tiles on and above the diagonal (the SYRK form), stored with their
                              // transposes unless K is packed
    KernParams kp;
    const float* norms;       // row norms of the represented rows (Gaussian)
    float* kdiag;
    const SplitState* split;  // SPLIT: the device's decision and scale
    int* err;
    // Error-path tests only (0 in every ordinary launch): CTA 0 leaves its first stage's copies out and
    // every wait of the launch gives up after wait_ns.
    int stall;
    unsigned long long wait_ns;
};

// tile t -> (row block i, column pair q).  The walk goes through bands of kBand row blocks, and in
// a band column pair by column pair, so that the tiles in flight at a time (152) touch kBand row blocks
// and about 19 column pairs (20 MB of W at d = 784): W is read from HBM once a band.  Row block by row
// block, it was read once a row block: 64 GB at n = 70,000, as much HBM time as the whole build takes
// now (11.8 -> 10.9 ms; BF16 4.96 -> 4.17).  (Bands of 2 gained 3% on rows of 400 KB and lost 10% at
// d = 30,000.)
// Band b of the upper triangle holds its row blocks and the pairs from its first diagonal block on;
// pair j of a band holds the first 2 j + 2 of its R row blocks (block (2q + 1, 2q) is the only one
// below the diagonal), so the pairs before F = R / 2 hold F (F + 1) tiles and a whole band
// kBand (kBand - 2) / 4 = 12 fewer than its rectangle.  (Walked with the rectangle's empty places, which
// the static round-robin gave to CTAs like tiles, BF16X3 took 2.30 ms at n = 10,000, d = 10,000 where it
// takes 2.11, and 49 at n = 50,000 where 45.6; FP32 68.3 and 63.4.)  A binary search over b, no
// floating point.  The full schedule takes every pair.
constexpr int kBand = 8;
__host__ __device__ inline long long band_start(long long b, int T2, int full) {
    if (full) return b * kBand * T2;
    return b * kBand * T2 - (long long)(kBand * kBand / 4) * b * (b - 1) - b * (kBand * (kBand - 2) / 4);
}
__device__ __forceinline__ void tile_coords(long long t, int T, int T2, int full, int* i, int* q) {
    int lo = 0, hi = (T - 1) / kBand;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (band_start(mid, T2, full) <= t) lo = mid;
        else hi = mid - 1;
    }
    const int R = min(kBand, T - kBand * lo), F = full ? 0 : R / 2;
    int r = (int)(t - band_start(lo, T2, full));
    int j;
    if (r < F * (F + 1)) {
        j = (r >= 2) + (r >= 6) + (r >= 12);   // (F <= 4)
        r -= j * (j + 1);
    } else {
        r -= F * (F + 1);
        j = F + r / R;
        r %= R;
    }
    *i = kBand * lo + r;
    *q = (full ? 0 : kBand / 2 * lo) + j;
}
long long tile_count(int T, int T2, int full) {
    const int b = (T - 1) / kBand, R = T - kBand * b, F = full ? 0 : R / 2;
    return band_start(b, T2, full) + F * (F + 1) + (long long)(T2 - (full ? 0 : kBand / 2 * b) - F) * R;
}

// The kernel kind is a template parameter: with a runtime branch an element, the epilogue's
// 128 elements a thread ran one after the other (about 300 clocks each, no overlap between
// their chains), and it, not the MMAs, bounded every Gaussian build (images: 18.2 ms for
// BF16 and BF16X3 alike; 4.9 and 7.9 ms with the kind a parameter and two epilogue
// warpgroups, 3.9 and 7.1 now).
template <int KIND>
__device__ __forceinline__ float kappa(float b, float ri, float rj, const KernParams& kp) {
    if constexpr (KIND == POPCORN_LINEAR) return b;
    if constexpr (KIND == POPCORN_POLYNOMIAL) {
        const float base = fmaf(kp.gamma, b, kp.coef0);
        float r = base;
        for (int e = 1; e < kp.degree; ++e) r *= base;
        return r;
    }
    const float d2 = fmaxf(fmaf(-2.f, b, ri + rj), 0.f);
    return expf(kp.neg_gamma_over_sigma2 * d2);
}
// kappa over a 32-element chunk: the polynomial's degree loop outside the elements, for the
// same reason.
template <int KIND>
__device__ __forceinline__ void kappa32(float (&v)[32], float ri, const float* rj, const KernParams& kp) {
    if constexpr (KIND == POPCORN_POLYNOMIAL) {
        float base[32];
#pragma unroll
        for (int x = 0; x < 32; ++x) v[x] = base[x] = fmaf(kp.gamma, v[x], kp.coef0);
        for (int e = 1; e < kp.degree; ++e) {
#pragma unroll
            for (int x = 0; x < 32; ++x) v[x] *= base[x];
        }
    } else if constexpr (KIND == POPCORN_GAUSSIAN) {
#pragma unroll
        for (int x = 0; x < 32; x += 4) {
            const float4 r = *reinterpret_cast<const float4*>(rj + x);
            v[x] = kappa<KIND>(v[x], ri, r.x, kp);
            v[x + 1] = kappa<KIND>(v[x + 1], ri, r.y, kp);
            v[x + 2] = kappa<KIND>(v[x + 2], ri, r.z, kp);
            v[x + 3] = kappa<KIND>(v[x + 3], ri, r.w, kp);
        }
    }
}

// Output of the epilogue, one instance each, since a runtime choice between staging stores
// slowed the epilogue about 2.8x: kOutFull (full square through tensor maps), kOutSw16 /
// kOutSw4 (the packed triangle in that layout), kOutHalf16 / kOutHalfB16 (packed FP16 / BF16
// triangle, kPackedSw128H: each 64-column box is staged whole -- two 32-column chunks -- and
// stored with one bulk copy; entries past n are zeros).
constexpr int kOutFull = 0, kOutSw16 = 1, kOutSw4 = 2, kOutHalf16 = 3, kOutHalfB16 = 4;

__device__ __forceinline__ uint32_t pack_half2(float x, float y, bool bf16) {
    if (bf16) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
        return *reinterpret_cast<const uint32_t*>(&h);
    }
    const __half2 h = __floats2half2_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float round_half(float x, bool bf16) {
    return bf16 ? __bfloat162float(__float2bfloat16_rn(x)) : __half2float(__float2half_rn(x));
}

// What the epilogue of one 128 x 128 block knows.
struct BlockCtx {
    int rb, j;                 // row block, column block
    int row_local, row;        // this thread's row
    int et;                    // thread within the warpgroup
    int bar;                   // the warpgroup's named barrier
    unsigned char* stg;        // the warpgroup's staging
    bool diag;
};

// Elements [32 c, 32 c + 32) of this thread's row of a block, kappa applied: staged and stored.
// ctr counts the staging fills of the warpgroup.
template <int OUT>
__device__ __forceinline__ void store_chunk(const TcArgs& a, const BlockCtx& b, const CUtensorMap* map_kd,
                                            const CUtensorMap* map_kt, int c, float (&v)[32], int& ctr) {
    auto begin = [&]() -> unsigned char* {   // the store that last used this buffer has read it
        unsigned char* sb = b.stg + (ctr & 1) * STG_BYTES;
        ++ctr;
        if (b.et == 0) bulk_wait_read<kStg - 1>();
        named_bar<128>(b.bar);
        return sb;
    };
    const long long tri = (long long)b.rb * a.T - (long long)b.rb * (b.rb - 1) / 2 + (b.j - b.rb);
    if constexpr (OUT == kOutHalf16 || OUT == kOutHalfB16) {
        constexpr bool HB16 = OUT == kOutHalfB16;
        // box c / 2 of the half tile: staged over two chunks, stored after the second
        unsigned char* sb;
        if ((c & 1) == 0) sb = begin();
        else sb = b.stg + ((ctr - 1) & 1) * STG_BYTES;
        const int col0 = b.j * BM + 32 * c;
        const bool rv = b.row < a.n;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            // logical 16-byte chunk 4 (c mod 2) + i of the row, at its swizzled place
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int x = 8 * i + 2 * e;
                const float x0 = (rv && col0 + x < a.n) ? v[x] : 0.f;
                const float x1 = (rv && col0 + x + 1 < a.n) ? v[x + 1] : 0.f;
                w[e] = pack_half2(x0, x1, HB16);
            }
            const int pc = (4 * (c & 1) + i) ^ (b.row_local & 7);
            *reinterpret_cast<uint4*>(sb + b.row_local * 128 + 16 * pc) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        if (c & 1) {
            fence_proxy_async();
            named_bar<128>(b.bar);
            if (b.et == 0) {
                bulk_store_1d(reinterpret_cast<unsigned char*>(a.Kp) + tri * 32768 + (c >> 1) * 16384, smem_u32(sb),
                              (uint32_t)STG_BYTES);
                bulk_commit();
            }
        }
    } else if constexpr (OUT == kOutSw4 || OUT == kOutSw16) {
        // the staged chunk is box c of packed tile (rb, j), byte for byte
        float* sd = reinterpret_cast<float*>(begin());
        if constexpr (OUT == kOutSw4) {
            // element x of row row_local at x ^ (row_local mod 32) (the 32 lanes hold 32
            // consecutive rows: 32 different banks per store)
#pragma unroll
            for (int x = 0; x < 32; ++x) sd[b.row_local * 32 + (x ^ (b.row_local & 31))] = v[x];
        } else {
            // 16-byte piece i of the row at i ^ (row % 8)
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4*>(sd + b.row_local * 32 + ((i ^ (b.row_local & 7)) * 4)) =
                    make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
        fence_proxy_async();
        named_bar<128>(b.bar);
        if (b.et == 0) {
            bulk_store_1d(a.Kp + tri * (BM * BM) + c * (BM * 32), smem_u32(sd), (uint32_t)STG_BYTES);
            bulk_commit();
        }
    } else {
        const bool transpose = !b.diag && !a.full;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            // 16 columns: the direct chunk in the 64-byte swizzle (16-byte piece i of a row at
            // i ^ ((row / 2) mod 4)), then the transpose, 16 rows of 128
            float* sd = reinterpret_cast<float*>(begin());
            float* sx = sd + BM * 16;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<float4*>(sd + b.row_local * 16 + ((i ^ ((b.row_local >> 1) & 3)) * 4)) =
                    make_float4(v[16 * half + 4 * i], v[16 * half + 4 * i + 1], v[16 * half + 4 * i + 2],
                                v[16 * half + 4 * i + 3]);
            if (transpose) {
#pragma unroll
                for (int x = 0; x < 16; ++x) sx[x * BM + b.row_local] = v[16 * half + x];
            }
            fence_proxy_async();
            named_bar<128>(b.bar);
            if (b.et == 0) {
                const int col = b.j * BM + 32 * c + 16 * half;
                if (col < a.n) {
                    tma_store_2d(map_kd, col, b.rb * BM, smem_u32(sd));
                    if (transpose) tma_store_2d(map_kt, b.rb * BM, col, smem_u32(sx));
                }
                bulk_commit();
            }
        }
    }
}

// SPLIT, a diagonal block: hi.lo and lo.hi reach element (r, c) in the opposite order of
// (c, r), so the elements on and above the diagonal are stored to both places (`below`: those
// on and below it, in a tile whose MMAs ran in the order of the blocks below the diagonal).
template <int OUT>
__device__ __forceinline__ void store_diag_chunk(const TcArgs& a, const BlockCtx& b, bool below, int c,
                                                 const float (&v)[32]) {
    const int r = b.row_local;
    float* tile = nullptr;
    if constexpr (OUT != kOutFull)
        tile = a.Kp + ((long long)b.rb * a.T - (long long)b.rb * (b.rb - 1) / 2) * (BM * BM);
    auto put = [&](int i, int l, float x) {
        if constexpr (OUT == kOutFull) {
            const int gi = b.rb * BM + i, gl = b.rb * BM + l;
            if (gi < a.n && gl < a.n) a.K[(int64_t)gi * a.ldk + gl] = x;
        } else if constexpr (OUT == kOutSw4) {
            tile[(l >> 5) * (BM * 32) + i * 32 + ((l & 31) ^ (i & 31))] = x;
        } else {
            tile[(l >> 5) * (BM * 32) + i * 32 + ((((l & 31) >> 2) ^ (i & 7)) << 2) + (l & 3)] = x;
        }
    };
#pragma unroll
    for (int x = 0; x < 32; ++x) {
        const int l = 32 * c + x;
        if (l == r || (l > r) != below) {
            put(r, l, v[x]);
            if (l != r) put(l, r, v[x]);
        }
    }
}

// a + b rounded away from zero (an exact sum stays exact).
__device__ __forceinline__ float add_away(float a, float b) {
    const float up = __fadd_ru(a, b), dn = __fadd_rd(a, b);
    return fabsf(up) >= fabsf(dn) ? up : dn;
}

template <int MODE, int OUT, int KIND>
__global__ void __launch_bounds__(NTHREADS, 1)
    kbuild_tc_kernel(const __grid_constant__ CUtensorMap map_r, const __grid_constant__ CUtensorMap map_c,
                     const __grid_constant__ CUtensorMap map_kd, const __grid_constant__ CUtensorMap map_kt,
                     TcArgs a) {
    constexpr bool SPLIT = MODE == kModeSplit, X3 = MODE != kModeBf16;
    grid_dependency_wait();                       // the operands come from the kernel before
    if (SPLIT && !split_taken(a.split)) return;   // the CUDA-core build takes this matrix
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + kOffBar;
    constexpr int S = kStages;
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
    auto accf_bar = [&](int b) { return bar0 + 8u * (2 * kStages + b); };
    auto acce_bar = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };
    const uint32_t down_bar = bar0 + 8u * (2 * kStages + 4);
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffMisc + 4);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(accf_bar(b), 1);
            mbar_init(acce_bar(b), 8);
        }
        mbar_init(down_bar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {   // whole warp: all 512 TMEM columns
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32((const void*)tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    // stage layout: columns (256 rows of W) | rows (128 rows), rows of kRowElems; lo 64 bytes behind hi
    constexpr int DK = kbuild_dk(MODE);
    constexpr uint32_t kCols = 0, kRows = 2 * BM * kRowElems * 2, kLo = 64;
    const long long G = gridDim.x;
    if (warp == 0) {
        if (lane == 0) {
            // ---------------- TMA producer ----------------
            int stage = 0;
            uint32_t phase = 0;
            uint32_t issued_parity[kStages];
            bool issued[kStages];
            for (int s = 0; s < kStages; ++s) issued[s] = false;
            bool ok = true, first = true;
            for (long long t = blockIdx.x; t < a.tiles && ok; t += G) {
                int i, q;
                tile_coords(t, a.T, a.T2, a.full, &i, &q);
                for (int kb = 0; kb < a.nkb; ++kb) {
                    if (!mbar_wait_for(empty_bar(stage), phase ^ 1u, abort_flag, a.err, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    if (!(a.stall && blockIdx.x == 0 && first)) {
                        const uint32_t st = sbase + (uint32_t)(stage * kStageBytes);
                        mbar_arrive_expect_tx(full_bar(stage), (uint32_t)kStageBytes);
                        tma_load_2d(st + kCols, &map_c, kb * kRowElems, q * 2 * BM, full_bar(stage));
                        tma_load_2d(st + kRows, &map_r, kb * kRowElems, i * BM, full_bar(stage));
                        issued[stage] = true;
                        issued_parity[stage] = phase;
                    }
                    first = false;
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!ok) {
                // aborted: let this CTA's own copies land before shared memory goes away
                for (int s = 0; s < S; ++s)
                    if (issued[s]) {
                        const unsigned long long t0 = globaltimer();
                        while (!mbar_try_wait(full_bar(s), issued_parity[s]) && globaltimer() - t0 < kWaitLimitNs) {
                        }
                    }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---------------- MMA issuer ----------------
            int stage = 0;
            uint32_t phase = 0;
            int fill = 0;   // accumulator fills: a tile, or (SPLIT) a 32-deep chunk
            bool ok = true;
            const uint64_t desc0 = sw128_desc(sbase);
            // both halves of the next buffer have been read by the epilogue
            auto take_buffer = [&](int ab, uint32_t use) {
                if (!mbar_wait_for(acce_bar(ab), (use & 1u) ^ 1u, abort_flag, a.err, a.wait_ns)) return false;
                tc_fence_after();
                return true;
            };
            for (long long t = blockIdx.x; t < a.tiles && ok; t += G) {
                bool below = false;   // SPLIT: the tile holds a block below the diagonal
                int i, q;
                tile_coords(t, a.T, a.T2, a.full, &i, &q);
                if (SPLIT && a.full) below = 2 * q < i;
                if (!SPLIT && !take_buffer(fill & 1, (uint32_t)(fill >> 1))) break;
                for (int kb = 0; kb < a.nkb && ok; ++kb) {
                    if (!mbar_wait_for(full_bar(stage), phase, abort_flag, a.err, a.wait_ns)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t st = sbase + (uint32_t)(stage * kStageBytes);
                    // 16 elements = 32 bytes further along K inside the swizzled row.  Descriptors are
                    // advanced by adds: the 14-bit address field never carries.
                    if constexpr (SPLIT) {
                        const int ab = fill & 1;
                        if (!take_buffer(ab, (uint32_t)(fill >> 1))) {
                            ok = false;
                            break;
                        }
                        ++fill;
                        const uint64_t sd = desc0 + (uint64_t)(uint32_t)(stage * (kStageBytes >> 4));
                        const uint64_t rh = sd + (kRows >> 4), rl = rh + (kLo >> 4);
                        const uint64_t ch = sd + (kCols >> 4), cl = ch + (kLo >> 4);
                        const uint32_t d_tmem = tmem + (uint32_t)(ab * 2 * BM);
                        // the small products first; hi.lo and lo.hi in the order of the
                        // transposed block below the diagonal (full schedule): K stays symmetric
                        const uint64_t r1 = below ? rl : rh, c1 = below ? ch : cl;
                        const uint64_t r2 = below ? rh : rl, c2 = below ? cl : ch;
                        mma_bf16(d_tmem, rl, cl, kIdescF16, 0u);
                        mma_bf16(d_tmem, rl + 2, cl + 2, kIdescF16, 1u);
                        mma_bf16(d_tmem, r1, c1, kIdescF16, 1u);
                        mma_bf16(d_tmem, r2, c2, kIdescF16, 1u);
                        mma_bf16(d_tmem, r1 + 2, c1 + 2, kIdescF16, 1u);
                        mma_bf16(d_tmem, r2 + 2, c2 + 2, kIdescF16, 1u);
                        mma_bf16(d_tmem, rh, ch, kIdescF16, 1u);
                        mma_bf16(d_tmem, rh + 2, ch + 2, kIdescF16, 1u);
                        mma_commit(accf_bar(ab));
                    } else {
                        const uint64_t sd = desc0 + (uint64_t)(uint32_t)(stage * (kStageBytes >> 4));
                        const uint64_t rh = sd + (kRows >> 4), rl = rh + (kLo >> 4);
                        const uint64_t ch = sd + (kCols >> 4), cl = ch + (kLo >> 4);
                        const uint32_t d_tmem = tmem + (uint32_t)((fill & 1) * 2 * BM);
#pragma unroll
                        for (int kk = 0; kk < DK / 16; ++kk) {
                            mma_bf16(d_tmem, rh + 2 * kk, ch + 2 * kk, kIdescBf16, (kb | kk) ? 1u : 0u);
                            if constexpr (X3) {
                                mma_bf16(d_tmem, rh + 2 * kk, cl + 2 * kk, kIdescBf16, 1u);
                                mma_bf16(d_tmem, rl + 2 * kk, ch + 2 * kk, kIdescBf16, 1u);
                            }
                        }
                    }
                    mma_commit(empty_bar(stage));   // stage free once these MMAs have read it
                    if (++stage == S) {
                        stage = 0;
                        phase ^= 1u;
                    }
                }
                if (!ok) break;
                if (!SPLIT) {
                    mma_commit(accf_bar(fill & 1));   // ready for the epilogue
                    ++fill;
                }
            }
            // all MMAs issued by this thread complete before TMEM is released
            mma_commit(down_bar);
            const unsigned long long t0 = globaltimer();
            while (!mbar_try_wait(down_bar, 0) && globaltimer() - t0 < kWaitLimitNs) {
            }
        }
    } else {
        // ---------------- epilogue: warpgroup h takes column block h, TMEM lanes 32 * (warp % 4) ----------------
        const int h = (warp - 2) >> 2;
        const int q = warp & 3;
        BlockCtx b;
        b.et = threadIdx.x - 64 - 128 * h;
        b.bar = 1 + h;
        b.stg = smem + kOffStg + h * kStg * STG_BYTES;
        b.row_local = 32 * q + lane;
        float* rj_s = reinterpret_cast<float*>(smem + kOffRj) + h * BM;
        const uint32_t tlane = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(h * BM);
        const float unscale = SPLIT ? a.split->unscale : 1.f;
        int fill = 0, ctr = 0;
        for (long long t = blockIdx.x; t < a.tiles; t += G) {
            int pair;
            tile_coords(t, a.T, a.T2, a.full, &b.rb, &pair);
            b.j = 2 * pair + h;           // 128-column block of K
            b.row = b.rb * BM + b.row_local;
            b.diag = b.rb == b.j;
            // blocks past the matrix and block (2q + 1, 2q) below the diagonal are not stored
            const bool store = b.rb < a.T && b.j < a.T && (a.full || b.rb <= b.j);
            const float ri = (KIND == POPCORN_GAUSSIAN && b.row < a.n) ? a.norms[b.row] : 0.f;
            if (KIND == POPCORN_GAUSSIAN) {   // column norms of this tile's column block j
                const int col = b.j * BM + b.et;
                named_bar<128>(b.bar);   // the warpgroup finished reading the previous tile's
                rj_s[b.et] = col < a.n ? a.norms[col] : 0.f;
                named_bar<128>(b.bar);
            }
            constexpr bool HALF = OUT == kOutHalf16 || OUT == kOutHalfB16;
            auto finish = [&](int c, float (&v)[32]) {
                kappa32<KIND>(v, ri, rj_s + 32 * c, a.kp);
                if (b.diag && (b.row_local >> 5) == c) {
#pragma unroll
                    for (int x = 0; x < 32; ++x)
                        if (x == (b.row_local & 31)) {
                            if (KIND == POPCORN_GAUSSIAN) v[x] = 1.f;
                            if (b.row < a.n) a.kdiag[b.row] = HALF ? round_half(v[x], OUT == kOutHalfB16) : v[x];
                        }
                }
                if (SPLIT && b.diag) store_diag_chunk<OUT>(a, b, a.full && 2 * pair < b.rb, c, v);
                else store_chunk<OUT>(a, b, &map_kd, &map_kt, c, v, ctr);
            };
            bool ok = true;
            if constexpr (SPLIT) {
                // the row's 128 sums, as f32x2 pairs: one chunk of 32 columns of P at a time
                unsigned long long acc[BM / 2];
#pragma unroll
                for (int x = 0; x < BM / 2; ++x) acc[x] = 0ull;
                for (int kb = 0; kb < a.nkb; ++kb, ++fill) {
                    const int ab = fill & 1;
                    const bool got = mbar_wait_for(accf_bar(ab), (uint32_t)(fill >> 1) & 1u, abort_flag, a.err, a.wait_ns);
                    if (__any_sync(0xffffffffu, !got)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t tacc = tlane + (uint32_t)(ab * 2 * BM);
                    const bool last = kb + 2 >= a.nkb;   // rounded away from zero (the reason and figures: file header)
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        uint32_t r[16];
                        tmem_ld16(tacc + 16 * c, r);
                        if (!last) {
#pragma unroll
                            for (int x = 0; x < 8; ++x)
                                acc[8 * c + x] = f2add(acc[8 * c + x], f2pack(__uint_as_float(r[2 * x]),
                                                                              __uint_as_float(r[2 * x + 1])));
                        } else {
#pragma unroll
                            for (int x = 0; x < 8; ++x) {
                                float a0, a1;
                                f2unpack(acc[8 * c + x], a0, a1);
                                acc[8 * c + x] = f2pack(add_away(a0, __uint_as_float(r[2 * x])),
                                                        add_away(a1, __uint_as_float(r[2 * x + 1])));
                            }
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(acce_bar(ab));
                }
                // the warpgroup agrees (one barrier, one AND) before touching staging
                if (!named_bar_all(b.bar, 128, ok && !*abort_flag)) break;
                if (!store) continue;
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    float v[32];
#pragma unroll
                    for (int x = 0; x < 16; ++x) {
                        f2unpack(acc[16 * c + x], v[2 * x], v[2 * x + 1]);
                        v[2 * x] *= unscale;
                        v[2 * x + 1] *= unscale;
                    }
                    finish(c, v);
                }
            } else {
                const int ab = fill & 1;
                ok = mbar_wait_for(accf_bar(ab), (uint32_t)(fill >> 1) & 1u, abort_flag, a.err, a.wait_ns);
                ++fill;
                if (!named_bar_all(b.bar, 128, ok && !*abort_flag)) break;
                tc_fence_after();
                for (int c = 0; c < BM / 32; ++c) {
                    float v[32];
                    tmem_ld32(tlane + (uint32_t)(ab * 2 * BM + 32 * c), v);
                    if (c == BM / 32 - 1) {
                        // accumulator fully read: hand it back to the MMA warp
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(acce_bar(ab));
                    }
                    if (store) finish(c, v);
                }
            }
        }
        if (b.et == 0) bulk_wait_all();
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// FP32 rows -> BF16 operand rows W (BF16X3: 32 columns of hi, then the same 32 of lo, and so on), zero
// padding, FP32 norms of the represented rows.  One warp per row.
__global__ void __launch_bounds__(256) prep_operands_kernel(const float* __restrict__ P, int n, int d, int64_t ldp,
                                                            int dpad, int x3, __nv_bfloat16* __restrict__ W,
                                                            float* __restrict__ norms) {
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (warp >= n) return;
    const int64_t ldw = (int64_t)(x3 ? 2 : 1) * dpad;
    __nv_bfloat16* wr = W + (int64_t)warp * ldw;
    float nrm = 0.f;
    for (int l = lane; l < dpad; l += 32) {
        const int at = x3 ? 2 * (l & ~31) + (l & 31) : l;
        const float p = l < d ? P[(int64_t)warp * ldp + l] : 0.f;
        const __nv_bfloat16 hi = __float2bfloat16_rn(p);
        const float hf = __bfloat162float(hi);
        wr[at] = hi;
        if (!x3) {
            nrm = fmaf(hf, hf, nrm);
        } else {
            const __nv_bfloat16 lo = __float2bfloat16_rn(p - hf);
            const float rep = hf + __bfloat162float(lo);
            wr[at + 32] = lo;
            nrm = fmaf(rep, rep, nrm);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    if (lane == 0) norms[warp] = nrm;
}

// ---- FP32 operands as two FP16 parts (SPLIT) ----------------------------------------------

// The scale, and whether the split build takes the matrix.  s is the power of two that puts
// the largest |p| into [2^14, 2^15).  hi = fp16(s p) keeps 11 bits, lo = fp16(s p - hi) the
// next 11 and a sign while |s p| >= 2^-2: p to 2^-23 of itself.  Below that lo is subnormal and the
// error at most 2^-25.  Every column's largest value must be at least 2^2 (after the scale), and for
// dot products every nonzero row's too: an element's error is then at most 2^-23 of itself or 2^-27
// of its column's and its row's largest value.  (Of the row's: K_ij of two short rows is small too,
// and has to be as exact as FP32 makes it.  Normal points, n = 300, d = 512, one row 1e4, 1e6, 1e7,
// 1e9 times as long: the representation alone puts K_ij of the others off by at most 0.4, 11, 165
// and 10,650 times 2^-24 |p_i| |p_j|, FP32 FMAs by 18.  The Gaussian's distances are compared with
// the largest norm by its own rule, and take no line for rows.)  Columns or rows
// further apart than that (a factor of 4096), values outside 2^+-40 (whose products could
// leave FP32) and non-finite points stay on CUDA cores, and so do dot products of points more than
// 1 / kSplitLowPart of whose nonzero entries are below 2^-2 (counted where the operands are written;
// of normal points it is 1 in 100,000): blocks of columns, each large in other rows, pass
// the maxima, and the products between blocks are of small entries only.  So do dot products of few nonzero
// terms, where FP32 FMAs round less than the truncated chunks: with a fraction f of nonzero
// entries a pair adds about d f^2 of them, and the two errors cross near 20 (measured, linear
// kernel, 80% zeros: d = 256 5.6e-8 in FMAs against 6.8e-8, d = 512 7.4e-8 in both).  The line
// is at 128 terms, four chunks a row: from there the objective of a fit, J = trace K - ..., is
// no further off either (2,000-point clusters, polynomial: d = 100 -3e-7 against -9e-8, d = 128
// -1.0e-7 against -1.3e-7, d = 256 -4e-8 against 1.4e-7).  The Gaussian has no such line: its error is that of the last rounding (3.6e-8
// either way), and the split takes it where the norm expansion applies (kbuild_simt.cu).
constexpr float kSplitMinTerms = 128.f;
constexpr unsigned long long kSplitLowPart = 64;
constexpr int kSplitMinD = 48;   // the Gaussian's line
// (All 256 threads of one block.)
__device__ void split_decide(const unsigned* colmax, const unsigned* rowmax, const unsigned long long* nonzero, int n,
                             int d, const unsigned* maxr, float expand_coef, SplitState* st) {
    __shared__ unsigned mx_s, mn_s;
    if (threadIdx.x == 0) {
        mx_s = 0u;
        mn_s = 0xffffffffu;
    }
    __syncthreads();
    unsigned mx = 0u, mn = 0xffffffffu;   // the largest entry; the smallest nonzero maximum of a column or row
    auto least = [&](unsigned v) { mn = min(mn, v ? v : 0xffffffffu); };
    for (int l = threadIdx.x; l < d; l += blockDim.x) {
        const unsigned v = __ldcg(colmax + l);
        mx = max(mx, v);
        least(v);
    }
    if (rowmax) {
        const uint4* r4 = reinterpret_cast<const uint4*>(rowmax);   // (zeros up to a multiple of four)
#pragma unroll 8
        for (int q = threadIdx.x; q < (n + 3) / 4; q += blockDim.x) {
            const uint4 v = __ldcg(r4 + q);
            least(v.x), least(v.y), least(v.z), least(v.w);
        }
    }
    atomicMax(&mx_s, mx);
    atomicMin(&mn_s, mn);
    __syncthreads();
    if (threadIdx.x) return;
    mx = mx_s;
    mn = mn_s;
    const bool gaussian = !rowmax;
    const unsigned long long nz = __ldcg(nonzero);
    const float fill = (float)nz / ((float)n * (float)d);
    bool use = gaussian ? __uint_as_float(*maxr) * expand_coef <= 1e-6f : (float)d * fill * fill >= kSplitMinTerms;
    int e = 0;   // s = 2^e
    if (mx) {
        e = 14 + 127 - (int)(mx >> 23);
        use = use && mx >= __float_as_uint(0x1p-40f) && mx < __float_as_uint(0x1p40f) &&
              ldexpf(__uint_as_float(mn), e) >= 4.f;
    }
    st->use = use ? 1 : 0;
    st->scale = use ? ldexpf(1.f, e) : 0.f;
    st->unscale = use ? ldexpf(1.f, -2 * e) : 0.f;
    st->low = 0ull;
    st->low_max = gaussian ? ~0ull : nz / kSplitLowPart;
}

// Largest |p| of every column and, where rowmax is given, of every row (bit patterns: non-negative
// floats order like them, and NaN and infinity lie above every finite value), and the number of
// nonzero entries.  A block takes `rows` rows (a multiple of 64) of 128 columns, a warp eight rows at
// a time with a lane to four columns (one 16-byte load each where rows are aligned); its eight row
// maxima leave in one instruction.  (A thread to a column, with a reduction and a shared-memory
// atomic a row of 32 columns, took 70 us at n = 20,000, d = 784.)  The last block to finish takes the
// decision.
constexpr int kScanCols = 128, kScanStep = 64;
__global__ void __launch_bounds__(256) split_scan_kernel(const float* __restrict__ P, int n, int d, int64_t ldp,
                                                         int rows, unsigned* __restrict__ colmax,
                                                         unsigned* __restrict__ rowmax,
                                                         unsigned long long* __restrict__ nonzero, unsigned* ticket,
                                                         const unsigned* maxr, float expand_coef, SplitState* st) {
    __shared__ unsigned cm[8][kScanCols];
    __shared__ int am_last;
    // a Gaussian whose norm expansion does not apply: the state stays as it was cleared, not taken
    if (!rowmax && !(__uint_as_float(*maxr) * expand_coef <= 1e-6f)) return;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t r0 = (int64_t)blockIdx.x * rows, r1 = r0 + rows < n ? r0 + rows : n;
    const bool vec = (ldp & 3) == 0 && ((uintptr_t)P & 15) == 0;
    unsigned nz = 0u;
    for (int c0 = blockIdx.y * kScanCols; c0 < d; c0 += gridDim.y * kScanCols) {
        const int l = c0 + 4 * lane;
        unsigned m[4] = {0u, 0u, 0u, 0u};
        for (int64_t r = r0 + 8 * warp; r < r1; r += kScanStep) {
            float v[8][4];
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                const float* p = P + (r + x < r1 ? r + x : r1 - 1) * ldp + l;   // (past the end: the last row again)
                if (vec && l + 3 < d) {
                    const float4 f = __ldg(reinterpret_cast<const float4*>(p));
                    v[x][0] = f.x, v[x][1] = f.y, v[x][2] = f.z, v[x][3] = f.w;
                } else {
#pragma unroll
                    for (int y = 0; y < 4; ++y) v[x][y] = l + y < d ? __ldg(p + y) : 0.f;
                }
            }
            unsigned mine = 0u;
#pragma unroll
            for (int x = 0; x < 8; ++x) {
                unsigned w = 0u;
#pragma unroll
                for (int y = 0; y < 4; ++y) {
                    const unsigned b = __float_as_uint(v[x][y]) & 0x7fffffffu;
                    m[y] = max(m[y], b);
                    w = max(w, b);
                    nz += b != 0u && r + x < r1;
                }
                if (rowmax) {
                    w = __reduce_max_sync(0xffffffffu, w);
                    if (lane == x) mine = w;
                }
            }
            if (rowmax && lane < 8 && r + lane < r1 && mine) atomicMax(rowmax + r + lane, mine);
        }
#pragma unroll
        for (int y = 0; y < 4; ++y) cm[warp][4 * lane + y] = m[y];
        __syncthreads();
        if (threadIdx.x < kScanCols && c0 + (int)threadIdx.x < d) {
            unsigned t = 0u;
#pragma unroll
            for (int w = 0; w < 8; ++w) t = max(t, cm[w][threadIdx.x]);
            if (t) atomicMax(colmax + c0 + threadIdx.x, t);
        }
        __syncthreads();
    }
    nz = __reduce_add_sync(0xffffffffu, nz);
    if (lane == 0 && nz) atomicAdd(nonzero, (unsigned long long)nz);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) am_last = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1;
    __syncthreads();
    if (!am_last) return;
    __threadfence();
    split_decide(colmax, rowmax, nonzero, n, d, maxr, expand_coef, st);
}

// FP32 rows -> W in FP16, hi and lo by 32 columns as above, zero padding.  A thread takes four columns of
// a row (float4 loads when rows are 16-byte aligned), 8-byte stores.
__global__ void __launch_bounds__(256) split_operands_kernel(const float* __restrict__ P, int n, int d, int64_t ldp,
                                                             int dpad, SplitState* st, __half* __restrict__ W) {
    grid_dependency_wait();
    if (!st->use) return;
    const float s = st->scale;
    unsigned low = 0u;
    const bool vec = (ldp & 3) == 0 && ((uintptr_t)P & 15) == 0;
    const int q4 = dpad / 4;
    const int64_t total = (int64_t)n * q4, step = (int64_t)gridDim.x * blockDim.x;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += step) {
        const int64_t r = t / q4;
        const int l = 4 * (int)(t - r * q4);
        const float* p = P + r * ldp + l;
        float v[4];
        if (vec && l + 3 < d) {
            const float4 f = __ldg(reinterpret_cast<const float4*>(p));
            v[0] = f.x, v[1] = f.y, v[2] = f.z, v[3] = f.w;
        } else {
#pragma unroll
            for (int x = 0; x < 4; ++x) v[x] = l + x < d ? __ldg(p + x) : 0.f;
        }
        __half2 hi[2], lo[2];
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const float f0 = v[2 * x] * s, f1 = v[2 * x + 1] * s;
            low += (f0 != 0.f && fabsf(f0) < 0.25f) + (f1 != 0.f && fabsf(f1) < 0.25f);
            hi[x] = __floats2half2_rn(f0, f1);
            const float2 h = __half22float2(hi[x]);
            lo[x] = __floats2half2_rn(f0 - h.x, f1 - h.y);
        }
        __half* w = W + r * (2 * (int64_t)dpad) + 2 * (l & ~31) + (l & 31);
        *reinterpret_cast<uint2*>(w) = *reinterpret_cast<const uint2*>(hi);
        *reinterpret_cast<uint2*>(w + 32) = *reinterpret_cast<const uint2*>(lo);
    }
    low = __reduce_add_sync(0xffffffffu, low);
    if ((threadIdx.x & 31) == 0 && low) atomicAdd(&st->low, (unsigned long long)low);
}

}  // namespace

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
        cudaGetLastError();
    }
    return fn;
}

bool make_tensor_map_2d(CUtensorMap* m, CUtensorMapDataType dt, void* base, uint64_t inner, uint64_t outer,
              uint64_t row_bytes, uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle sw) {
    auto fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {inner, outer};
    cuuint64_t strides[1] = {row_bytes};
    cuuint32_t box[2] = {box_inner, box_outer};
    cuuint32_t es[2] = {1, 1};
    return fn(m, dt, 2, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}


size_t kbuild_tc_workspace(int n, int d, int precision) {
    const size_t dpad = ((size_t)d + 63) / 64 * 64;
    const size_t ldw = (precision == POPCORN_BF16X3 ? 2 : 1) * dpad;
    const size_t ops = (size_t)n * ldw * 2;
    return ((ops + 255) & ~(size_t)255) + (size_t)n * 4 + 256;
}

namespace {

using TcFn = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, TcArgs);

template <int MODE, int OUT>
TcFn tc_fn_kind(int kind) {
    switch (kind) {
        case POPCORN_LINEAR: return kbuild_tc_kernel<MODE, OUT, POPCORN_LINEAR>;
        case POPCORN_POLYNOMIAL: return kbuild_tc_kernel<MODE, OUT, POPCORN_POLYNOMIAL>;
        default: return kbuild_tc_kernel<MODE, OUT, POPCORN_GAUSSIAN>;
    }
}
template <int MODE>
TcFn tc_fn_out(int out, int kind) {
    if constexpr (MODE != kModeSplit) {   // (SPLIT: FP32 K only)
        if (out == kOutHalf16) return tc_fn_kind<MODE, kOutHalf16>(kind);
        if (out == kOutHalfB16) return tc_fn_kind<MODE, kOutHalfB16>(kind);
    }
    if (out == kOutSw16) return tc_fn_kind<MODE, kOutSw16>(kind);
    if (out == kOutSw4) return tc_fn_kind<MODE, kOutSw4>(kind);
    return tc_fn_kind<MODE, kOutFull>(kind);
}
TcFn tc_fn(int mode, int out, int kind) {
    if (mode == kModeSplit) return tc_fn_out<kModeSplit>(out, kind);
    return mode == kModeX3 ? tc_fn_out<kModeX3>(out, kind) : tc_fn_out<kModeBf16>(out, kind);
}

}  // namespace

cudaError_t configure_kbuild_tc() {
    encode_fn();
    for (int mode = kModeBf16; mode <= kModeSplit; ++mode)
        for (int out = kOutFull; out <= (mode == kModeSplit ? kOutSw4 : kOutHalfB16); ++out)
            for (int kind = POPCORN_LINEAR; kind <= POPCORN_GAUSSIAN; ++kind) {
                const cudaError_t e = cudaFuncSetAttribute(tc_fn(mode, out, kind),
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
                if (e != cudaSuccess) return e;
            }
    return cudaSuccess;
}

namespace {

// The tile kernel on operand rows W (n x ldw 16-bit elements).
cudaError_t launch_tiles(int mode, const void* W, int n, int64_t ldw, int dpad, const SplitState* split,
                         const KernParams& kp, const float* norms, float* K, int64_t ldk, float* kdiag, int* err,
                         int num_sms, cudaStream_t s, int out, int full) {
    CUtensorMap mr, mc, mkd, mkt;
    memset(&mkd, 0, sizeof mkd);
    memset(&mkt, 0, sizeof mkt);
    const CUtensorMapDataType dt = split ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    void* w = const_cast<void*>(W);
    const CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_128B;
    if (!make_tensor_map_2d(&mr, dt, w, (uint64_t)ldw, (uint64_t)n, (uint64_t)ldw * 2, kRowElems, BM, sw) ||
        !make_tensor_map_2d(&mc, dt, w, (uint64_t)ldw, (uint64_t)n, (uint64_t)ldw * 2, kRowElems, 2 * BM, sw))
        return cudaErrorInvalidValue;
    // the full-square stores go through tensor maps; the packed stores are plain bulk copies
    if (out == kOutFull && (!make_tensor_map_2d(&mkd, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, K, (uint64_t)n, (uint64_t)n,
                                                (uint64_t)ldk * 4, 16, BM, CU_TENSOR_MAP_SWIZZLE_64B) ||
                            !make_tensor_map_2d(&mkt, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, K, (uint64_t)n, (uint64_t)n,
                                                (uint64_t)ldk * 4, BM, 16, CU_TENSOR_MAP_SWIZZLE_NONE)))
        return cudaErrorInvalidValue;
    TcArgs a;
    a.n = n;
    a.T = (n + BM - 1) / BM;
    a.T2 = (a.T + 1) / 2;
    a.nkb = dpad / kbuild_dk(mode);
    a.full = full;
    a.tiles = tile_count(a.T, a.T2, a.full);
    a.K = K;
    a.ldk = ldk;
    a.Kp = out == kOutFull ? nullptr : K;
    a.kp = kp;
    a.norms = norms;
    a.kdiag = kdiag;
    a.split = split;
    a.err = err;
    // Error-path test hook: POPCORN_TEST_BUILD_STALL_MS=<ms> in the environment makes one wait of every
    // tensor-core build run out.  Unset in every ordinary run.
    const char* env = getenv("POPCORN_TEST_BUILD_STALL_MS");
    const int stall_ms = env && *env ? atoi(env) : 0;
    a.stall = stall_ms > 0 && stall_ms <= 10000 ? 1 : 0;
    a.wait_ns = a.stall ? (unsigned long long)stall_ms * 1000000ull : kWaitLimitNs;
    const int grid = (int)(a.tiles < num_sms ? a.tiles : num_sms);
    return launch_pdl(tc_fn(mode, out, kp.kind), dim3(grid), dim3(NTHREADS), kSmemBytes, s, mr, mc, mkd, mkt, a);
}

int packed_out(int packed) { return packed == kPackedSw4 ? kOutSw4 : packed == kPackedSw16 ? kOutSw16 : kOutFull; }

}  // namespace

cudaError_t launch_kbuild_tc(const float* P, int n, int d, int64_t ldp, KernParams kp, int precision, float* K,
                             int64_t ldk, float* kdiag, void* workspace, int* err, int num_sms, cudaStream_t s,
                             int* launches, int packed, int full, int k_storage) {
    // packed kPackedSw128H: K is the FP16 / BF16 packed triangle (k_storage)
    int out = packed_out(packed);
    if (packed == kPackedSw128H) {
        if (k_storage != POPCORN_K_FP16 && k_storage != POPCORN_K_BF16) return cudaErrorInvalidValue;
        out = k_storage == POPCORN_K_BF16 ? kOutHalfB16 : kOutHalf16;
    }
    const int x3 = precision == POPCORN_BF16X3 ? 1 : 0;
    const int dk = kbuild_dk(x3 ? kModeX3 : kModeBf16), dpad = (d + dk - 1) / dk * dk;
    const int64_t ldw = (int64_t)(x3 ? 2 : 1) * dpad;
    __nv_bfloat16* W = static_cast<__nv_bfloat16*>(workspace);
    const size_t ops = (size_t)n * ldw * 2;
    float* norms = reinterpret_cast<float*>(static_cast<char*>(workspace) + ((ops + 255) & ~(size_t)255));

    prep_operands_kernel<<<(unsigned)(((int64_t)n * 32 + 255) / 256), 256, 0, s>>>(P, n, d, ldp, dpad, x3, W, norms);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_tiles(x3 ? kModeX3 : kModeBf16, W, n, ldw, dpad, nullptr, kp, norms, K, ldk, kdiag, err, num_sms, s, out,
                     full && !packed ? 1 : 0);
    if (launches) *launches += 2;
    return e;
}

// Where the split build is the faster one.  The CUDA-core build takes its tiles in waves, each
// as long as d; the split build costs four more launches (15 to 20 us, also where it refuses the
// points) and then a small fraction of that.  Measured (a whole call, us, CUDA cores / split): n = 2,000: d = 400 78 / 77,
// 512 89 / 78, 784 109 / 91; n = 4,000: d = 128 91 / 88, 256 140 / 95; n = 6,000: d = 48 90 / 101,
// 96 127 / 103; n = 8,000: d = 64 154 / 134, 784 953 / 266; n = 20,000: d = 48 609 / 441,
// 784 5397 / 1163.  Below 128 columns the device's rule on the number of terms refuses dot
// products (linear, polynomial) anyway.
bool kbuild_split_applies(int n, int d, bool dot) {
    const long long T = (n + BM - 1) / BM, tiles = T * (T + 1) / 2;
    return d >= (dot ? (int)kSplitMinTerms : kSplitMinD) && (tiles < 136 ? 136 : tiles) * d >= 65000;
}

size_t kbuild_split_workspace(int n, int d) {
    const size_t dpad = ((size_t)d + 31) / 32 * 32;
    return (((size_t)n * 2 * dpad * 2 + 255) & ~(size_t)255) + (((size_t)d * 4 + 255) & ~(size_t)255) +
           ((size_t)n + 3) / 4 * 16 + 512;
}

cudaError_t launch_kbuild_split(const float* P, int n, int d, int64_t ldp, KernParams kp, float* K, int64_t ldk,
                                float* kdiag, void* workspace, const float* rn, const unsigned* maxr,
                                float expand_coef, int* err, int num_sms, cudaStream_t s, int* launches, int packed,
                                int full, const SplitState** state) {
    const int dpad = (d + 31) / 32 * 32;
    unsigned char* w = static_cast<unsigned char*>(workspace);
    const size_t ops = ((size_t)n * 2 * dpad * 2 + 255) & ~(size_t)255;
    const size_t cols = ((size_t)d * 4 + 255) & ~(size_t)255;
    __half* W = reinterpret_cast<__half*>(w);
    unsigned long long* nonzero = reinterpret_cast<unsigned long long*>(w + ops);
    unsigned* ticket = reinterpret_cast<unsigned*>(w + ops + 64);
    unsigned* colmax = reinterpret_cast<unsigned*>(w + ops + 256);
    SplitState* st = reinterpret_cast<SplitState*>(w + ops + 128);
    const bool dot = kp.kind != POPCORN_GAUSSIAN;
    unsigned* rowmax = dot ? reinterpret_cast<unsigned*>(w + ops + 256 + cols) : nullptr;
    cudaError_t e = cudaMemsetAsync(w + ops, 0, 256 + cols + (dot ? ((size_t)n + 3) / 4 * 16 : 0), s);
    if (e != cudaSuccess) return e;
    // about eight blocks an SM over (rows, columns)
    const int cy = (d + kScanCols - 1) / kScanCols;
    int64_t rows = ((int64_t)n * cy + 8 * num_sms - 1) / (8 * num_sms);
    rows = ((rows < n ? rows : n) + kScanStep - 1) / kScanStep * kScanStep;
    split_scan_kernel<<<dim3((unsigned)((n + rows - 1) / rows), (unsigned)(cy < 65535 ? cy : 65535)), 256, 0, s>>>(
        P, n, d, ldp, (int)rows, colmax, rowmax, nonzero, ticket, maxr, expand_coef, st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t work = (int64_t)n * (dpad / 4);
    const int64_t blocks = (work + 255) / 256;
    e = launch_pdl(split_operands_kernel, dim3((unsigned)(blocks < 16 * num_sms ? blocks : 16 * num_sms)), dim3(256), 0, s,
                   P, n, d, ldp, dpad, st, W);
    if (e != cudaSuccess) return e;
    e = launch_tiles(kModeSplit, W, n, 2 * (int64_t)dpad, dpad, st, kp, rn, K, ldk, kdiag, err, num_sms, s,
                     packed_out(packed), full && !packed ? 1 : 0);
    if (launches) *launches += 3;
    *state = st;
    return e;
}

}  // namespace popcorn
