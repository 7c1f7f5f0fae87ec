// K stream over the block-packed triangle with a lane to a row: S_ic = sum_{j in L_c} K_ij (the
// SpMM of Alg. 2 line 7) for any number of clusters, FP32 K.  Used by fits with more than 32
// clusters and by batched mode.
//
// A unit is a 128-row block I of K against a run of its column blocks J.  The four warps of a CTA
// own 32 rows each: lane l of warp g owns row 32 g + l and its k sums in shared memory
// (acc[c][row]: bank = lane), all lanes are at the same column at a time, whose label is one
// value for the warp, and nothing is added up across lanes.  K is stored as the packed upper
// triangle (kPackedSw4): block (I, J) is tile (I, J) for I <= J, and for I > J the transpose of
// tile (J, I), which the XOR-32 layout reads as easily (a column and a row of a box are both 32
// different banks).  A producer thread bulk-copies 16 KB pieces, 32 columns of the block, through
// a ring: one box of the tile, or, transposed, 32 rows of its four boxes.
//
// Each tile is read twice, once for its rows and once for its columns, by the CTAs of blocks I
// and J.  Block row I takes its columns in the order J = (s - I) mod T, s = 0, 1, ..., so both
// are at that tile in the same step s: the second read finds it in L2, and HBM delivers half of
// the square a pass, without the slots that the one-read symmetric pass writes for its column
// sums (their bytes grow with k).
//
// What bounds it: the chain of a warp's shared-memory additions, with k x 512 bytes of sums a CTA
// (2 CTAs an SM at k = 100, 3 at 64) to hide it behind; without the additions the stream takes
// 0.49 ms where it takes 0.71 (k = 100, n = 30,011; HBM delivers 2.05 GB of the 3.6 GB square).
// Two warps a row group, half a piece's columns each with sums of their own (16 consumer warps an
// SM in place of 12 at k = 64, 8 in one CTA at 100), were slower: 142 -> 153 ms for the batch below
// (30 passes), 27.0 -> 32.2 ms for 30 passes here.
// So the labels come as byte offsets with the piece (the record below: no label arithmetic, no
// global load) and four columns of different labels are added together.  The row-major stream it
// replaces (iterate.cu: a lane every 32nd float4, k x 32 sums to add up a row, 15 instructions an
// element) took 1.09 ms there, 0.81 at k = 64 (now 0.63), 0.79 at 40 (0.51) and 1.75 at 200
// (1.31).  Batch of 256 instances, n 500 to 8,000, k up to 64: 4.7 -> 3.6 ms a pass.  A first form
// with 32 x 32 pieces of row-major rows (128 bytes at a 120 KB stride) stayed at 3.2 TB/s.
//
// Every so many column blocks a cluster's sums join the segment's, a pair of floats (Srun) until the
// unit's end; the segments are added in float-float too.  How often goes by the cluster's size m:
// after 4 sqrt(m) of its columns (at least 32), rounded to a power of two of blocks (tile_plan).  A
// chain of L additions of one size is off by about 0.4 u sqrt(L / 3) of its own sum (u = 2^-24), m / L
// such chains by 0.4 u L / sqrt(3 m), and L = 4 sqrt(2 m) makes that the 1.3 u of the row-major stream
// (32 lanes' partial sums, added one after the other): so S is no further off than there for clusters
// of any size, with few joins.
// A cluster that holds four times its share of a block's columns (points in the order of their
// classes) joins at the block's end, and equal labels among four columns are added up first.  (As runs
// of 64 k columns for all clusters, joined in FP32, a row's sum over one cluster of 30,011 was 1.5e-6
// off at k = 100 and 4.5e-6 at 256; now below 2.6e-7.  There are fewer joins of clusters of one size now,
// and equal labels do not wait for one another: 30 passes at n = 30,011, k = 40 20.9 -> 19.4 ms, 64
// 25.4 -> 23.7, 100 27.0 -> 26.5, with 97% in one cluster 27.6 -> 27.3; the batch below 146 -> 136.)
#include <algorithm>
#include <cmath>

#include "popcorn_internal.cuh"
#include "stream_common.cuh"
#include "tc_common.cuh"

namespace popcorn {
namespace {

using namespace stream;
using namespace tc;

constexpr int kTilesThreads = 160;        // four consumer warps, one producer
constexpr int kPiece = 16 * 1024;         // 32 columns x 128 rows
constexpr int kRecord = kTilesRecord;     // the piece's labels: 32 byte offsets into a row of sums (label x 512), then
                                          // a word whose bit m says that columns 4 m .. 4 m + 3 have four labels, and, in
                                          // a block's last piece, 12 bytes: the number of clusters that hold far more of
                                          // the block than their share, and their labels
constexpr int kDense = 11;                // the most of those
constexpr int kPlanUpto = 16;             // the plan behind the records: upto[j], the clusters that join every 2^j
constexpr int kPlanBytes = 4 * kPlanUpto + kMaxClusters;   // blocks or more often; the clusters, in that order
constexpr int kStage = kPiece + 256;
constexpr int kTilesMaxStages = 4;
constexpr int kTilesBars = 2 * kTilesMaxStages;

struct TilesArgs {
    // one fit
    const float* K;
    int n, k, T, nseg, segblocks;
    const uint8_t* lab8;
    const unsigned char* rec;
    float* Spart;
    float2* Srun;
    double* zpart;
    double* zsum;
    double* cnorm;
    double* invm;
    const int32_t* counts;
    LoopState* st;
    double* J_hist;
    // a batch
    const BatchInst* I;
    const int2* units;     // (instance, segment x T + row block)
    int nunits;
    int eval_only, stages, kmax;
    int* err;
    // Error-path tests only (0 in every ordinary launch): CTA 0 leaves its first copy out and every
    // wait of the launch gives up after wait_ns.
    int stall;
    unsigned long long wait_ns;
};

// What one unit reads and writes.
struct TileUnit {
    const unsigned char* K;   // packed triangle
    const unsigned char* rec; // the pieces' label records
    const uint8_t* lab;
    float* S;                 // this segment's sums [c][i]
    float2* run;              // and, while they grow, pairs of floats
    int n, k, T, I, s0, s1;
};

__device__ __forceinline__ const unsigned char* tile_at(const TileUnit& u, int I, int J) {
    return u.K + ((size_t)I * u.T - (size_t)I * (I - 1) / 2 + (size_t)(J - I)) * 65536;
}

__device__ __forceinline__ float lds(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts(uint32_t addr, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v));
}

__device__ __forceinline__ uint4 lds4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) { return __float_as_uint(lds(addr)); }

// Adds four consecutive columns of this lane's row to its sums (acc: shared address; o: the
// columns' offsets from it, one value each for the warp).  apart: the four labels differ, so the
// additions do not wait for one another.
__device__ __forceinline__ void add4(uint32_t acc, const uint4& o, bool apart, float v0, float v1, float v2, float v3) {
    const uint32_t p0 = acc + o.x, p1 = acc + o.y, p2 = acc + o.z, p3 = acc + o.w;
    if (apart) {
        const float a0 = lds(p0), a1 = lds(p1), a2 = lds(p2), a3 = lds(p3);
        sts(p0, a0 + v0);
        sts(p1, a1 + v1);
        sts(p2, a2 + v2);
        sts(p3, a3 + v3);
    } else {
        // equal labels are added up first
        const float a0 = lds(p0), a1 = lds(p1), a2 = lds(p2), a3 = lds(p3);
        float s3 = v3, s2 = v2, s1 = v1, s0 = v0;
        s2 = p2 == p3 ? s2 + s3 : s2;
        s0 = p0 == p1 ? s0 + s1 : s0;
        const float r0 = a0 + (p0 == p2 ? s0 + s2 : p0 == p3 ? s0 + s3 : s0);
        const float r1 = a1 + (p1 == p2 ? s1 + s2 : p1 == p3 ? s1 + s3 : s1);
        sts(p3, a3 + s3);
        sts(p2, a2 + s2);
        sts(p1, r1);
        sts(p0, r0);
    }
}

// The plan of a pass, by one block: after how many column blocks (2^j) each cluster's sums join the
// segment's, as an order of the clusters by j (equal ones in any order: their sums are their own).
__device__ __forceinline__ void tile_plan(int n, int k, const int32_t* __restrict__ m, unsigned char* plan) {
    __shared__ int upto[kPlanUpto], at[kPlanUpto];
    if (threadIdx.x < kPlanUpto) upto[threadIdx.x] = 0;
    __syncthreads();
    int js[(kMaxClusters + 127) / 128];
#pragma unroll
    for (int x = 0; x < (kMaxClusters + 127) / 128; ++x) {
        const int c = threadIdx.x + 128 * x;
        js[x] = kPlanUpto - 1;   // an empty cluster, or none
        if (c < k && m[c] > 0) {
            const float mc = (float)m[c], blocks = fmaxf(32.f, 4.f * sqrtf(mc)) * (float)n / (128.f * mc);
            js[x] = min(kPlanUpto - 2, max(0, (int)floorf(log2f(blocks) + 0.5f)));
        }
        if (c < k) atomicAdd(&upto[js[x]], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int j = 0; j < kPlanUpto; ++j) {
            at[j] = t;
            t += upto[j];
            upto[j] = t;
        }
    }
    __syncthreads();
#pragma unroll
    for (int x = 0; x < (kMaxClusters + 127) / 128; ++x) {
        const int c = threadIdx.x + 128 * x;
        if (c < k) plan[4 * kPlanUpto + atomicAdd(&at[js[x]], 1)] = (unsigned char)c;
    }
    if (threadIdx.x < kPlanUpto) reinterpret_cast<int*>(plan)[threadIdx.x] = upto[threadIdx.x];
}

// The label records of column block J, a warp a piece of 32 columns (past n: label 0, never added),
// and the clusters that hold more than four times their share of it and 10 columns.  m: the clusters'
// sizes.
__device__ __forceinline__ void write_records(const uint8_t* __restrict__ lab, int n, int k, int J,
                                              const int32_t* __restrict__ m, unsigned char* rec) {
    __shared__ int hist[kMaxClusters], dense;
    for (int c = threadIdx.x; c < k; c += blockDim.x) hist[c] = 0;
    if (threadIdx.x == 0) dense = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, piece = 4 * J + (threadIdx.x >> 5), pieces = (n + 31) / 32;
    if (piece < pieces) {
        const int col = 32 * piece + lane;
        const uint32_t l = col < n ? lab[col] : 0u;
        // (every lane takes part in every exchange)
        const uint32_t l1 = __shfl_xor_sync(0xffffffffu, l, 1), l2 = __shfl_xor_sync(0xffffffffu, l, 2),
                       l3 = __shfl_xor_sync(0xffffffffu, l, 3);
        const unsigned eq = __ballot_sync(0xffffffffu, l == l1 || l == l2 || l == l3);
        if (col < n) atomicAdd(&hist[l], 1);
        uint32_t* r = reinterpret_cast<uint32_t*>(rec + (size_t)piece * kRecord);
        r[lane] = l * 512u;
        if (lane < 4) {
            unsigned f = 0u;
            for (int q = 0; q < 8; ++q) f |= (eq >> (4 * q) & 15u ? 0u : 1u) << q;
            r[32 + lane] = lane == 0 ? f : 0u;
        }
    }
    __syncthreads();
    unsigned char* list = rec + (size_t)min(4 * J + 3, pieces - 1) * kRecord + 4 * 33;
    for (int c = threadIdx.x; c < k; c += blockDim.x)
        if (hist[c] > 10 && (float)hist[c] > 512.f * (float)m[c] / (float)n + 10.f)
            list[1 + atomicAdd(&dense, 1)] = (unsigned char)c;   // (11 columns each, of 128: at most kDense)
    __syncthreads();
    if (threadIdx.x == 0) list[0] = (unsigned char)dense;
    if (J == 0) tile_plan(n, k, m, rec + (size_t)pieces * kRecord);
}
__global__ void __launch_bounds__(128) tile_records_kernel(const uint8_t* __restrict__ lab, int n, int k,
                                                           const int32_t* __restrict__ counts, unsigned char* rec,
                                                           const LoopState* st, int eval) {
    if (pass_skip(st, eval)) return;
    write_records(lab, n, k, (int)blockIdx.x, counts + (size_t)(st->iter & 1) * k, rec);
}
// a block a 128-column block of an instance
__global__ void __launch_bounds__(128) batched_records_kernel(const BatchInst* I, int count, int eval) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (I[mid].vblock0 <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const BatchInst& b = I[lo];
    if (pass_skip(b.st, eval)) return;
    write_records(b.lab8, b.n, b.k, (int)blockIdx.x - b.vblock0, b.counts + (size_t)(b.st->iter & 1) * b.k, b.V);
}

template <bool BATCH, int CTAS>
__global__ void __launch_bounds__(kTilesThreads, CTAS) reduce_tiles_kernel(TilesArgs a) {
    if constexpr (!BATCH) {
        if (pass_skip(a.st, a.eval_only)) {
            // J(final labels) is already known when the last pass changed nothing
            if (a.eval_only && blockIdx.x == 0 && threadIdx.x == 0) a.st->J_eval = a.st->J_last;
            return;
        }
    }
    extern __shared__ __align__(1024) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, S = a.stages;
    // ring | sums [kmax][128] | float-float z partials [4][k] hi, lo (one fit)
    float* acc_s = reinterpret_cast<float*>(smem + S * kStage);
    float* zhi = acc_s + (size_t)a.kmax * 128;
    float* zlo = zhi + 4 * a.kmax;
    __shared__ __align__(8) unsigned long long bars[kTilesBars];
    __shared__ int abort_s;
    volatile int* abort_flag = &abort_s;
    const uint32_t bar0 = smem_u32(bars), ring = smem_u32(smem);
    auto full_bar = [&](int s) { return bar0 + 8u * s; };
    auto empty_bar = [&](int s) { return bar0 + 8u * (kTilesMaxStages + s); };
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_bar(s), 1);
            mbar_init(empty_bar(s), 4);
        }
        abort_s = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int nunits = BATCH ? a.nunits : a.T * a.nseg;
    // unit x: its geometry; false when its instance has stopped
    auto unit = [&](int x, TileUnit* u) -> bool {
        int q;
        if constexpr (BATCH) {
            const int2 w = a.units[x];
            const BatchInst& b = a.I[w.x];
            if (pass_skip(b.st, a.eval_only)) return false;
            q = w.y / b.T;
            u->I = w.y - q * b.T;
            u->K = reinterpret_cast<const unsigned char*>(b.K);
            u->lab = b.lab8;
            u->rec = b.V;
            u->n = b.n;
            u->k = b.k;
            u->T = b.T;
            u->s0 = q * (b.seglen >> 7);
            u->s1 = min(b.T, u->s0 + (b.seglen >> 7));
            u->S = b.Spart + (size_t)q * b.k * b.n;
            u->run = b.Srun + (size_t)q * b.k * b.n;
        } else {
            q = x / a.T;
            u->I = x - q * a.T;
            u->K = reinterpret_cast<const unsigned char*>(a.K);
            u->lab = a.lab8;
            u->rec = a.rec;
            u->n = a.n;
            u->k = a.k;
            u->T = a.T;
            u->s0 = q * a.segblocks;
            u->s1 = min(a.T, u->s0 + a.segblocks);
            u->S = a.Spart + (size_t)q * a.k * a.n;
            u->run = a.Srun + (size_t)q * a.k * a.n;
        }
        return true;
    };
    int stage = 0;
    uint32_t phase = 0;
    auto advance = [&]() {
        if (++stage == S) {
            stage = 0;
            phase ^= 1u;
        }
    };
    if (warp == 4) {
        if (lane == 0) {
            // ---------------- producer ----------------
            uint32_t issued = 0, issued_par = 0;
            bool ok = true, first = true;
            for (int x = blockIdx.x; x < nunits && ok; x += gridDim.x) {
                TileUnit u;
                if (!unit(x, &u)) continue;
                for (int s = u.s0; s < u.s1 && ok; ++s) {
                    const int J = s >= u.I ? s - u.I : s - u.I + u.T;
                    const bool rows = u.I <= J;
                    const unsigned char* t = rows ? tile_at(u, u.I, J) : tile_at(u, J, u.I);
                    for (int p = 0; p < 4 && 128 * J + 32 * p < u.n; ++p) {
                        if (!mbar_wait_for(empty_bar(stage), phase ^ 1u, abort_flag, a.err, a.wait_ns)) {
                            ok = false;
                            break;
                        }
                        if (!(a.stall && blockIdx.x == 0 && first)) {
                            mbar_arrive_expect_tx(full_bar(stage), kPiece + kRecord);
                            const uint32_t dst = ring + (uint32_t)(stage * kStage);
                            bulk_load_1d(dst + kPiece, u.rec + (size_t)(4 * J + p) * kRecord, kRecord, full_bar(stage));
                            if (rows) {
                                bulk_load_1d(dst, t + p * kPiece, kPiece, full_bar(stage));
                            } else {
#pragma unroll
                                for (int g = 0; g < 4; ++g)
                                    bulk_load_1d(dst + 4096u * g, t + g * kPiece + p * 4096, 4096, full_bar(stage));
                            }
                            issued |= 1u << stage;
                            issued_par = (issued_par & ~(1u << stage)) | (phase << stage);
                        }
                        first = false;
                        advance();
                    }
                }
            }
            if (!ok) {
                // aborted: let this CTA's own copies land before shared memory goes away
                for (int s = 0; s < S; ++s)
                    if (issued >> s & 1u) {
                        const unsigned long long t0 = globaltimer();
                        while (!mbar_try_wait(full_bar(s), issued_par >> s & 1u) && globaltimer() - t0 < kWaitLimitNs) {
                        }
                    }
            }
        }
    } else {
        // ---------------- consumers: warp g takes rows 32 g .. 32 g + 31 of the block ----------------
        const int g = warp;
        const uint32_t acc_u = smem_u32(acc_s + 32 * g + lane);   // (this lane's sums: only it reads and writes them)
        float* zwh = zhi + g * a.kmax;
        float* zwl = zlo + g * a.kmax;
        for (int c = 0; c < a.kmax; ++c) sts(acc_u + 512u * c, 0.f);
        if (!BATCH)
            for (int c = lane; c < a.kmax; c += 32) zwh[c] = zwl[c] = 0.f;
        __syncwarp();
        bool ok = true;
        for (int x = blockIdx.x; x < nunits && ok; x += gridDim.x) {
            TileUnit u;
            if (!unit(x, &u)) continue;
            const int i = 128 * u.I + 32 * g + lane;
            const int li = i < u.n ? (int)u.lab[i] : -1;
            float own = 0.f;   // (one fit) the row's sum over its own cluster
            float* out = u.S + i;
            float2* run = u.run + i;
            const int* upto = reinterpret_cast<const int*>(u.rec + (size_t)((u.n + 31) / 32) * kRecord);
            const unsigned* order = reinterpret_cast<const unsigned*>(upto + kPlanUpto);   // four clusters a word
            // clusters, from the front of the order, whose sums have joined by the end of step t
            auto joined = [&](int t) { return t > 0 ? __ldg(upto + (31 - __clz(t))) : 0; };
            bool all = false;    // all clusters' entries of run are set
            for (int s = u.s0; s < u.s1 && ok; ++s) {
                const int J = s >= u.I ? s - u.I : s - u.I + u.T;
                const bool rows = u.I <= J;
                unsigned d0 = 0u, d1 = 0u, d2 = 0u;   // the block's dense clusters: number and labels
                for (int p = 0; p < 4 && 128 * J + 32 * p < u.n; ++p) {
                    const int col = 128 * J + 32 * p;
                    const bool got = mbar_wait_for(full_bar(stage), phase, abort_flag, a.err, a.wait_ns);
                    if (__any_sync(0xffffffffu, !got)) {
                        ok = false;
                        break;
                    }
                    // column x of the piece: row 32 g + lane of a box at x ^ lane, or (transposed) row x
                    // of box g at lane ^ x
                    const uint32_t st = ring + (uint32_t)(stage * kStage), rec = st + kPiece;
                    d0 = lds_u32(rec + 132);
                    if (d0) {
                        d1 = lds_u32(rec + 136);
                        d2 = lds_u32(rec + 140);
                    }
                    const uint32_t at = st + (uint32_t)((rows ? (32 * g + lane) * 128 : g * 4096) + 4 * lane);
                    if (col + 32 <= u.n) {
                        float v[32];
                        if (rows) {
#pragma unroll
                            for (int x2 = 0; x2 < 32; ++x2) v[x2] = lds(at ^ (4u * x2));
                        } else {
#pragma unroll
                            for (int x2 = 0; x2 < 32; ++x2) v[x2] = lds((at ^ (4u * x2)) + 128u * x2);
                        }
                        const uint32_t flags = lds_u32(rec + 128);
#pragma unroll
                        for (int m = 0; m < 8; ++m)
                            add4(acc_u, lds4(rec + 16 * m), flags >> m & 1u, v[4 * m], v[4 * m + 1], v[4 * m + 2],
                                 v[4 * m + 3]);
                    } else {
                        // the last columns of a ragged matrix (entries past n are not K)
                        for (int x2 = 0; x2 < u.n - col; ++x2) {
                            const uint32_t p = acc_u + lds_u32(rec + 4 * x2);
                            sts(p, lds(p) + lds((at ^ (4u * x2)) + (rows ? 0u : 128u * x2)));
                        }
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty_bar(stage));
                    advance();
                }
                if (!ok) break;
                const bool last = s + 1 == u.s1;
                const int t = s + 1 - u.s0;
                if (d0 && !last) {
                    if (!all && li >= 0)
                        for (int e = joined(t - 1); e < u.k; ++e)
                            run[(size_t)__ldg(reinterpret_cast<const unsigned char*>(order) + e) * u.n] = make_float2(0.f, 0.f);
                    all = true;
                    const int nd = min((int)(d0 & 255u), kDense);
                    for (int e = 1; e <= nd; ++e) {
                        const int c = (e < 4 ? d0 : e < 8 ? d1 : d2) >> (8 * (e & 3)) & 255;
                        const float v = lds(acc_u + 512u * c);
                        sts(acc_u + 512u * c, 0.f);
                        if (li < 0) continue;
                        float2* r = run + (size_t)c * u.n;
                        float2 h = *r;
                        ff_add(h.x, h.y, v);
                        *r = h;
                    }
                }
                // the clusters whose turn it is (all at the end) join the segment's sums
                const int nj = last ? u.k : __ldg(upto + (__ffs(t) - 1)), had = all ? u.k : nj ? joined(t - 1) : 0;
                for (int e0 = 0; e0 < nj; e0 += 4) {
                    const unsigned cs = __ldg(order + (e0 >> 2));
                    float2 h[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x)
                        h[x] = li >= 0 && e0 + x < min(nj, had) ? run[(size_t)(cs >> (8 * x) & 255u) * u.n]
                                                                 : make_float2(0.f, 0.f);
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        if (e0 + x >= nj) break;
                        const int c = cs >> (8 * x) & 255;
                        const float v = lds(acc_u + 512u * c);
                        sts(acc_u + 512u * c, 0.f);
                        ff_add(h[x].x, h[x].y, v);
                        if (li < 0) continue;
                        if (last) {
                            const float sum = h[x].x + h[x].y;
                            out[(size_t)c * u.n] = sum;
                            if (c == li) own = sum;
                        } else {
                            run[(size_t)c * u.n] = h[x];
                        }
                    }
                }
            }
            if (!ok) break;
            if constexpr (!BATCH) {
                // the sums of the rows' own clusters, row by row (lane c mod 32 adds to cluster c)
                for (int r = 0; r < 32; ++r) {
                    const int c = __shfl_sync(0xffffffffu, li, r);
                    const float v = __shfl_sync(0xffffffffu, own, r);
                    if (c >= 0 && (c & 31) == lane) ff_add(zwh[c], zwl[c], v);
                }
            }
        }
    }
    if constexpr (!BATCH) {
        __syncthreads();
        // block partial of sum_{i in L_c} S_ic, fixed warp order
        for (int c = threadIdx.x; c < a.k; c += blockDim.x) {
            double t = 0.0;
            for (int w = 0; w < 4; ++w) t += (double)zhi[w * a.kmax + c] + (double)zlo[w * a.kmax + c];
            a.zpart[(size_t)blockIdx.x * a.k + c] = t;
        }
        __threadfence();
        __syncthreads();
        __shared__ int am_last;
        if (threadIdx.x == 0) am_last = (atomicAdd(&a.st->reduce_ticket, 1u) == gridDim.x - 1);
        __syncthreads();
        if (!am_last) return;
        __threadfence();
        finalize_pass(a.zpart, (int)gridDim.x, a.k, a.counts, a.zsum, a.cnorm, a.invm, a.st, a.J_hist, a.eval_only);
    }
}

// The kernel is built for at least 4 CTAs an SM (87 to 89 registers), and for batches of few clusters,
// whose shared memory leaves room for a fifth, for 5 (72).  Left to itself the compiler takes 64 and
// spills (with joins every 64 columns a cluster: 27.7 ms for 30 passes at n = 30,011, k = 100
// where 26.5 with 4; batch of k up to 20 127.6, 129.4 with 4 and 123.4 with 5).
using TilesFn = void (*)(TilesArgs);
constexpr TilesFn kTilesOne = reduce_tiles_kernel<false, 4>, kTilesBatch = reduce_tiles_kernel<true, 4>,
                  kTilesBatchFew = reduce_tiles_kernel<true, 5>;

// Ring depth, CTAs an SM and shared memory for sums of up to k clusters: as many CTAs as fit
// (their warps hide one another's chains of shared-memory additions), then the deeper ring.
bool tiles_shape(TilesFn fn, int k, int per_sm_req, int* stages, int* per_sm, size_t* smem) {
    int best = 0;
    for (int S = kTilesMaxStages; S >= 2; --S) {
        const size_t bytes = (size_t)S * kStage + (size_t)k * 512 + (size_t)k * 32;
        int c = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c, fn, kTilesThreads, bytes);
        cudaGetLastError();
        if (per_sm_req > 0 && c > per_sm_req) c = per_sm_req;
        if (c > best) {
            best = c;
            *stages = S;
            *per_sm = c;
            *smem = bytes;
        }
    }
    return best > 0;
}

}  // namespace

cudaError_t configure_reduce_tiles(int smem_optin) {
    for (TilesFn fn : {kTilesOne, kTilesBatch, kTilesBatchFew}) {
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, fn);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     optin_minus_static(smem_optin, fa.sharedSizeBytes));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

bool plan_reduce_tiles(int n, int k, int num_sms, ReducePlan* p) {
    int S, per_sm;
    size_t smem;
    if (!tiles_shape(kTilesOne, k, 0, &S, &per_sm, &smem)) return false;
    const int T = (n + 127) / 128, grid = num_sms * per_sm;
    // Segments: whole rounds of the grid's CTAs, against the slots' traffic (8 k n bytes a segment
    // beside 2 n^2 of K, and the argmin's walk over them).
    double best = -1.0;
    for (int want = 1; want <= std::min(T, 24); ++want) {
        const int len = (T + want - 1) / want, seg = (T + len - 1) / len;
        const double rounds = (double)T * seg / grid;
        const double score = rounds / std::ceil(rounds) / (1.0 + 4.0 * seg * k / n) * T / ((double)seg * len);
        if (score > best) {
            best = score;
            p->nseg = seg;
            p->seglen = 128 * len;
        }
    }
    p->variant = kReduceTiles;
    p->k_storage = POPCORN_K_FP32;
    p->grid = grid;
    p->warps = S;   // (ring depth)
    p->smem = smem;
    p->labels_in_smem = false;
    return true;
}

size_t tiles_record_bytes(int n) { return (size_t)((n + 31) / 32) * kRecord + kPlanBytes; }

cudaError_t launch_reduce_tiles(const PassBuffers& b, const ReducePlan& plan, int* err, int eval_only, cudaStream_t s,
                                int stall_ms) {
    tile_records_kernel<<<(b.n + 127) / 128, 128, 0, s>>>(b.lab8, b.n, b.k, b.counts, b.sym_meta, b.st, eval_only);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    TilesArgs a{};
    a.K = static_cast<const float*>(b.K);
    a.n = b.n;
    a.k = b.k;
    a.T = (b.n + 127) / 128;
    a.nseg = plan.nseg;
    a.segblocks = plan.seglen / 128;
    a.lab8 = b.lab8;
    a.rec = b.sym_meta;
    a.Spart = b.Spart;
    a.Srun = b.Srun;
    a.zpart = b.zpart;
    a.zsum = b.zsum;
    a.cnorm = b.cnorm;
    a.invm = b.invm;
    a.counts = b.counts;
    a.st = b.st;
    a.J_hist = b.J_hist;
    a.eval_only = eval_only;
    a.stages = plan.warps;
    a.kmax = b.k;
    a.err = err;
    a.stall = stall_ms > 0 ? 1 : 0;
    a.wait_ns = stall_ms > 0 ? (unsigned long long)stall_ms * 1000000ull : kWaitLimitNs;
    kTilesOne<<<plan.grid, kTilesThreads, plan.smem, s>>>(a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ batched mode

bool plan_batched_tiles(BatchPlan* bp, int num_sms, int per_sm_req) {
    if (!tiles_shape(kTilesBatchFew, bp->kmax, per_sm_req, &bp->mstages, &bp->per_sm, &bp->smem)) return false;
    if (bp->per_sm < 5 && !tiles_shape(kTilesBatch, bp->kmax, per_sm_req, &bp->mstages, &bp->per_sm, &bp->smem))
        return false;
    bp->warps = 4;
    bp->grid = num_sms * bp->per_sm;
    return true;
}

cudaError_t launch_batched_tiles(const BatchInst* dI, const int2* units, const BatchPlan& bp, int* err, int eval,
                                 cudaStream_t s, int stall_ms) {
    batched_records_kernel<<<bp.vblocks, 128, 0, s>>>(dI, bp.count, eval);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    TilesArgs a{};
    a.I = dI;
    a.units = units;
    a.nunits = bp.units;
    a.eval_only = eval;
    a.stages = bp.mstages;
    a.kmax = bp.kmax;
    a.err = err;
    a.stall = stall_ms > 0 ? 1 : 0;
    a.wait_ns = stall_ms > 0 ? (unsigned long long)stall_ms * 1000000ull : kWaitLimitNs;
    const int grid = bp.units < bp.grid ? bp.units : bp.grid;
    (bp.per_sm < 5 ? kTilesBatch : kTilesBatchFew)<<<grid, kTilesThreads, bp.smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace popcorn
