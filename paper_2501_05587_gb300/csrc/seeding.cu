// K-means++ seeding (Sec. 2.1) in the feature space of the kernel, on the GPU.
//
// The paper names K-means++ as the initialization that samples each next initial centroid
// from a weighted distribution favouring points far from those already chosen; the weight of
// the cited method is the squared distance to the nearest chosen point, here in the feature
// space Kernel K-means clusters in:
//   D(i) = min over chosen c of ||phi(p_i) - phi(p_c)||^2 = min_c (K_ii - 2 K_ic + K_cc).
// K is never formed: every step evaluates kappa(p_i, p_c) for all i from the points, in FP64
// (the sampling decision compares running sums of D against a fraction of their total, so it
// is taken in FP64).  The caller supplies the k uniform draws u.  The first point is
// floor(u_0 n); point t >= 1 is the first i, in index order, at which the running sum of D
// exceeds u_t sum_i D(i) (floor(u_t n) if that sum is 0).  Each point's label is the index of
// its nearest chosen point (the lowest on ties): the initial labels for popcorn_fit.
//
// kmeanspp_kernel: one cooperative launch, one CTA of 512 threads per SM.  CTA b owns the
// points [b n / G, (b + 1) n / G) and keeps their D, labels and K_ii in shared memory.  A step:
// the CTA's sum of D and a copy of its D go to global memory -> grid barrier -> every CTA adds
// the G sums, locates the CTA whose range holds the target and, from that CTA's D, the point
// (all alike, in one order) -> the threads evaluate kappa against the new point for their rows
// and lower D.  D and the sums alternate between two buffers, so a CTA that is ahead never
// overwrites what another still reads, and one barrier a step is enough.  All orders are fixed:
// runs are bit-identical.  Every wait is bounded (grid_sync.cuh).
//
// What bounds a step is FP64 (2 multiply-adds a clock an SM on GB300), so no FP64 instruction
// runs on a lane whose result is not used: a point has as many lanes as leave the CTA's threads
// busy (one from 512 rows a CTA on), so that the inner product, kappa and the distance are not
// computed 32 times over, as they were with a warp a point (its butterfly, the exponential and
// the last three operations on every lane: about 1,400 FP64 lane operations a point at d = 64
// where 230 are needed), and the sums of D are scans, not one thread's chain of 512 additions.
// n = 50,000, d = 64, k = 32, Gaussian: 5.57 -> 1.35 ms a call.
#include <cmath>

#include "grid_sync.cuh"
#include "popcorn_internal.cuh"
#include "tc_common.cuh"

namespace popcorn {
namespace {

constexpr int kSeedThreads = 512;
constexpr int kSeedWarps = kSeedThreads / 32;

struct SeedArgs {
    const float* P;
    int64_t ldp;
    int n, d, k;
    int kind, degree;
    double gamma, coef0, neg_gamma_over_sigma2;   // kappa in FP64
    const double* u;           // k draws in [0, 1)
    int32_t* labels;           // n
    int32_t* centers;          // k
    double* part;              // [2][G] the CTAs' sums of D, by step parity
    double* Dg;                // [2][n] D, by step parity
    unsigned* bar;             // grid barrier words
    int* err;
    int rows_max;              // ceil(n / G)
};

// Dynamic shared memory: the center's coordinates [d], then per owned row D, K_ii (doubles)
// and the label (int), then the threads' running sums [kSeedThreads] and the CTAs' sums [G]
// (doubles).
struct SeedLayout {
    size_t cs, D, kii, lab, inc, part, bytes;
};
__host__ __device__ inline SeedLayout seed_layout(int d, int rows_max, int G) {
    SeedLayout L;
    L.cs = 0;
    L.D = L.cs + (size_t)d * 8;
    L.kii = L.D + (size_t)rows_max * 8;
    L.inc = L.kii + (size_t)rows_max * 8;
    L.part = L.inc + 2 * (size_t)kSeedThreads * 8;   // (half of it spare: the largest n stays where it was)
    L.lab = L.part + (size_t)G * 8;
    L.bytes = L.lab + (size_t)rows_max * 4;
    return L;
}

// kappa from the inner product (linear, polynomial) or the squared distance (Gaussian), FP64;
// the polynomial power by repeated multiplication
__device__ __forceinline__ double kappa_of(const SeedArgs& a, double s) {
    if (a.kind == POPCORN_GAUSSIAN) return exp(a.neg_gamma_over_sigma2 * s);
    if (a.kind == POPCORN_POLYNOMIAL) {
        const double base = fma(a.gamma, s, a.coef0);
        double v = base;
        for (int e = 1; e < a.degree; ++e) v *= base;
        return v;
    }
    return s;
}

// The FP64 inner product (or squared distance, Gaussian) of a point with the center in shared
// memory, by a group of `lanes` (a power of two) neighbouring lanes: lane s takes coordinates s,
// s + lanes, ... in order, then a butterfly.
__device__ __forceinline__ double group_pair(const SeedArgs& a, const float* __restrict__ p, const double* __restrict__ cs,
                                             int s, int lanes) {
    double t = 0.0;
    if (a.kind == POPCORN_GAUSSIAN) {
#pragma unroll 4
        for (int l = s; l < a.d; l += lanes) {
            const double x = (double)__ldg(p + l) - cs[l];
            t = fma(x, x, t);
        }
    } else {
#pragma unroll 4
        for (int l = s; l < a.d; l += lanes) t = fma((double)__ldg(p + l), cs[l], t);
    }
    for (int o = lanes >> 1; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

// Inclusive running sums over the warp's lanes.
__device__ __forceinline__ double warp_scan(double v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Running sums over the CTA: inc[t] = sum of s over threads 0 .. t (a fixed order); the total.
__device__ double block_scan(double s, double* inc, double* wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double v = warp_scan(s, lane);
    if (lane == 31) wsum[warp] = v;
    __syncthreads();
    double before = 0.0;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    inc[threadIdx.x] = warp ? before + v : v;
    __syncthreads();
    return inc[kSeedThreads - 1];
}

__global__ void __launch_bounds__(kSeedThreads, 1) kmeanspp_kernel(SeedArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int G = gridDim.x, n = a.n, k = a.k;
    const SeedLayout L = seed_layout(a.d, a.rows_max, G);
    double* cs = reinterpret_cast<double*>(smem + L.cs);
    double* D = reinterpret_cast<double*>(smem + L.D);
    double* kii = reinterpret_cast<double*>(smem + L.kii);
    double* inc = reinterpret_cast<double*>(smem + L.inc);
    double* part_s = reinterpret_cast<double*>(smem + L.part);
    int* lab = reinterpret_cast<int*>(smem + L.lab);
    __shared__ double kcc_s, tgt_s, wsum[kSeedWarps];
    __shared__ int bstar_s, pick_s, pos_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto first_row = [&](int b) { return (int)((int64_t)b * n / G); };
    const int lo = first_row(blockIdx.x), hi = first_row(blockIdx.x + 1), rows = hi - lo;
    // lanes a point: as many (a power of two, up to a warp) as the CTA's threads give each row
    int lanes = 32;
    while (lanes > 1 && lanes * a.rows_max > kSeedThreads) lanes >>= 1;
    const int sub = threadIdx.x & (lanes - 1), slot = threadIdx.x / lanes, slots = kSeedThreads / lanes;

    // K_ii of the owned points (the Gaussian's is 1)
    for (int r0 = 0; r0 < rows; r0 += slots) {
        const int r = r0 + slot;
        double v = 1.0;
        if (a.kind != POPCORN_GAUSSIAN) {
            const float* p = a.P + (int64_t)(lo + min(r, rows - 1)) * a.ldp;
            double s = 0.0;
            for (int l = sub; l < a.d; l += lanes) {
                const double x = (double)__ldg(p + l);
                s = fma(x, x, s);
            }
            for (int o = lanes >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (sub == 0) v = kappa_of(a, s);
        }
        if (sub == 0 && r < rows) kii[r] = v;
    }

    // point c joins the chosen set as number t: D and the labels of the owned points, and (for
    // the next step's choice) D to the buffer of that step
    auto add_center = [&](int t, int c) {
        const float* pc = a.P + (int64_t)c * a.ldp;
        for (int l = threadIdx.x; l < a.d; l += blockDim.x) cs[l] = (double)__ldg(pc + l);
        __syncthreads();
        if (warp == 0) {
            double s = 0.0;
            if (a.kind != POPCORN_GAUSSIAN) {
                for (int l = lane; l < a.d; l += 32) s = fma(cs[l], cs[l], s);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            }
            if (lane == 0) kcc_s = a.kind == POPCORN_GAUSSIAN ? 1.0 : kappa_of(a, s);
        }
        __syncthreads();
        const double kcc = kcc_s;
        double* Dn = a.Dg + (size_t)((t + 1) & 1) * n + lo;
        for (int r0 = 0; r0 < rows; r0 += slots) {   // (uniform trips: the groups shuffle)
            const int r = r0 + slot;
            const double s = group_pair(a, a.P + (int64_t)(lo + min(r, rows - 1)) * a.ldp, cs, sub, lanes);
            if (sub == 0 && r < rows) {
                const double dc = fmax(kii[r] - 2.0 * kappa_of(a, s) + kcc, 0.0);
                if (t == 0 || dc < D[r]) {
                    D[r] = dc;
                    lab[r] = t;
                }
                Dn[r] = D[r];
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) a.centers[t] = c;
        __syncthreads();
    };

    __syncthreads();
    add_center(0, min((int)floor(a.u[0] * n), n - 1));
    for (int t = 1; t < k; ++t) {
        double* part = a.part + (size_t)(t & 1) * G;
        // the CTA's sum of D: each thread's contiguous rows in order, then the threads
        {
            const int ch = (rows + kSeedThreads - 1) / kSeedThreads;
            const int r0 = min(rows, ch * (int)threadIdx.x), r1 = min(rows, r0 + ch);
            double s = 0.0;
            for (int r = r0; r < r1; ++r) s += D[r];
            const double total = block_scan(s, inc, wsum);
            if (threadIdx.x == 0) part[blockIdx.x] = total;
        }
        if (!gsync::grid_barrier(a.bar, a.err)) return;
        for (int b = threadIdx.x; b < G; b += blockDim.x) part_s[b] = __ldcg(part + b);
        if (threadIdx.x == 0) {
            pick_s = kSeedThreads;
            pos_s = -1;
        }
        __syncthreads();
        // every CTA alike: the running sums of the CTAs in order, the target, and the first CTA
        // whose running sum exceeds it.  (Neighbouring running sums come from scans of different
        // shape, so one may exceed another by a rounding with nothing added between them: here and below
        // only what has a positive weight is taken.)
        if (warp == 0) {
            const int per = (G + 31) / 32, b0 = min(G, lane * per), b1 = min(G, b0 + per);
            double s = 0.0;
            int lastpos = -1;
            for (int b = b0; b < b1; ++b) {
                s += part_s[b];
                if (part_s[b] > 0.0) lastpos = b;
            }
            const double upto = warp_scan(s, lane);
            double before = __shfl_up_sync(0xffffffffu, upto, 1);
            if (lane == 0) before = 0.0;
            const double W = __shfl_sync(0xffffffffu, upto, 31), target = a.u[t] * W;
            int b = -1;
            double run = before;
            for (int x = b0; x < b1 && b < 0; ++x) {
                const double next = run + part_s[x];
                if (next > target && part_s[x] > 0.0) b = x;
                else run = next;
            }
            const unsigned have = __ballot_sync(0xffffffffu, b >= 0);
            lastpos = __reduce_max_sync(0xffffffffu, lastpos);
            const int owner = have ? __ffs(have) - 1 : (lastpos >= 0 ? lastpos / per : 0);
            if (!have && lane == owner) {   // u_t W rounded up to W: the last CTA with a positive sum
                b = lastpos;
                run = before;
                for (int x = b0; x < lastpos; ++x) run += part_s[x];
            }
            if (lane == owner) {
                bstar_s = W > 0.0 ? b : -1;
                tgt_s = target - run;   // the target inside CTA bstar's range
            }
        }
        __syncthreads();
        const int bstar = bstar_s;
        int c;
        if (bstar < 0) {
            c = min((int)floor(a.u[t] * n), n - 1);
        } else {
            // the first of its rows whose running sum exceeds the target; its last row with a
            // positive D if rounding leaves the target past the end
            const double tgt = tgt_s;
            const int blo = first_row(bstar), brows = first_row(bstar + 1) - blo;
            const double* Db = a.Dg + (size_t)(t & 1) * n + blo;
            const int ch = (brows + kSeedThreads - 1) / kSeedThreads;
            const int r0 = min(brows, ch * (int)threadIdx.x), r1 = min(brows, r0 + ch);
            double s = 0.0;
            int lastpos = -1;
            for (int r = r0; r < r1; ++r) {
                const double x = __ldcg(Db + r);
                if (x > 0.0) lastpos = r;
                s += x;
            }
            block_scan(s, inc, wsum);
            if (s > 0.0 && inc[threadIdx.x] > tgt) atomicMin(&pick_s, (int)threadIdx.x);
            if (lastpos >= 0) atomicMax(&pos_s, lastpos);
            __syncthreads();
            const int pick = pick_s;
            __syncthreads();
            if ((int)threadIdx.x == pick) {
                double run = pick ? inc[pick - 1] : 0.0;
                int found = -1;
                for (int r = r0; r < r1; ++r) {
                    const double x = __ldcg(Db + r);
                    run += x;
                    if (run > tgt && x > 0.0) {
                        found = r;
                        break;
                    }
                }
                if (found < 0) found = lastpos;   // rounding at the chunk's end
                pos_s = found;
            }
            __syncthreads();
            c = blo + max(0, pos_s);
        }
        add_center(t, c);
    }
    for (int i = lo + threadIdx.x; i < hi; i += blockDim.x) a.labels[i] = lab[i - lo];
}

}  // namespace

size_t kmeanspp_smem(int n, int d, int num_sms) {
    return seed_layout(d, (n + num_sms - 1) / num_sms, num_sms).bytes;
}

int kmeanspp_dynamic_limit(int smem_optin) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kmeanspp_kernel) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return optin_minus_static(smem_optin, fa.sharedSizeBytes);
}

cudaError_t configure_kmeanspp(int smem_optin) {
    return cudaFuncSetAttribute(kmeanspp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kmeanspp_dynamic_limit(smem_optin));
}

bool kmeanspp_fits(int n, int d, int num_sms, int smem_optin) {
    return kmeanspp_smem(n, d, num_sms) <= (size_t)kmeanspp_dynamic_limit(smem_optin);
}

cudaError_t launch_kmeanspp(const float* P, int n, int d, int64_t ldp, int k, const popcorn_kernel& kern,
                            const double* u, int32_t* labels, int32_t* centers, double* part, double* Dg,
                            unsigned* bar, int* err, int num_sms, cudaStream_t s) {
    SeedArgs a;
    a.P = P;
    a.ldp = ldp;
    a.n = n;
    a.d = d;
    a.k = k;
    a.kind = kern.kind;
    a.degree = kern.degree;
    a.gamma = kern.gamma;
    a.coef0 = kern.coef0;
    a.neg_gamma_over_sigma2 = kern.kind == POPCORN_GAUSSIAN ? -kern.gamma / (kern.sigma * kern.sigma) : 0.0;
    a.u = u;
    a.labels = labels;
    a.centers = centers;
    a.part = part;
    a.Dg = Dg;
    a.bar = bar;
    a.err = err;
    a.rows_max = (n + num_sms - 1) / num_sms;
    cudaError_t e = cudaMemsetAsync(bar, 0, 32 * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)num_sms);
    cfg.blockDim = dim3(kSeedThreads);
    cfg.dynamicSmemBytes = kmeanspp_smem(n, d, num_sms);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kmeanspp_kernel, a);
}

}  // namespace popcorn
