// C ABI of the TSENOR hot path (see include/tsenor.h): argument checks on the
// host, then kernel launches on the caller's stream.  No allocation, no
// synchronisation, no CPU fallback.
#include "tsenor.h"
#include "tsenor_device.cuh"

#include <atomic>
#include <cmath>

namespace {

thread_local int g_last_cuda_error = 0;
std::atomic<long long> g_launches{0};

inline bool valid_M(int M) { return M == 4 || M == 8 || M == 16 || M == 32; }

int check_matrix(int64_t rows, int64_t cols, int64_t ld, int M) {
    if (rows < 0 || cols < 0 || ld < cols) return TSENOR_ERR_SHAPE;
    if (rows % M || cols % M) return TSENOR_ERR_SHAPE;
    return TSENOR_OK;
}

int finish_launch() {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_last_cuda_error = (int)e;
        return TSENOR_ERR_CUDA;
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return TSENOR_OK;
}

inline bool aligned16(const void* p, int64_t ld) {
    return (reinterpret_cast<uintptr_t>(p) % 16 == 0) && (ld % 4 == 0);
}

tsenor::ScoreSrc abs_source(const float* scores, int64_t ld) {
    tsenor::ScoreSrc S{};
    S.kind = tsenor::SC_ABS;
    S.w = scores; S.ld = ld;
    S.vec_w = aligned16(scores, ld);
    return S;
}

// Validates a caller's descriptor and turns it into the device-side form.
int make_source(const tsenor_scores_t* d, int64_t cols, tsenor::ScoreSrc* out) {
    if (!d) return TSENOR_ERR_NULL;
    if (d->kind < TSENOR_SCORES_ABS || d->kind > TSENOR_SCORES_COLMUL) return TSENOR_ERR_ARG;
    if (d->ld < cols) return TSENOR_ERR_SHAPE;
    if (!d->w) return TSENOR_ERR_NULL;
    tsenor::ScoreSrc S{};
    S.kind = d->kind;
    S.w_is_bf16 = d->w_is_bf16 ? 1 : 0;
    S.w = d->w; S.ld = d->ld;
    S.vec_w = d->w_is_bf16 ? ((reinterpret_cast<uintptr_t>(d->w) % 8 == 0) && (d->ld % 4 == 0))
                           : aligned16(d->w, d->ld);
    if (d->kind == TSENOR_SCORES_ADMM) {
        if (!d->v) return TSENOR_ERR_NULL;
        if (d->ld_v < cols) return TSENOR_ERR_SHAPE;
        if (!std::isfinite(d->scalar)) return TSENOR_ERR_ARG;
        S.v = d->v; S.ld_v = d->ld_v; S.scalar = d->scalar;
        S.vec_v = aligned16(d->v, d->ld_v);
    }
    if (d->kind == TSENOR_SCORES_COLDIV || d->kind == TSENOR_SCORES_COLMUL) {
        if (!d->colvec) return TSENOR_ERR_NULL;
        S.colvec = d->colvec;
        S.vec_c = (reinterpret_cast<uintptr_t>(d->colvec) % 16 == 0);
    }
    *out = S;
    return TSENOR_OK;
}

std::atomic<int> g_layout{TSENOR_LAYOUT_AUTO};

// Units (= warps) a matrix is cut into under layout V, and the slots of a block row: whole mask
// words, except that a single block column needs no padding.
template <int M, int V>
int64_t unit_count(const tsenor::Params& P, int64_t* nbp_out) {
    using G = tsenor::Geom<M, V>;
    const int64_t nbc = P.cols / M, nbp = (nbc == 1) ? 1 : (nbc + G::GPW - 1) / G::GPW * G::GPW;
    *nbp_out = nbp;
    return ((P.rows / M) * nbp + G::BPW - 1) / G::BPW;
}

int sm_count() {
    static thread_local int cached_dev = -1, cached = 148;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != cached_dev) {
        int n = 0;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0) cached = n;
        cached_dev = dev;
    }
    return cached;
}

template <int M, int MODE, int V, bool EE>
int launch_layout(const tsenor::Params& P, cudaStream_t st) {
    using G = tsenor::Geom<M, V>;
    tsenor::Params Q = P;
    const int64_t units = unit_count<M, V>(P, &Q.nbp);
    if (units == 0) return TSENOR_OK;
    if (units > 0x7fffffffLL) return TSENOR_ERR_SHAPE;
    constexpr int WPC = tsenor::CtaWarps<M, V, EE>::value;
    const size_t smem = WPC * sizeof(tsenor::SmemLayout<G, MODE, EE>);
    static thread_local int configured_device = -1;
    int dev = 0;
    cudaGetDevice(&dev);
    if (configured_device != dev) {
        cudaError_t e = cudaFuncSetAttribute(tsenor::tsenor_kernel<M, MODE, V, EE>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) {
            g_last_cuda_error = (int)e;
            return TSENOR_ERR_CUDA;
        }
        configured_device = dev;
    }
    tsenor::tsenor_kernel<M, MODE, V, EE><<<(unsigned)((units + WPC - 1) / WPC), 32 * WPC, smem, st>>>(Q);
    return finish_launch();
}

// Chooses the register layout by w, the warps per SM that units of one mask word make, and by the number
// of iterations T: the wider units of the throughput layout round several passes in series, which counts
// the more the fewer iterations there are.  One rule for the whole method and for Algorithm 1 alone, so
// that the mask is the rounding of the very plan that tsenor_dykstra returns.  Both sides of each line, in us
// (square matrices, Gaussian; [Algorithm 1 alone]):
//   M = 4   one lane a block needs no exchange at all, so only a small matrix, or few iterations, favour
//           the latency layout: w <= 6 + 600 / T, at most 16.  Latency / throughput at T = 300: w 7.8 28.7 / 30.5
//           [27.9 / 27.8], 10.6 32.5 / 30.4; T = 100: 10.6 13.8 / 16.7, 13.8 16.2 / 16.5 [14.6 / 12.0]; T = 50: 13.8 10.5 /
//           13.2 [8.7 / 7.6]; T = 20: 13.8 7.1 / 11.0 [5.1 / 5.1], 21.6 [6.4 / 6.1]; T = 0: 13.8 4.5 / 8.8.
//   M = 8   latency up to three warps per scheduler; beyond, spread while w <= 32 and w T <= 3200, or w <= 28 and
//           w T <= 6400.  Spread / throughput, Gaussian (Student-t in brackets): T = 300: 13.1 51.2 / 53.5 [34.8 / 47.6], 18.3 58.1 /
//           75.1 [46.5 / 66.0], 21.2 67.5 / 75.4 [49.3 / 55.6], 24.3 78.6 / 75.2 [51.3 / 62.4]; T = 200: 27.7 55.6 / 56.3, 31.2 63.4 / 56.6;
//           T = 100: 31.2 37.5 / 38.3, 43 50.2 / 50.2; T = 20: 27.7 15.4 / 23.2, 62 28.8 / 33.0 [Algorithm 1 alone 17.7 / 16.6].
//   M = 16  latency while a scheduler has one warp (T = 300: w 3.5 44.6, spread 53; 4.4 63.2, spread 57.5); beyond,
//           spread while T <= 50, w T <= 1800 or w <= 16.  Spread / throughput at T = 300: 15.6 80.9 [Student-t 42.3] / 92,
//           17.5 - / 108.7 [51.4]; T = 100: 22 50.7 / 53.1 [Algorithm 1 alone 41.9 / 41.3]; T = 50: 221 250 / 292 [180 / 180];
//           T = 20: 221 191 / 227 [94 / 104].
//   M = 32  the same layout in both builds: the one for latency while all its warps are resident (6.9 86.1 /
//           93.0; 15.6 142.9 / 145.1).
// The stopping test does not say beforehand how many iterations it will run: spread up to w = 16 (768 x 768
// 4:8, Student / Gaussian: 26.8 / 53.1, latency 24.9 / 66.0, throughput 37.8 / 53.3; 1024 x 1024 8:16: 35.7 / 84.6,
// 42.9 / 123, 43.8 / 85.4).
template <int M> int64_t latency_warps_per_sm(int T) {
    if (M == 4) return T <= 60 ? 16 : 6 + 600 / T;
    return M == 8 ? 12 : M == 16 ? 4 : 16;
}
template <int M, bool EE> bool spread_is_best(int64_t warps, int64_t sms, int T) {
    const auto up_to = [&](int64_t w) { return warps <= w * sms; };
    const int64_t wT = warps * T;
    if (EE && up_to(16)) return true;
    if (M == 8) return (up_to(32) && wT <= 3200 * sms) || (up_to(28) && wT <= 6400 * sms);
    return T <= 50 || wT <= 1800 * sms || up_to(16);
}
// Rounding alone has no iterations to share lanes for, and units of one mask word are one rounding pass: more
// warps and nothing serial (log-plans, us against the wider units: 1024 x 1024 M = 8 7.0 / 10.1, M = 16 9.3 / 12.1;
// 4096 x 4096 74.5 / 72.6 and 76.7 / 81.3).  At M = 4 a pass is so short that the wider units win once the GPU is
// full (w 55 7.6 / 8.5, 87 10.2 / 10.7, 125 13.7 / 13.0, 221 22.3 / 20.3).
constexpr int64_t ROUNDING_WARPS_PER_SM_M4 = 64;

template <int M, int MODE, bool EE>
int launch(const tsenor::Params& P, cudaStream_t st) {
    int64_t nbp = 0;
    const int64_t warps = unit_count<M, 1>(P, &nbp), sms = sm_count();
    if constexpr (MODE == 2) {
        if constexpr (M == 4)
            if (warps > ROUNDING_WARPS_PER_SM_M4 * sms) return launch_layout<M, MODE, 0, EE>(P, st);
        return launch_layout<M, MODE, (M < 32) ? 1 : 0, EE>(P, st);
    } else {
        const int policy = g_layout.load(std::memory_order_relaxed);
        if (policy == TSENOR_LAYOUT_LATENCY ||
            (policy == TSENOR_LAYOUT_AUTO && warps <= latency_warps_per_sm<M>(P.iters) * sms))
            return launch_layout<M, MODE, 1, EE>(P, st);
        if constexpr (M == 8 || M == 16)
            if (policy == TSENOR_LAYOUT_AUTO && spread_is_best<M, EE>(warps, sms, P.iters))
                return launch_layout<M, MODE, 3, EE>(P, st);
        return launch_layout<M, MODE, 0, EE>(P, st);
    }
}

template <int MODE, bool EE>
int dispatch_size(const tsenor::Params& P, int M, cudaStream_t st) {
    switch (M) {
        case 4: return launch<4, MODE, EE>(P, st);
        case 8: return launch<8, MODE, EE>(P, st);
        case 16: return launch<16, MODE, EE>(P, st);
        default: return launch<32, MODE, EE>(P, st);
    }
}

// The stopping-test mode has kernels of its own: the test's code stays out of the others.
template <int MODE>
int dispatch(const tsenor::Params& P, int M, cudaStream_t st) {
    if constexpr (MODE != 2)
        if (P.ee_eps > 0.0f && P.iters > 0) return dispatch_size<MODE, true>(P, M, st);
    return dispatch_size<MODE, false>(P, M, st);
}

void set_N(tsenor::Params& P, int N) {
    P.N = N; P.Nf = (float)N; P.log2N = (float)std::log2((double)N);
    P.inv_N.hi = 1.0f / P.Nf;
    P.inv_N.lo = (float)(1.0 / (double)N - (double)P.inv_N.hi);
}

void set_tau(tsenor::Params& P, float tau) {
    const double c = (double)tau * 1.4426950408889634074;  // tau * log2(e)
    P.c_hi = (float)c;
    P.c_lo = (float)(c - (double)P.c_hi);
}

// ------------------------------------------------------------ small kernels

__global__ void fill_mask_kernel(uint32_t* bits, int64_t rows, int64_t wpr, int64_t cols, uint32_t value) {
    const int64_t n = rows * wpr;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < n;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t wd = idx % wpr;
        uint32_t v = value;
        const int64_t left = cols - wd * 32;
        if (left < 32) v &= (left <= 0) ? 0u : ((1u << left) - 1u);
        bits[idx] = v;
    }
}

// Walk over the quads (4 columns) of a matrix: quad idx is (row(idx), 4 * (idx - row(idx) * qpr)).
// Rows by a 32-bit multiplication with magic = ceil(2^(31+L) / qpr), L = ceil(log2 qpr), exact while the
// quads number less than 2^31: the quotient is then too large by less than idx / 2^31 / qpr < 1 / qpr.
struct QuadWalk {
    int64_t qpr, nq;
    unsigned magic, shift;        // magic 0: divide
    __device__ __forceinline__ int64_t row(int64_t idx) const {
        return magic ? (int64_t)(__umulhi((unsigned)idx, magic) >> shift) : idx / qpr;
    }
};
QuadWalk quad_walk(int64_t rows, int64_t cols) {
    QuadWalk q{};
    q.qpr = cols / 4;
    q.nq = rows * q.qpr;
    if (q.qpr > 1 && q.nq < (1LL << 31)) {
        int L = 1;
        while ((1LL << L) < q.qpr) ++L;
        q.magic = (unsigned)(((1ULL << (31 + L)) + q.qpr - 1) / q.qpr);
        q.shift = L - 1;
    }
    return q;
}

// Aligned fp32 |W|, the common source of the scans: where a thread has four of its quads or more they are
// read at once, in a kernel of its own (PLAIN).  Everything else reads a quad at a time through
// load_score_quad, whose branches keep a loop's reads from being batched: in one kernel with the batched
// loop it lost 10 to 45 % (maximum of (W + V / rho)^2 at 14336 x 4096: 110 us together, 80 apart), and a
// matrix that is too small to be batched up to a third (14336 x 32: 5.8 and 4.9 us).
constexpr int SCAN_U = 4;
bool batched_scan(const tsenor::ScoreSrc& S, int64_t quads, int64_t threads) {
    return S.kind == tsenor::SC_ABS && S.vec_w && !S.w_is_bf16 && quads > (SCAN_U - 1) * threads;
}
__device__ __forceinline__ float4 load_plain_quad(const tsenor::ScoreSrc& S, int64_t r, int64_t c) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(S.w) + r * S.ld + c));
    return make_float4(fabsf(v.x), fabsf(v.y), fabsf(v.z), fabsf(v.w));
}
template <bool PLAIN>
__device__ __forceinline__ float4 load_quad(const tsenor::ScoreSrc& S, int64_t r, int64_t c) {
    return PLAIN ? load_plain_quad(S, r, c) : tsenor::load_score_quad(S, r, c);
}

// Retained score of one mask or two (TWO) under one score source (quads of 4 columns).
template <bool PLAIN, bool TWO>
__global__ void objective_kernel(const tsenor::ScoreSrc S, const uint32_t* __restrict__ bits_a,
                                 const uint32_t* __restrict__ bits_b, const QuadWalk q, int64_t wpr, double* out) {
    static_assert(!(PLAIN && TWO), "two masks are scanned a quad at a time");
    double acc_a = 0.0, acc_b = 0.0;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if constexpr (PLAIN) {   // 14336 x 4096: 88 us a quad at a time, 51 this way; 2048 x 2048: 10.2, 8.2
        for (; idx + (SCAN_U - 1) * step < q.nq; idx += SCAN_U * step) {
            float4 v[SCAN_U];
            uint32_t m[SCAN_U];
#pragma unroll
            for (int u = 0; u < SCAN_U; ++u) {
                const int64_t r = q.row(idx + u * step), c = (idx + u * step - r * q.qpr) * 4;
                m[u] = bits_a[r * wpr + c / 32] >> (c % 32);
                v[u] = load_plain_quad(S, r, c);
            }
#pragma unroll
            for (int u = 0; u < SCAN_U; ++u) {
                const float e[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if ((m[u] >> k) & 1u) acc_a += (double)e[k];
            }
        }
    }
    for (; idx < q.nq; idx += step) {
        const int64_t r = idx / q.qpr, c = (idx % q.qpr) * 4;
        const uint32_t ma = (bits_a[r * wpr + c / 32] >> (c % 32)) & 15u;
        const uint32_t mb = TWO ? (bits_b[r * wpr + c / 32] >> (c % 32)) & 15u : 0u;
        if ((ma | mb) == 0u) continue;
        const float4 v = load_quad<PLAIN>(S, r, c);
        const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if ((ma >> k) & 1u) acc_a += (double)e[k];
            if (TWO && ((mb >> k) & 1u)) acc_b += (double)e[k];
        }
    }
    for (int off = 16; off > 0; off >>= 1) {
        acc_a += __shfl_xor_sync(0xffffffffu, acc_a, off);
        if (TWO) acc_b += __shfl_xor_sync(0xffffffffu, acc_b, off);
    }
    __shared__ double part[2][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { part[0][warp] = acc_a; part[1][warp] = acc_b; }
    __syncthreads();
    if (warp == 0) {
        acc_a = (lane < (int)(blockDim.x >> 5)) ? part[0][lane] : 0.0;
        acc_b = (lane < (int)(blockDim.x >> 5)) ? part[1][lane] : 0.0;
        for (int off = 16; off > 0; off >>= 1) {
            acc_a += __shfl_xor_sync(0xffffffffu, acc_a, off);
            if (TWO) acc_b += __shfl_xor_sync(0xffffffffu, acc_b, off);
        }
        if (lane == 0) {
            atomicAdd(out, acc_a);
            if (TWO) atomicAdd(out + 1, acc_b);
        }
    }
}

// mask_inout <- prev wherever the previous mask retained more score (obj2 = {new, prev}).
__global__ void keep_better_kernel(const double* __restrict__ obj2, const uint32_t* __restrict__ prev,
                                   uint32_t* __restrict__ mask_inout, int64_t nwords) {
    if (!(obj2[0] < obj2[1])) return;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < nwords;
         idx += (int64_t)gridDim.x * blockDim.x)
        mask_inout[idx] = prev[idx];
}

// One atomic per CTA: with one per warp, 19,000 of them queued on a single word were two thirds of the
// time (2048 x 2048: 16.4 us, 8.4 now; 14336 x 4096: 51.7, 37.4 now, at the copy bandwidth).
template <bool PLAIN>
__global__ void scores_max_kernel(const tsenor::ScoreSrc S, const QuadWalk q, unsigned int* out_bits) {
    float m = 0.f;
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if constexpr (PLAIN) {
        for (; idx + (SCAN_U - 1) * step < q.nq; idx += SCAN_U * step) {
            float4 v[SCAN_U];
#pragma unroll
            for (int u = 0; u < SCAN_U; ++u) {
                const int64_t r = q.row(idx + u * step);
                v[u] = load_plain_quad(S, r, (idx + u * step - r * q.qpr) * 4);
            }
#pragma unroll
            for (int u = 0; u < SCAN_U; ++u)     // fmaxf drops NaN
                m = fmaxf(fmaxf(m, fmaxf(v[u].x, v[u].y)), fmaxf(v[u].z, v[u].w));
        }
    }
    for (; idx < q.nq; idx += step) {
        const float4 v = load_quad<PLAIN>(S, idx / q.qpr, (idx % q.qpr) * 4);
        m = fmaxf(fmaxf(m, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
    }
    // non-negative floats order like their bit patterns
    const unsigned warp_max = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    __shared__ unsigned part[32];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = warp_max;
    __syncthreads();
    if (threadIdx.x < 32) {
        const unsigned p = (threadIdx.x < (blockDim.x >> 5)) ? part[threadIdx.x] : 0u;
        const unsigned cta_max = __reduce_max_sync(0xffffffffu, p);
        if (threadIdx.x == 0) atomicMax(out_bits, cta_max);
    }
}

// (By plain divisions: with QuadWalk::row, whose 64-bit alternative stays in the loop, 2 to 7 % slower.)
__global__ void materialize_kernel(const tsenor::ScoreSrc S, int64_t rows, int64_t cols, float* out,
                                   int64_t ld_out) {
    const int64_t qpr = cols / 4, nq = rows * qpr;
    for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < nq;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = idx / qpr, c = (idx % qpr) * 4;
        const float4 v = tsenor::load_score_quad(S, r, c);
        float* p = out + r * ld_out + c;
        p[0] = v.x; p[1] = v.y; p[2] = v.z; p[3] = v.w;
    }
}

// One thread per block of the mask; bound by the wait for its M words, which are all read before the first is
// used (one after the other, 4096 x 4096: 12.3 / 8.3 / 6.2 / 6.2 us for M = 4 / 8 / 16 / 32; this way 10.3 / 6.9 / 5.9 / 5.8; 256 x 256:
// 4.2 / 4.8 / 6.0 / 6.2, now 4.2 at every M).
template <int M>
__global__ void check_kernel(const uint32_t* __restrict__ bits, int64_t rows, int64_t cols, int64_t wpr, int N,
                             unsigned long long* bad_out) {
    constexpr uint32_t GM = (M == 32) ? 0xffffffffu : ((1u << (M & 31)) - 1u);
    const int64_t nbc = cols / M, nblk = (rows / M) * nbc;
    unsigned long long bad = 0;
    for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nblk;
         b += (int64_t)gridDim.x * blockDim.x) {
        const int64_t br = tsenor::div_slots(b, nbc), c0 = (b - br * nbc) * M;
        const uint32_t* const p = bits + br * M * wpr + c0 / 32;
        uint32_t row[M];
#pragma unroll
        for (int i = 0; i < M; ++i) row[i] = __ldg(p + i * wpr);
        bool ok = true;
        uint32_t colcnt[5] = {0, 0, 0, 0, 0};  // bit-sliced column counters (counts up to 31)
        uint32_t over = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            uint32_t carry = (row[i] >> (c0 % 32)) & GM;
            ok = ok && (__popc(carry) == N);
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const uint32_t t = colcnt[k] & carry;
                colcnt[k] ^= carry;
                carry = t;
            }
            over |= carry;  // a column reached 32
        }
        uint32_t eq = GM;
#pragma unroll
        for (int k = 0; k < 5; ++k) eq &= ((N >> k) & 1) ? colcnt[k] : ~colcnt[k];
        if (N == 32) ok = ok && (over == GM); else ok = ok && (over == 0) && (eq == GM);
        bad += ok ? 0 : 1;
    }
    for (int off = 16; off > 0; off >>= 1) bad += __shfl_xor_sync(0xffffffffu, bad, off);
    if ((threadIdx.x & 31) == 0 && bad) atomicAdd(bad_out, bad);
}

int grid_for(int64_t work, int threads) {
    int64_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > 148 * 16) g = 148 * 16;
    return (int)g;
}

// CTAs of 256 threads for the maximum over quads: two waves of full SMs, since every CTA ends in an atomic.
int scan_grid(int64_t quads) {
    const int64_t g = (quads + 255) / 256, wave = 16LL * sm_count();
    return (int)(g < 1 ? 1 : g < wave ? g : wave);
}

// Threads of a CTA for the objectives.  One mask: 256.  Two masks: 512 from some 32,768 quads on, since the
// atomics of the CTAs, two each, queue on one line (safeguard of a 1024 x 1024 matrix 10.3 us with 256, 9.0
// with 512; 256 x 264: 6.2 and 7.0).  One mask with 512: 12.2 us at 2048 x 2048 against 8.2.
int objective_threads(bool two, int64_t quads) { return two && quads > 32768 ? 512 : 256; }
// CTAs for them: one full wave for one mask, two for two (the fp64 sums make the CTAs uneven).
int objective_grid(bool two, int64_t quads) {
    const int t = objective_threads(two, quads);
    const int64_t g = (quads + t - 1) / t, waves = (two ? 4096 : 2048) / t * (int64_t)sm_count();
    return (int)(g < 1 ? 1 : g < waves ? g : waves);
}

// Simple rounding, on the units of the rounding stage that are one mask word wide.
template <int M>
int launch_simple_round(const float* key, int64_t ld, int64_t rows, int64_t cols, int N, uint32_t* bits,
                        cudaStream_t st) {
    tsenor::Params P{};
    P.rows = rows; P.cols = cols;
    int64_t nbp = 0;
    const int64_t units = unit_count<M, (M < 32) ? 1 : 0>(P, &nbp);
    const int64_t ctas = (units + tsenor::SIMPLE_WARPS - 1) / tsenor::SIMPLE_WARPS;
    if (ctas > 0x7fffffffLL) return TSENOR_ERR_SHAPE;
    tsenor::simple_round_kernel<M><<<(unsigned)ctas, 32 * tsenor::SIMPLE_WARPS, 0, st>>>(
        key, ld, rows, cols, (cols + 31) / 32, nbp, units, aligned16(key, ld), N, bits);
    return finish_launch();
}

int trivial_mask(uint32_t* bits, int64_t rows, int64_t cols, bool ones, cudaStream_t st) {
    const int64_t wpr = (cols + 31) / 32;
    if (rows * wpr == 0) return TSENOR_OK;
    fill_mask_kernel<<<grid_for(rows * wpr, 256), 256, 0, st>>>(bits, rows, wpr, cols, ones ? 0xffffffffu : 0u);
    return finish_launch();
}

}  // namespace

extern "C" {

struct Extras {   // optional settings carried by tsenor_scores_t
    int per_block_tau = 0;
    float ee_eps = 0.0f;
    unsigned long long* iter_sum = nullptr;
};

static int extras_of(const tsenor_scores_t* s, Extras* x) {
    x->per_block_tau = s->per_block_tau ? 1 : 0;
    if (!(s->early_exit_eps >= 0.0f) || !std::isfinite(s->early_exit_eps)) return TSENOR_ERR_ARG;
    x->ee_eps = s->early_exit_eps;
    x->iter_sum = reinterpret_cast<unsigned long long*>(s->dev_iters_out);
    return TSENOR_OK;
}

static int solve_on(const tsenor::ScoreSrc& src, const Extras& x, int64_t rows, int64_t cols, int N, int M,
                    float tau, int iters, int ls_steps, uint32_t* mask_bits_out, int32_t* dev_status,
                    cudaStream_t st) {
    if (N == 0 || N == M) return trivial_mask(mask_bits_out, rows, cols, N == M, st);
    tsenor::Params P{};
    P.src = src;
    P.bits = mask_bits_out; P.wpr = (cols + 31) / 32;
    P.rows = rows; P.cols = cols;
    set_N(P, N);
    set_tau(P, tau);
    P.per_block_tau = x.per_block_tau;
    P.ee_eps = x.ee_eps; P.iter_sum = x.iter_sum;
    P.iters = iters; P.ls_steps = ls_steps;
    P.status = dev_status;
    return dispatch<0>(P, M, st);
}

int tsenor_solve(const float* scores, int64_t rows, int64_t cols, int64_t ld, int N, int M, float tau, int iters,
                 int ls_steps, uint32_t* mask_bits_out, int32_t* dev_status, tsenor_stream_t stream) {
    if (!valid_M(M) || N < 0 || N > M) return TSENOR_ERR_NM;
    if (int rc = check_matrix(rows, cols, ld, M)) return rc;
    if (iters < 0 || !(tau >= 0.0f) || !std::isfinite(tau)) return TSENOR_ERR_ARG;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!scores || !mask_bits_out) return TSENOR_ERR_NULL;
    return solve_on(abs_source(scores, ld), Extras{}, rows, cols, N, M, tau, iters, ls_steps, mask_bits_out,
                    dev_status, (cudaStream_t)stream);
}

int tsenor_solve_scores(const tsenor_scores_t* s, int64_t rows, int64_t cols, int N, int M, float tau, int iters,
                        int ls_steps, uint32_t* mask_bits_out, int32_t* dev_status, tsenor_stream_t stream) {
    if (!valid_M(M) || N < 0 || N > M) return TSENOR_ERR_NM;
    if (int rc = check_matrix(rows, cols, cols, M)) return rc;
    if (iters < 0 || !(tau >= 0.0f) || !std::isfinite(tau)) return TSENOR_ERR_ARG;
    tsenor::ScoreSrc src{};
    if (int rc = make_source(s, cols, &src)) return rc;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!mask_bits_out) return TSENOR_ERR_NULL;
    Extras x;
    if (int rc = extras_of(s, &x)) return rc;
    return solve_on(src, x, rows, cols, N, M, tau, iters, ls_steps, mask_bits_out, dev_status,
                    (cudaStream_t)stream);
}

static int max_on(const tsenor::ScoreSrc& src, int64_t rows, int64_t cols, float* dev_max_out, cudaStream_t st) {
    if (cudaMemsetAsync(dev_max_out, 0, sizeof(float), st) != cudaSuccess) return finish_launch(), TSENOR_ERR_CUDA;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    const int64_t quads = rows * (cols / 4), grid = scan_grid(quads);
    const auto kernel = batched_scan(src, quads, grid * 256) ? scores_max_kernel<true> : scores_max_kernel<false>;
    kernel<<<(unsigned)grid, 256, 0, st>>>(src, quad_walk(rows, cols), reinterpret_cast<unsigned int*>(dev_max_out));
    return finish_launch();
}

int tsenor_scores_max(const tsenor_scores_t* s, int64_t rows, int64_t cols, float* dev_max_out,
                      tsenor_stream_t stream) {
    if (rows < 0 || cols < 0 || cols % 4) return TSENOR_ERR_SHAPE;
    tsenor::ScoreSrc src{};
    if (int rc = make_source(s, cols, &src)) return rc;
    if (!dev_max_out) return TSENOR_ERR_NULL;
    return max_on(src, rows, cols, dev_max_out, (cudaStream_t)stream);
}

int tsenor_scores_materialize(const tsenor_scores_t* s, int64_t rows, int64_t cols, float* scores_out,
                              int64_t ld_out, tsenor_stream_t stream) {
    if (rows < 0 || cols < 0 || cols % 4 || ld_out < cols) return TSENOR_ERR_SHAPE;
    tsenor::ScoreSrc src{};
    if (int rc = make_source(s, cols, &src)) return rc;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!scores_out) return TSENOR_ERR_NULL;
    materialize_kernel<<<grid_for(rows * (cols / 4), 256), 256, 0, (cudaStream_t)stream>>>(
        src, rows, cols, scores_out, ld_out);
    return finish_launch();
}

int tsenor_keep_better(const tsenor_scores_t* s, int64_t rows, int64_t cols, const uint32_t* prev_mask,
                       uint32_t* mask_inout, double* dev_obj2_out, tsenor_stream_t stream) {
    if (rows < 0 || cols < 0 || cols % 4) return TSENOR_ERR_SHAPE;
    tsenor::ScoreSrc src{};
    if (int rc = make_source(s, cols, &src)) return rc;
    if (!dev_obj2_out) return TSENOR_ERR_NULL;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(dev_obj2_out, 0, 2 * sizeof(double), st) != cudaSuccess)
        return finish_launch(), TSENOR_ERR_CUDA;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!prev_mask || !mask_inout) return TSENOR_ERR_NULL;
    const int64_t wpr = (cols + 31) / 32;
    const int64_t quads = rows * (cols / 4);
    objective_kernel<false, true><<<objective_grid(true, quads), objective_threads(true, quads), 0, st>>>(
        src, mask_inout, prev_mask, quad_walk(rows, cols), wpr, dev_obj2_out);
    if (int rc = finish_launch()) return rc;
    keep_better_kernel<<<grid_for(rows * wpr, 256), 256, 0, st>>>(dev_obj2_out, prev_mask, mask_inout, rows * wpr);
    return finish_launch();
}

int tsenor_simple_round(const float* plan_key, int64_t ld_plan, int64_t rows, int64_t cols, int N, int M,
                        uint32_t* mask_bits_out, tsenor_stream_t stream) {
    if (!valid_M(M) || N < 1 || N >= M) return TSENOR_ERR_NM;
    if (int rc = check_matrix(rows, cols, ld_plan, M)) return rc;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!plan_key || !mask_bits_out) return TSENOR_ERR_NULL;
    cudaStream_t st = (cudaStream_t)stream;
    switch (M) {
        case 4: return launch_simple_round<4>(plan_key, ld_plan, rows, cols, N, mask_bits_out, st);
        case 8: return launch_simple_round<8>(plan_key, ld_plan, rows, cols, N, mask_bits_out, st);
        case 16: return launch_simple_round<16>(plan_key, ld_plan, rows, cols, N, mask_bits_out, st);
        default: return launch_simple_round<32>(plan_key, ld_plan, rows, cols, N, mask_bits_out, st);
    }
}

static int dykstra_on(const tsenor::ScoreSrc& src, const Extras& x, int64_t rows, int64_t cols, int N, int M,
                      float tau, int iters, float* plan_out, int64_t ld_plan, int plan_is_log,
                      int32_t* dev_status, cudaStream_t st) {
    tsenor::Params P{};
    P.src = src;
    P.plan = plan_out; P.ld_plan = ld_plan; P.plan_is_log = plan_is_log;
    P.vec_plan = aligned16(plan_out, ld_plan);
    P.rows = rows; P.cols = cols;
    set_N(P, N);
    set_tau(P, tau);
    P.per_block_tau = x.per_block_tau;
    P.ee_eps = x.ee_eps; P.iter_sum = x.iter_sum;
    P.iters = iters; P.ls_steps = -1;
    P.status = dev_status;
    return dispatch<1>(P, M, st);
}

int tsenor_dykstra(const float* scores, int64_t rows, int64_t cols, int64_t ld, int N, int M, float tau, int iters,
                   float* plan_out, int64_t ld_plan, int plan_is_log, int32_t* dev_status, tsenor_stream_t stream) {
    if (!valid_M(M) || N < 1 || N >= M) return TSENOR_ERR_NM;
    if (int rc = check_matrix(rows, cols, ld, M)) return rc;
    if (ld_plan < cols) return TSENOR_ERR_SHAPE;
    if (iters < 0 || !(tau >= 0.0f) || !std::isfinite(tau)) return TSENOR_ERR_ARG;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!scores || !plan_out) return TSENOR_ERR_NULL;
    return dykstra_on(abs_source(scores, ld), Extras{}, rows, cols, N, M, tau, iters, plan_out, ld_plan, plan_is_log,
                      dev_status, (cudaStream_t)stream);
}

int tsenor_dykstra_scores(const tsenor_scores_t* s, int64_t rows, int64_t cols, int N, int M, float tau, int iters,
                          float* plan_out, int64_t ld_plan, int plan_is_log, int32_t* dev_status,
                          tsenor_stream_t stream) {
    if (!valid_M(M) || N < 1 || N >= M) return TSENOR_ERR_NM;
    if (int rc = check_matrix(rows, cols, cols, M)) return rc;
    if (ld_plan < cols) return TSENOR_ERR_SHAPE;
    if (iters < 0 || !(tau >= 0.0f) || !std::isfinite(tau)) return TSENOR_ERR_ARG;
    tsenor::ScoreSrc src{};
    if (int rc = make_source(s, cols, &src)) return rc;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!plan_out) return TSENOR_ERR_NULL;
    Extras x;
    if (int rc = extras_of(s, &x)) return rc;
    return dykstra_on(src, x, rows, cols, N, M, tau, iters, plan_out, ld_plan, plan_is_log,
                      dev_status, (cudaStream_t)stream);
}

int tsenor_round(const float* plan_key, int64_t ld_plan, const float* scores, int64_t ld, int64_t rows,
                 int64_t cols, int N, int M, int ls_steps, uint32_t* mask_bits_out, int32_t* dev_status,
                 tsenor_stream_t stream) {
    if (!valid_M(M) || N < 0 || N > M) return TSENOR_ERR_NM;
    if (int rc = check_matrix(rows, cols, ld, M)) return rc;
    if (ld_plan < cols) return TSENOR_ERR_SHAPE;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!plan_key || !scores || !mask_bits_out) return TSENOR_ERR_NULL;
    cudaStream_t st = (cudaStream_t)stream;
    if (N == 0 || N == M) return trivial_mask(mask_bits_out, rows, cols, N == M, st);
    tsenor::Params P{};
    P.src = abs_source(scores, ld);
    P.keys = plan_key; P.ld_keys = ld_plan;
    P.bits = mask_bits_out; P.wpr = (cols + 31) / 32;
    P.rows = rows; P.cols = cols;
    P.N = N; P.Nf = (float)N; P.log2N = 0.f;
    P.iters = 0; P.ls_steps = ls_steps;
    P.status = dev_status;
    P.vec_keys = aligned16(plan_key, ld_plan);
    return dispatch<2>(P, M, st);
}

int tsenor_objective(const float* scores, int64_t ld, const uint32_t* mask_bits, int64_t rows, int64_t cols,
                     double* dev_sum_out, tsenor_stream_t stream) {
    if (rows < 0 || cols < 0 || ld < cols || cols % 4) return TSENOR_ERR_SHAPE;
    if (!dev_sum_out) return TSENOR_ERR_NULL;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(dev_sum_out, 0, sizeof(double), st) != cudaSuccess) return finish_launch(), TSENOR_ERR_CUDA;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!scores || !mask_bits) return TSENOR_ERR_NULL;
    const int64_t wpr = (cols + 31) / 32, quads = rows * (cols / 4), grid = objective_grid(false, quads);
    const tsenor::ScoreSrc src = abs_source(scores, ld);
    const int threads = objective_threads(false, quads);
    const auto kernel =
        batched_scan(src, quads, grid * threads) ? objective_kernel<true, false> : objective_kernel<false, false>;
    kernel<<<(unsigned)grid, threads, 0, st>>>(src, mask_bits, nullptr, quad_walk(rows, cols), wpr, dev_sum_out);
    return finish_launch();
}

int tsenor_check(const uint32_t* mask_bits, int64_t rows, int64_t cols, int N, int M, int64_t* dev_bad_blocks_out,
                 tsenor_stream_t stream) {
    if (!valid_M(M) || N < 0 || N > M) return TSENOR_ERR_NM;
    if (int rc = check_matrix(rows, cols, cols, M)) return rc;
    if (!dev_bad_blocks_out) return TSENOR_ERR_NULL;
    cudaStream_t st = (cudaStream_t)stream;
    if (cudaMemsetAsync(dev_bad_blocks_out, 0, sizeof(int64_t), st) != cudaSuccess)
        return finish_launch(), TSENOR_ERR_CUDA;
    if (rows == 0 || cols == 0) return TSENOR_OK;
    if (!mask_bits) return TSENOR_ERR_NULL;
    const int64_t nblk = (rows / M) * (cols / M), wpr = (cols + 31) / 32;
    const auto kernel = M == 4 ? check_kernel<4> : M == 8 ? check_kernel<8> : M == 16 ? check_kernel<16> : check_kernel<32>;
    kernel<<<grid_for(nblk, 128), 128, 0, st>>>(mask_bits, rows, cols, wpr, N,
                                                reinterpret_cast<unsigned long long*>(dev_bad_blocks_out));
    return finish_launch();
}

int tsenor_max_abs(const float* scores, int64_t rows, int64_t cols, int64_t ld, float* dev_max_out,
                   tsenor_stream_t stream) {
    if (rows < 0 || cols < 0 || ld < cols || cols % 4) return TSENOR_ERR_SHAPE;
    if (!dev_max_out) return TSENOR_ERR_NULL;
    if (rows > 0 && cols > 0 && !scores) return TSENOR_ERR_NULL;
    return max_on(abs_source(scores, ld), rows, cols, dev_max_out, (cudaStream_t)stream);
}

int64_t tsenor_mask_words_per_row(int64_t cols) { return cols <= 0 ? 0 : (cols + 31) / 32; }

const char* tsenor_strerror(int status) {
    switch (status) {
        case TSENOR_OK: return "ok";
        case TSENOR_ERR_NULL: return "a required pointer is NULL";
        case TSENOR_ERR_SHAPE: return "bad shape: negative size, ld < cols, or rows/cols not a multiple of M (of 4)";
        case TSENOR_ERR_NM: return "bad N:M: M must be 4, 8, 16 or 32 and N within range";
        case TSENOR_ERR_ARG: return "bad argument: iters < 0 or tau negative / not finite";
        case TSENOR_ERR_CUDA: return "CUDA launch failed: see tsenor_last_cuda_error()";
        default: return "unknown status";
    }
}

int tsenor_last_cuda_error(void) { return g_last_cuda_error; }

int64_t tsenor_launch_count(void) { return (int64_t)g_launches.load(std::memory_order_relaxed); }

#ifdef TSENOR_BOUNDS
// Checked flavour only: *dev_flags_out (device) = what the index checks of all kernels have seen since
// the library was loaded (0: none has fired).
int tsenor_bounds_seen(int32_t* dev_flags_out, tsenor_stream_t stream) {
    if (!dev_flags_out) return TSENOR_ERR_NULL;
    const cudaError_t e = cudaMemcpyFromSymbolAsync(dev_flags_out, tsenor::g_bounds_seen, sizeof(int32_t), 0,
                                                    cudaMemcpyDeviceToDevice, (cudaStream_t)stream);
    if (e != cudaSuccess) g_last_cuda_error = (int)e;
    return e == cudaSuccess ? TSENOR_OK : TSENOR_ERR_CUDA;
}
#endif

int tsenor_set_layout(int layout) {
    if (layout < TSENOR_LAYOUT_AUTO || layout > TSENOR_LAYOUT_LATENCY) return TSENOR_ERR_ARG;
    return g_layout.exchange(layout, std::memory_order_relaxed);
}

}  // extern "C"
