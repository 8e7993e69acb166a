// Device code of the TSENOR hot path for sm_100a: block loader, log-domain
// Dykstra iterations (Algorithm 1), greedy selection and local search
// (Algorithm 2, Eq. 6), bit-packed mask writer.
//
// Layout in one sentence: a warp owns a unit of BPW consecutive blocks, stages
// their scores in shared memory with coalesced loads, runs Dykstra for them
// entirely in registers, hands the log-plan to the rounding stage through shared
// memory, and writes whole 32-bit mask words back.  Nothing in the method couples
// two warps, so a CTA is one warp and there is no barrier to wait at (the
// stopping-test mode at M = 32 excepted, see CtaWarps).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace tsenor {

constexpr unsigned FULL = 0xffffffffu;

enum : int { DEV_NONFINITE = 1, DEV_UNDERFILLED = 2, DEV_INTERNAL = 4 };

// Checked build flavour (-DTSENOR_BOUNDS, a second library built from the same sources): every
// data-dependent or computed index of the loaders, the rounding tables, the local search and the
// writers is tested against the extent of its array before the access; a bad one ORs
// DEV_INTERNAL into the status word and the access is skipped (nothing traps, nothing faults).
// It stands in for a memory checker on machines where none can be run.  In the normal build
// TS_CHECK(x) is the constant true and costs nothing.
// A kernel that makes such checks calls bounds_begin and bounds_end with all its threads; what they saw
// is also kept in g_bounds_seen (tsenor_bounds_seen reads it), for entry points without a status word.
#ifdef TSENOR_BOUNDS
__shared__ int g_bounds_flags;
__device__ int g_bounds_seen;
#define TS_CHECK(cond) ((cond) ? true : (atomicOr(&tsenor::g_bounds_flags, tsenor::DEV_INTERNAL), false))
__device__ __forceinline__ void bounds_begin() {
    if (threadIdx.x == 0) g_bounds_flags = 0;
    __syncthreads();
}
__device__ __forceinline__ int bounds_end() {
    __syncthreads();
    if (threadIdx.x == 0 && g_bounds_flags) atomicOr(&g_bounds_seen, g_bounds_flags);
    return g_bounds_flags;
}
#else
#define TS_CHECK(cond) true
__device__ __forceinline__ void bounds_begin() {}
__device__ __forceinline__ int bounds_end() { return 0; }
#endif

// ---------------------------------------------------------------------------
// Dykstra register layouts.
//   V = 0  throughput: a block is spread over LPB = PR*PC lanes arranged as PR x PC; each lane
//          keeps an MR x MC sub-tile, 4 x 8 (4 x 4 for M = 4), the fewest exchanges per element
//          that the registers allow.  Row sums are reduced over the PC lanes that share rows,
//          column sums over the PR lanes that share columns.  Used whenever the matrix has
//          enough blocks to fill the GPU.
//   V = 1  latency, for matrices too small for that.  M < 32: a block over M lanes, of which lane i
//          keeps row i and, a second time, column i ("twin" layout, see twin_plan): twice the
//          element-wise work, but all sums are a lane's own and the scalings cross the lanes by two
//          shared-memory broadcasts an iteration where sub-tiles need six to eight dependent
//          shuffles.  M = 32: the sub-tiles of V = 0 with what a lone warp waits for taken out: scalar
//          adds in the exchanges, one vote on the range test, scores kept beside the keys.
//   V = 3  spread, M = 8 and 16: a block over M lanes as in V = 1 (so a unit rounds in one pass), but
//          in sub-tiles, each element once: for what lies between V = 1 and a full GPU, and for few iterations.
// ---------------------------------------------------------------------------
template <int M, int V> struct Tile;
template <int V> struct Tile<32, V> { static constexpr int PR = 8, PC = 4, MR = 4, MC = 8; };
template <int V> struct Tile<16, V> { static constexpr int PR = 4, PC = 2, MR = 4, MC = 8; };
template <int V> struct Tile<8, V>  { static constexpr int PR = 2, PC = 1, MR = 4, MC = 8; };
template <int V> struct Tile<4, V>  { static constexpr int PR = 1, PC = 1, MR = 4, MC = 4; };
template <> struct Tile<16, 3> { static constexpr int PR = 4, PC = 4, MR = 4, MC = 4; };
template <> struct Tile<8, 3>  { static constexpr int PR = 4, PC = 2, MR = 2, MC = 4; };

template <int M_, int V_> struct Geom {
    static constexpr int M = M_, V = V_;
    static constexpr bool TWIN = (V == 1 && M < 32);
    using T = Tile<M, V>;
    static constexpr int LPB = TWIN ? M : T::PR * T::PC;   // lanes per block (Dykstra)
    static constexpr int BPW = 32 / LPB;             // blocks per warp
    static constexpr int UW = BPW * M;               // columns of a unit: its blocks side by side
    static constexpr int WS = UW + 1;                // shared row stride (floats)
    static constexpr int GPW = 32 / M;               // rounding groups per warp (blocks of one mask word)
    static constexpr int PASSES = BPW / GPW;         // rounding passes per warp
    static constexpr int RO = TWIN ? 1 : T::MR / T::PC, CO = TWIN ? 1 : T::MC / T::PR;   // lines a lane finishes
    static_assert(T::MR >= T::PC && T::MC >= T::PR && T::MC % 2 == 0 && (T::MR * T::MC) % 4 == 0, "tile shape");
    static_assert(T::PR * T::MR == M && T::PC * T::MC == M, "tile covers the block");
    static_assert(BPW % GPW == 0, "a unit is a whole number of mask words wide");
    static_assert(TWIN || 32 * T::MR * T::MC <= M * WS, "the stash of t0 fits in the key panel");
};

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// NaN if either is: a block poisoned by a non-finite score stays NaN as a whole (see out_of_window).
__device__ __forceinline__ float min_nan(float a, float b) {
    float y;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
    return y;
}

// Register r of a lane holds line (r ^ perm) of its sub-tile, where perm is
// built from the lane's coordinate along the reduction direction.  With that
// permutation the recursive-halving exchange below needs no selects: every
// lane always sends its upper half and keeps its lower half.
template <int K, int P> __device__ __forceinline__ int xor_perm(int l) {
    int g = 0;
#pragma unroll
    for (int s = 0; (1 << s) < P; ++s) g |= ((l >> s) & 1) * (K >> (s + 1));
    return g;
}

struct OpAdd {
    static constexpr bool packed = false;
    __device__ __forceinline__ float operator()(float a, float b) const { return a + b; }
};
struct OpAdd2 : OpAdd { static constexpr bool packed = true; };   // pairs by the packed add
struct OpMax {
    static constexpr bool packed = false;
    __device__ __forceinline__ float operator()(float a, float b) const { return fmaxf(a, b); }
};

// After the call v[0 .. K/P) hold the reduction over the P lanes (lane stride
// `base`) of the lines those registers stand for.
template <int K, int P, class Op>
__device__ __forceinline__ void reduce_scatter(float (&v)[K], int base, Op op) {
#pragma unroll
    for (int s = 0; (1 << s) < P; ++s) {
        const int h = K >> (s + 1);
#pragma unroll
        for (int k = 0; k < h; k += 2) {
            const float x = __shfl_xor_sync(FULL, v[k + h], base << s);
            if (h == 1) {
                v[k] = op(v[k], x);
                continue;
            }
            const float y = __shfl_xor_sync(FULL, v[k + 1 + h], base << s);
            if (Op::packed) {
                const float2 r = __fadd2_rn(make_float2(v[k], v[k + 1]), make_float2(x, y));
                v[k] = r.x;
                v[k + 1] = r.y;
            } else {
                v[k] = op(v[k], x);
                v[k + 1] = op(v[k + 1], y);
            }
        }
    }
}
// Inverse exchange: v[0 .. K/P) valid on entry, all K valid on return.
template <int K, int P>
__device__ __forceinline__ void all_gather(float (&v)[K], int base) {
    constexpr int S = (P == 1) ? 0 : (P == 2) ? 1 : (P == 4) ? 2 : 3;
#pragma unroll
    for (int s = S - 1; s >= 0; --s) {
        const int h = K >> (s + 1);
#pragma unroll
        for (int k = 0; k < h; ++k)
            v[k + h] = __shfl_xor_sync(FULL, v[k], base << s);
    }
}

// Adds log2 of a running product of scalings (sign -1: of its reciprocal) to a Kahan-compensated potential.  The potentials
// (one row and one column at M = 32) live in shared memory, private to the lane: they are touched
// once in up to 48 iterations, and without them the loop fits in the 96 registers of 20 warps per SM.
// Near 1, where the products of converged blocks are, by the Taylor series of log2(1 + t) (error below 4e-10;
// lg2.approx is only good to 2^-22 there, and what comes in at the end stays in the plan).
__device__ __forceinline__ float log2_of_product(float p) {
    const float t = p - 1.0f;
    const float series = t * fmaf(t, fmaf(t, fmaf(t, -0.36067376f, 0.48089835f), -0.72134752f), 1.44269504f);
    return fabsf(t) < 0.015625f ? series : lg2_approx(p);
}
template <bool LAST = false>
__device__ __forceinline__ float add_potential(float2* p, float prod, float sign = 1.0f) {
    const float2 c = *p;                     // value, compensation
    const float y = sign * (LAST ? log2_of_product(prod) : lg2_approx(prod)) - c.y;
    const float v = c.x + y;
    *p = make_float2(v, (v - c.x) - y);
    return v;
}

// ---------------------------------------------------------------------------
// Algorithm 1 in potential form, with stabilised linear-domain steps.
//
// In the log domain the three projections only ever add a row term and a
// column term to x + q, and after the clip x = min(t, 0), q = max(t, 0) for
// t = x + q.  So the whole state is t_ij = t0_ij + F_i + G_j with
// t0 = tau |w| (base-2 units here), and with U = 2^t (the unclipped S .* Q)
// one iteration is
//     e_ij   = min(U_ij, 1)                        (S after the previous clip)
//     rho_i  = N / sum_j e_ij                      (projection on C1)
//     kap_j  = N / sum_i e_ij rho_i                (projection on C2)
//     U_ij  <- U_ij rho_i kap_j ,  F_i += log2 rho_i ,  G_j += log2 kap_j
// with the clip (C3) and the dual update implicit in the next e.  U is the
// linear-domain iterate of Algorithm 1 (kept as U / R_i in the registers, see
// the loop below).  It is trusted only while the scalings
// applied since it was last rebuilt stay small, and is then rebuilt as
// 2^(t0 + F + G) from the log-domain potentials; that is what keeps large
// tau |w| safe in fp32.  Every CHECK iterations the products of rho_i and of
// kap_j since the last rebuild are tested against [2^-16, 2^17), and U is
// rebuilt when one of them has left that range or after MAXRUN iterations.
// From iteration 1 on a row sum of e is in [N/M, M] and a column sum of e*rho in [N/M, N M] (an entry of e
// is at most its row's sum, and no column of e sums to less than 1), so rho is in [N/M, M], kap in [1/M, M],
// and an iteration moves an entry of U by at most 2^10: between two rebuilds by at most
// 2^(34 + 10 CHECK) = 2^74 relative to its value U0 at the first.  Where ex2 overflowed, U is still
// above the cap, and where it flushed U0 (below 2^-126) still below 2^-52, when the rebuild restores it.
// The registers hold V = U / R = U0 K (below; R and K the products of rho and kap), which may leave the
// floats in the middle of a run though U0 did not.  The products keep subnormal numbers, so that an entry
// is lost only below 2^-150; K was then at least 2^-26 (2^-16 at the tests before and after it, 2^-5 an
// iteration in between), so U = U0 K' R' stays below 2^(-150 + 74 + 26) = 2^-50 until the rebuild.
// One that overflows (K at most 2^27) stays above 2^(128 - 72 - 27) = 2^29.  All of this is the worst case
// (in practice the scalings are within a few percent of 1 after the first
// dozen iterations and the runs reach MAXRUN).  Iteration 0 has no clip yet and is done
// entirely in the log domain with the column maximum subtracted, because
// 2^t0 of a whole column can underflow against a large entry elsewhere in
// its rows.
//
// On entry t holds t0 with its row maximum subtracted (exact no-op for the
// method: the first row projection removes any row constant); on return t
// holds the final t = x + q.  stash: 32 * MR * MC floats of shared memory
// private to the warp (keeps t0 while the registers hold U); pot: 32 * (RO + CO)
// float2 of it for the owned potentials.
// ---------------------------------------------------------------------------
constexpr int CHECK = 4;     // iterations between range tests of the accumulated scalings
constexpr int MAXRUN = 48;   // longest run of linear-domain iterations (multiple of CHECK; see run_length)

// Exponent field outside [127-16, 127+16] <=> product outside [2^-16, 2^17).  A product that is inf or
// NaN (exponent field 255: a block poisoned by a non-finite score) does not vote, so that it cannot
// change when the other blocks of its warp rebuild.
__device__ __forceinline__ bool out_of_window(float p) {
    const unsigned e = (__float_as_uint(p) >> 23) & 0xffu;
    return (e - 111u) > 32u && e != 255u;
}

// Products in the window, and no others, are at most WINDOW from its lower end as bit patterns.
constexpr unsigned WINDOW = (33u << 23) - 1u;
__device__ __forceinline__ unsigned window_distance(float p) { return __float_as_uint(p) - (111u << 23); }

// One iteration t >= 1 on the linear-domain iterate.  Element-wise work runs on
// pairs of columns with the packed fp32x2 add / mul / fma of sm_100 (half the
// issue slots).  The row scalings are never applied to the tile: the registers
// hold V = U / R_i with R_i the product of the rho_i since the last rebuild, and
// one multiply per element (by kap_j) is left.  Four fp32 operations per element
// and iteration, in one of two forms:
//   M = 32   rs[a] = R_i:    e = sat(V R_i) = min(U, 1) by a saturating multiply (FMA pipe), row
//            sums of e give rho_i = N / sum, column sums are sum_i e_ij rho_i, kap_j = N / sum,
//            R_i <- R_i rho_i in every lane of the row;
//   M <= 16  rs[a] = 1/R_i:  m = min(V, 1/R_i) = e / R_i (the clip threshold moves instead of the
//            tile), whose row sums s give the new 1/R_i = s / N and the column sums c = sum_i m_ij / s_i
//            (= sum_i e_ij rho_i / N) give kap_j = 1 / c.  Only s carries a rounding from one iteration
//            to the next: 1/N is split in two floats, so that s / N is rounded once whatever N is.
// The product form rounds e, rho_i and R_i as well, every iteration, and that shows where few entries of
// a line are left between 0 and the cap: distance of the log-plan from the fp64 iterate (2-norm, 512 x 512,
// eighteen matrices) 1.36e-7 at 1:4 by products and 1.14e-7 by thresholds, 3.15e-7 and 2.84e-7 at 3:4,
// 7.1e-7 and 6.3e-7 at 7:8; of the plan 3.8e-7 and 3.3e-7 at 1:4.  Time 946 us against 930 (4096 x 4096
// 2:4), 858 against 853 (4:8): no factor N is left, which pays for the half-rate min.  (Without the split of
// 1/N 912 and 831, but at N = 3, 6, 7 no more exact than the products.)  At M = 16, where the thresholds need a
// second gather, the two take the same time (875 us, 4096 x 4096 8:16), but by thresholds a converged block
// recurs sooner (see below; Student-t scores 301 us against 409) and the log-plan is as exact or more so (15:16:
// 0.73 of the distance).  At M = 32 the thresholds are 3.5 % slower.
//
// Whether the exchanges' adds and (M >= 16) the row factors are packed too (PACK) is a matter of how the
// packed and the scalar instructions of the other warps interleave on the FMA pipes: the factors
// gain 1 to 2 % at every size, the adds as much for M >= 16 and nothing for M = 8.  A lone warp, and
// the stopping test's mixture, only see the packed ones' longer latency (14336 x 32: 69.4 us
// without, 74.5 with).
template <int M> struct PackAdd { static constexpr bool value = (M >= 16); };
template <int M> struct ByThreshold { static constexpr bool value = (M <= 16); };

// 1/N as the sum of two floats (made on the host).
struct InvN {
    float hi, lo;
    __device__ __forceinline__ float times(float s) const { return fmaf(s, hi, s * lo); }
    __device__ __forceinline__ float2 times(float2 s) const {
        return __ffma2_rn(s, make_float2(hi, hi), __fmul2_rn(s, make_float2(lo, lo)));
    }
};

// Copy of a lane's state in local memory (registers are what the loop is short of).
template <int CELLS> struct Snapshot {
    alignas(8) unsigned cell[CELLS];
    __device__ __forceinline__ unsigned* hidden() {     // keeps the compiler from making registers of it
        unsigned* p = cell;
        asm volatile("" : "+l"(p));
        return p;
    }
    template <int K> __device__ __forceinline__ void take(int at, const float (&v)[K]) {
        unsigned* const p = hidden() + at;
#pragma unroll
        for (int k = 0; k < K; ++k) p[k] = __float_as_uint(v[k]);
    }
    template <int K> __device__ __forceinline__ void take(int at, const float2 (&v)[K]) {
        uint2* const p = reinterpret_cast<uint2*>(hidden() + at);
#pragma unroll
        for (int k = 0; k < K; ++k) p[k] = make_uint2(__float_as_uint(v[k].x), __float_as_uint(v[k].y));
    }
    // Bits in which v differs from what was taken.
    template <int K> __device__ __forceinline__ unsigned differ(int at, const float (&v)[K]) {
        const unsigned* const p = hidden() + at;
        unsigned d = 0u;
#pragma unroll
        for (int k = 0; k < K; ++k) d |= p[k] ^ __float_as_uint(v[k]);
        return d;
    }
    template <int K> __device__ __forceinline__ unsigned differ(int at, const float2 (&v)[K]) {
        const uint2* const p = reinterpret_cast<const uint2*>(hidden() + at);
        unsigned d = 0u;
#pragma unroll
        for (int k = 0; k < K; ++k) d |= (p[k].x ^ __float_as_uint(v[k].x)) | (p[k].y ^ __float_as_uint(v[k].y));
        return d;
    }
};

// KEEP: last receives the column scalings of the lines this lane owns.
// DELTA: also returns this lane's share of the marginal violation seen by the iteration,
// max over the lines it owns of |row sum of e - N| and |column sum of e rho - N|.
template <class G, bool PACK, bool DELTA = false, bool KEEP = false>
__device__ __forceinline__ float dykstra_step(float2 (&V)[G::T::MR][G::T::MC / 2], float (&rs)[G::T::MR],
                                              float (&Pc)[G::CO], float (&last)[G::CO], float Nf, const InvN& iN) {
    using T = typename G::T;
    constexpr int M = G::M;
    constexpr bool THR = ByThreshold<M>::value;
    constexpr int MR = T::MR, MC = T::MC, PR = T::PR, PC = T::PC;
    constexpr int RO = G::RO, CO = G::CO, MP = MC / 2;
    using Add = typename std::conditional<PACK && PackAdd<M>::value, OpAdd2, OpAdd>::type;
    float2 m[MR][MP];
    float rp[MR], sc[MR], cp[MC], kap[MC];
#pragma unroll
    for (int a = 0; a < MR; ++a) {
        float2 s2;
#pragma unroll
        for (int b = 0; b < MP; ++b) {
            if (THR) m[a][b] = make_float2(min_nan(V[a][b].x, rs[a]), min_nan(V[a][b].y, rs[a]));
            else m[a][b] = make_float2(__saturatef(V[a][b].x * rs[a]), __saturatef(V[a][b].y * rs[a]));
            s2 = (b == 0) ? m[a][b] : __fadd2_rn(s2, m[a][b]);
        }
        rp[a] = s2.x + s2.y;
    }
    reduce_scatter<MR, PC>(rp, 1, Add());
    float delta = 0.0f;
    if (DELTA) {   // row sums of e
#pragma unroll
        for (int k = 0; k < RO; ++k) delta = fmaxf(delta, fabsf((THR ? rp[k] * rcp_approx(rs[k]) : rp[k]) - Nf));
    }
#pragma unroll
    for (int k = 0; k < RO; ++k) sc[k] = THR ? rcp_approx(rp[k]) : Nf * rcp_approx(rp[k]);
    all_gather<MR, PC>(sc, 1);
#pragma unroll
    for (int b = 0; b < MP; ++b) {
        float2 c2 = __fmul2_rn(m[0][b], make_float2(sc[0], sc[0]));
#pragma unroll
        for (int a = 1; a < MR; ++a) c2 = __ffma2_rn(m[a][b], make_float2(sc[a], sc[a]), c2);
        cp[2 * b] = c2.x;
        cp[2 * b + 1] = c2.y;
    }
    reduce_scatter<MC, PR>(cp, PC, Add());
    if (DELTA) {
#pragma unroll
        for (int k = 0; k < CO; ++k) delta = fmaxf(delta, fabsf((THR ? Nf * cp[k] : cp[k]) - Nf));
    }
#pragma unroll
    for (int k = 0; k < CO; ++k) {
        kap[k] = THR ? rcp_approx(cp[k]) : Nf * rcp_approx(cp[k]);
        Pc[k] *= kap[k];
        if (KEEP) last[k] = kap[k];
    }
    all_gather<MC, PR>(kap, PC);
    if constexpr (THR) {
        if constexpr (RO == 1) {
            rs[0] = iN.times(rp[0]);
        } else {
#pragma unroll
            for (int k = 0; k < RO; k += 2) {
                const float2 r = iN.times(make_float2(rp[k], rp[k + 1]));
                rs[k] = r.x;
                rs[k + 1] = r.y;
            }
        }
        all_gather<MR, PC>(rs, 1);
    } else if constexpr (PACK) {
#pragma unroll
        for (int a = 0; a < MR; a += 2) {
            const float2 r = __fmul2_rn(make_float2(rs[a], rs[a + 1]), make_float2(sc[a], sc[a + 1]));
            rs[a] = r.x;
            rs[a + 1] = r.y;
        }
    } else {
#pragma unroll
        for (int a = 0; a < MR; ++a) rs[a] *= sc[a];
    }
#pragma unroll
    for (int a = 0; a < MR; ++a)
#pragma unroll
        for (int b = 0; b < MP; ++b) V[a][b] = __fmul2_rn(V[a][b], make_float2(kap[2 * b], kap[2 * b + 1]));
    return delta;
}

// Returns the number of iterations run: iters, or fewer in the stopping-test mode (EE, ee_eps > 0):
// after every group of CHECK iterations, i.e. at iterations 5, 9, 13, ... of Algorithm 1, the
// warp stops once the marginal violation of every block it holds is below ee_eps.
// ---------------------------------------------------------------------------
// Recurring states.  Algorithm 1 converges, and the state of the linear-domain loop (V and the row
// factors) is a few thousand floats that depend on nothing but themselves: once the scalings are within
// rounding of 1 it returns, bit for bit, to where it was one, two or four iterations before.  All that
// is left of the T iterations then repeats what was seen, so the warp runs (T - t) mod 4 more and is done:
// its state is the one that all T would end in.  Nothing is assumed about convergence; a state that has not
// recurred, in every bit and in every block of the warp, is iterated on.
//
// Looking costs a copy of the state and a comparison per four iterations, so a warp looks only once a run
// has ended with every column scaling within NEAR_ONE of 1, and in a run of its own (at most LOOKS of them)
// that begins with a rebuild: that takes out the roundings which V has gathered, so that the plan is as
// exact as after all T (log-plan's distance from the fp64 iterate, mean over 1:M to M-1:M and four
// distributions, against running on: 1.00 at M = 4 and 8, 0.97 at 16, 1.00 at 32).  The first runs are
// short, since that is when most blocks of heavy-tailed scores get there: of |Student-t| and outlier-column
// matrices under tau = 200 / max nearly all within 30 to 80 iterations; of Gaussian ones hardly any in 300.
// 4096 x 4096, us before / now, for Student, outlier, Wanda-style and Gaussian scores:
//   2:4    933 / 296, 928 / 438, 931 / 680, 924 / 902        4:8    862 / 315, 857 / 474, 863 / 574, 851 / 835
//   8:16   871 / 284, 863 / 438, 872 / 633, 858 / 856        16:32  864 / 375, 855 / 418, 865 / 671, 855 / 864
// V = 1 does not look: with a warp or two per scheduler the slowest block of the matrix sets the time
// (256 x 264 2:4 with outlier columns: 26.2, 28.1 with looking).
// ---------------------------------------------------------------------------
constexpr float NEAR_ONE = 3.6e-7f;      // three units in the last place above 1
constexpr int LOOKS = 2;
template <class G, bool EE> struct Recurrence { static constexpr bool value = !EE && (G::V == 0 || G::V == 3); };
// Length of the run that starts at iteration t: one more than a multiple of CHECK, so that the loop after the
// groups of CHECK leaves the scalings to be looked at in registers.  At M = 32 one short run, else two, where
// enough iterations are left to pay for a rebuild more (2048 x 2048 4:8, 50 iterations: 73.6 us without, 80.1 with).
template <class G, bool LOOK> __device__ __forceinline__ int run_length(int t, int iters) {
    if (!LOOK) return MAXRUN;
    return (G::V == 0 && iters >= 120 && t <= (G::M == 32 ? 1 : MAXRUN / 2 + 2)) ? MAXRUN / 2 + 1 : MAXRUN + 1;
}
constexpr int WORTH_LOOKING = 32;        // iterations left

template <class G, bool EE>
__device__ __forceinline__ int dykstra_iterate(float (&t)[G::T::MR][G::T::MC], float* stash, float2* pot, int lane,
                                               float Nf, const InvN& iN, float log2N, int iters, float ee_eps) {
    using T = typename G::T;
    constexpr int MR = T::MR, MC = T::MC, PR = T::PR, PC = T::PC;
    constexpr int RO = G::RO, CO = G::CO;
    constexpr int MP = MC / 2, NQ = MR * MC / 4;
    constexpr bool PACK = (G::V == 0 && !EE);
    constexpr bool LOOK = Recurrence<G, EE>::value;
    float F[MR], Gc[MC];
    float rs[MR];
    float Pc[CO];              // products of kap since the last rebuild; rs[0 .. RO): those of rho, or 1 / them
    constexpr float SIGN = ByThreshold<G::M>::value ? -1.0f : 1.0f;
    if (iters <= 0) return 0;
    float2* const fpot = pot + lane;                 // the owned potentials, compensated
    float2* const gpot = pot + RO * 32 + lane;
    float4* const st4 = reinterpret_cast<float4*>(stash) + lane;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {   // sub-tile in row-major order, four elements per slot
        const int e = 4 * q;
        st4[q * 32] = make_float4(t[e / MC][e % MC], t[(e + 1) / MC][(e + 1) % MC], t[(e + 2) / MC][(e + 2) % MC],
                                  t[(e + 3) / MC][(e + 3) % MC]);
    }
    {   // iteration 0, log domain
        float rp[MR];
#pragma unroll
        for (int a = 0; a < MR; ++a) {
            float s = 0.f;
#pragma unroll
            for (int b = 0; b < MC; ++b) s += ex2_approx(t[a][b]);
            rp[a] = s;
        }
        reduce_scatter<MR, PC>(rp, 1, OpAdd());
#pragma unroll
        for (int k = 0; k < RO; ++k) {
            F[k] = log2N - lg2_approx(rp[k]);
            fpot[k * 32] = make_float2(F[k], 0.f);
            rs[k] = 1.0f;
        }
        all_gather<MR, PC>(F, 1);
        float cm[MC];
#pragma unroll
        for (int b = 0; b < MC; ++b) {
            float m = t[0][b] + F[0];
#pragma unroll
            for (int a = 1; a < MR; ++a) m = fmaxf(m, t[a][b] + F[a]);
            cm[b] = m;
        }
        reduce_scatter<MC, PR>(cm, PC, OpMax());
        all_gather<MC, PR>(cm, PC);
        float cp[MC];
#pragma unroll
        for (int b = 0; b < MC; ++b) {
            float s = 0.f;
#pragma unroll
            for (int a = 0; a < MR; ++a) s += ex2_approx((t[a][b] + F[a]) - cm[b]);
            cp[b] = s;
        }
        reduce_scatter<MC, PR>(cp, PC, OpAdd());
#pragma unroll
        for (int k = 0; k < CO; ++k) {
            gpot[k * 32] = make_float2((log2N - cm[k]) - lg2_approx(cp[k]), 0.f);
            Pc[k] = 1.0f;
        }
    }
    // Iterations 1 .. iters-1 in runs: rebuild U from the potentials, then groups of
    // CHECK iterations with the range test of the accumulated scalings between groups.
    float2 V[MR][MP];
    float last[CO];            // column scalings of the last iteration
    int it = 1;
    int look = 0;              // 2 x (runs that looked for a recurring state) + (the next one is to)
#pragma unroll 1
    while (it < iters) {
#pragma unroll
        for (int k = 0; k < RO; ++k) F[k] = add_potential(fpot + k * 32, rs[k], SIGN);
#pragma unroll
        for (int k = 0; k < CO; ++k) { Gc[k] = add_potential(gpot + k * 32, Pc[k]); Pc[k] = 1.0f; }
        all_gather<MR, PC>(F, 1);
        all_gather<MC, PR>(Gc, PC);
#pragma unroll
        for (int q = 0; q < NQ; ++q) {   // pairs never straddle a row (MC is even)
            const int a0 = (4 * q) / MC, b0 = (4 * q) % MC, a1 = (4 * q + 2) / MC, b1 = (4 * q + 2) % MC;
            const float4 v = st4[q * 32];
            const float2 x0 = __fadd2_rn(__fadd2_rn(make_float2(v.x, v.y), make_float2(F[a0], F[a0])),
                                         make_float2(Gc[b0], Gc[b0 + 1]));
            const float2 x1 = __fadd2_rn(__fadd2_rn(make_float2(v.z, v.w), make_float2(F[a1], F[a1])),
                                         make_float2(Gc[b1], Gc[b1 + 1]));
            V[a0][b0 / 2] = make_float2(ex2_approx(x0.x), ex2_approx(x0.y));
            V[a1][b1 / 2] = make_float2(ex2_approx(x1.x), ex2_approx(x1.y));
        }
#pragma unroll
        for (int a = 0; a < MR; ++a) rs[a] = 1.0f;     // R_i = 1
        int run_end = LOOK ? min(iters, it + run_length<G, LOOK>(it, iters)) : (iters - it > MAXRUN) ? it + MAXRUN : iters;
        const auto out_of_range = [&]() {
            // V = 0: a first, cheap test (a subtraction and a maximum per line, every four iterations)
            // that also catches inf, NaN and zero; what it catches is looked at properly (1.5 to 4 %
            // of the loop).  A lone warp waits longer for the second vote than it saves.
            unsigned far = 0u;
#pragma unroll
            for (int k = 0; k < RO; ++k) far = max(far, window_distance(rs[k]));
#pragma unroll
            for (int k = 0; k < CO; ++k) far = max(far, window_distance(Pc[k]));
            bool w = false;
            if (G::V != 0 || __any_sync(FULL, far > WINDOW)) {
#pragma unroll
                for (int k = 0; k < RO; ++k) w |= out_of_window(rs[k]);
#pragma unroll
                for (int k = 0; k < CO; ++k) w |= out_of_window(Pc[k]);
                w = __any_sync(FULL, w);
            }
            return w;
        };
        bool wide = false;
        if (LOOK && (look & 1)) {
            Snapshot<MR * MC + MR> before;
            bool recurs = false;
#pragma unroll 1
            while (!wide && !recurs && it + CHECK <= run_end) {
#pragma unroll
                for (int a = 0; a < MR; ++a) before.take(a * MC, V[a]);
                before.take(MR * MC, rs);
#pragma unroll 1
                for (int u = 0; u < CHECK; ++u) dykstra_step<G, PACK>(V, rs, Pc, last, Nf, iN);
                it += CHECK;
                unsigned differ = before.differ(MR * MC, rs);
#pragma unroll
                for (int a = 0; a < MR; ++a) differ |= before.differ(a * MC, V[a]);
                wide = out_of_range();
                recurs = !wide && __all_sync(FULL, differ == 0u);
            }
            if (recurs) run_end = it + (iters - it) % CHECK;
            if (!wide) {
#pragma unroll 1
                for (; it < run_end; ++it) dykstra_step<G, PACK>(V, rs, Pc, last, Nf, iN);
            }
            if (recurs) break;
            look += 2;
            if (wide || look > 2 * LOOKS || iters - it < WORTH_LOOKING) look &= ~1;
            continue;
        }
#pragma unroll 1
        while (!wide && it + CHECK <= run_end) {
            // Two iterations of code where many warps share the instruction cache with other warps' rounding
            // (four: 5 to 15 % slower on matrices that converge), four where few do (two: 4 % slower) or an iteration
            // is short (65536 x 4 2:4: 30.8 us, 33.0 with two).  The stopping test at M = 32 is mostly code that runs once.
#pragma unroll(EE && G::M == 32 ? 1 : (EE || G::V != 0 || G::M == 4) ? CHECK : 2)
            for (int u = 0; u < CHECK - (EE ? 1 : 0); ++u) dykstra_step<G, PACK>(V, rs, Pc, last, Nf, iN);
            if constexpr (EE) {
                const float delta = dykstra_step<G, PACK, true>(V, rs, Pc, last, Nf, iN);
                if (__all_sync(FULL, delta < ee_eps)) {   // every block of the warp has converged
                    it += CHECK;
                    iters = it;
                    wide = true;                          // skips the remainder loop as well
                    break;
                }
            }
            it += CHECK;
            wide = out_of_range();
        }
        if (!wide) {   // fewer than CHECK iterations left
#pragma unroll
            for (int k = 0; k < CO; ++k) last[k] = 2.0f;  // (no value of the loop above has to be kept)
#pragma unroll 1
            for (; it < run_end; ++it) dykstra_step<G, PACK, false, LOOK>(V, rs, Pc, last, Nf, iN);
            if constexpr (LOOK) {
                float off = 0.0f;                         // (fmaxf drops NaN)
#pragma unroll
                for (int k = 0; k < CO; ++k) off = fmaxf(off, fabsf(last[k] - 1.0f));
                if (look < 2 * LOOKS && iters - it >= WORTH_LOOKING && __all_sync(FULL, off <= NEAR_ONE)) look |= 1;
            }
        }
    }
    // final potentials and t = t0 + F + G
#pragma unroll
    for (int k = 0; k < RO; ++k) F[k] = add_potential<true>(fpot + k * 32, rs[k], SIGN);
#pragma unroll
    for (int k = 0; k < CO; ++k) Gc[k] = add_potential<true>(gpot + k * 32, Pc[k]);
    all_gather<MR, PC>(F, 1);
    all_gather<MC, PR>(Gc, PC);
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int e = 4 * q;
        const float4 v = st4[q * 32];
        t[e / MC][e % MC] = (v.x + F[e / MC]) + Gc[e % MC];
        t[(e + 1) / MC][(e + 1) % MC] = (v.y + F[(e + 1) / MC]) + Gc[(e + 1) % MC];
        t[(e + 2) / MC][(e + 2) % MC] = (v.z + F[(e + 2) / MC]) + Gc[(e + 2) % MC];
        t[(e + 3) / MC][(e + 3) % MC] = (v.w + F[(e + 3) / MC]) + Gc[(e + 3) % MC];
    }
    return iters;
}

// ---------------------------------------------------------------------------
// Score source: the matrix the solver works on, described rather than
// materialised (Section 4: magnitude, ADMM D-update, SparseGPT group, Wanda).
// One fp32 rounding per operation, no fused multiply-add.
// ---------------------------------------------------------------------------
enum : int { SC_ABS = 0, SC_ADMM = 1, SC_COLDIV = 2, SC_COLMUL = 3 };

struct ScoreSrc {
    int kind, w_is_bf16;
    const void* w; int64_t ld;
    const float* v; int64_t ld_v;
    float scalar;
    const float* colvec;
    int vec_w, vec_v, vec_c;       // 16-byte (8-byte for bf16) vector loads allowed
};

__device__ __forceinline__ float score_of(int kind, float w, float v, float scalar, float cv) {
    switch (kind) {
        case SC_ADMM: { const float s = __fadd_rn(w, __fmul_rn(v, scalar)); return __fmul_rn(s, s); }
        case SC_COLDIV: return fabsf(__fdiv_rn(w, cv));
        case SC_COLMUL: return __fmul_rn(fabsf(w), cv);
        default: return fabsf(w);
    }
}

__device__ __forceinline__ float4 widen_bf16(unsigned lo, unsigned hi) {
    return make_float4(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u),
                       __uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
}
__device__ __forceinline__ float4 load_float_quad(const float* p, bool vec) {
    return vec ? __ldg(reinterpret_cast<const float4*>(p))
               : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
}
// Weights of the four consecutive elements (r, c .. c+3); c is a multiple of 4.
__device__ __forceinline__ float4 load_weight_quad(const ScoreSrc& S, int64_t r, int64_t c) {
    if (!S.w_is_bf16) return load_float_quad(static_cast<const float*>(S.w) + r * S.ld + c, S.vec_w != 0);
    const unsigned short* p = static_cast<const unsigned short*>(S.w) + r * S.ld + c;
    if (S.vec_w) {
        const uint2 q = __ldg(reinterpret_cast<const uint2*>(p));
        return widen_bf16(q.x, q.y);
    }
    return widen_bf16(__ldg(p) | ((unsigned)__ldg(p + 1) << 16), __ldg(p + 2) | ((unsigned)__ldg(p + 3) << 16));
}
// Entries c .. c+3 of the column vector (ones for the kinds without one).
__device__ __forceinline__ float4 load_colvec_quad(const ScoreSrc& S, int64_t c) {
    return (S.kind >= SC_COLDIV) ? load_float_quad(S.colvec + c, S.vec_c != 0) : make_float4(1.f, 1.f, 1.f, 1.f);
}
__device__ __forceinline__ float4 score_quad(const ScoreSrc& S, const float4& w, const float4& v, const float4& cv) {
    return make_float4(score_of(S.kind, w.x, v.x, S.scalar, cv.x), score_of(S.kind, w.y, v.y, S.scalar, cv.y),
                       score_of(S.kind, w.z, v.z, S.scalar, cv.z), score_of(S.kind, w.w, v.w, S.scalar, cv.w));
}
// Scores of the four consecutive elements (r, c .. c+3).  One branch picks the second operand: with two
// the scans of large ADMM and SparseGPT sources take up to a tenth longer.
__device__ __forceinline__ float4 load_score_quad(const ScoreSrc& S, int64_t r, int64_t c) {
    const float4 w = load_weight_quad(S, r, c);
    if (S.kind == SC_ABS) return make_float4(fabsf(w.x), fabsf(w.y), fabsf(w.z), fabsf(w.w));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f), cv = make_float4(1.f, 1.f, 1.f, 1.f);
    if (S.kind == SC_ADMM) v = load_float_quad(S.v + r * S.ld_v + c, S.vec_v != 0);
    else cv = load_float_quad(S.colvec + c, S.vec_c != 0);
    return score_quad(S, w, v, cv);
}
// The same with the column vector's entries in hand.
__device__ __forceinline__ float4 load_score_quad(const ScoreSrc& S, int64_t r, int64_t c, const float4& cv) {
    const float4 w = load_weight_quad(S, r, c);
    if (S.kind == SC_ABS) return make_float4(fabsf(w.x), fabsf(w.y), fabsf(w.z), fabsf(w.w));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (S.kind == SC_ADMM) v = load_float_quad(S.v + r * S.ld_v + c, S.vec_v != 0);
    return score_quad(S, w, v, cv);
}

__device__ __forceinline__ int any_nan(const float4& v) {
    return !(v.x == v.x) | !(v.y == v.y) | !(v.z == v.z) | !(v.w == v.w);
}
// ---------------------------------------------------------------------------
// Where a unit's blocks live in the matrix.  The blocks of the matrix are numbered
// row by row, every block row padded to a whole number of mask words (`nbp` slots of
// which `nbc` hold blocks; a single block column, as in the column groups of
// SparseGPT, is not padded), and a unit is BPW consecutive slots: it runs on into the
// next block row where one ends, so ragged widths and slabs fill their warps too.  In
// shared memory slot b of the unit occupies columns [b M, b M + M).
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t div_slots(int64_t a, int64_t b) {   // 0 <= a, 0 < b
    return (((uint64_t)a | (uint64_t)b) >> 32) ? a / b : (int64_t)((unsigned)a / (unsigned)b);
}
// Volatile: read again where it is needed, so that no position in the matrix stays in registers
// over the iterations.
__device__ __forceinline__ int64_t this_cta() {
    unsigned u;
    asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(u));
    return u;
}
template <int WPC> __device__ __forceinline__ int64_t this_unit() {
    return this_cta() * WPC + threadIdx.x / 32;
}
template <int M> struct UnitMap {
    int64_t rows, cols;    // extent of the matrix
    int64_t nbc, nbp;      // blocks per block row, and slots
    int64_t bi0, bj0;      // block row and slot of the unit's first slot
    __device__ __forceinline__ UnitMap(int64_t rows_, int64_t cols_, int64_t nbp_, int64_t first)
        : rows(rows_), cols(cols_), nbc(cols_ / M), nbp(nbp_) {
        bi0 = div_slots(first, nbp_);
        bj0 = first - bi0 * nbp_;
    }
    // Origin of slot b of the unit; false if there is no such block.
    __device__ __forceinline__ bool locate(int b, int64_t& r0, int64_t& c0) const {
        int64_t bi = bi0, bj = bj0 + b;
        if (bj >= nbp) {                     // the unit ran on into a later block row
            const int64_t q = div_slots(bj, nbp);
            bi += q;
            bj -= q * nbp;
        }
        r0 = bi * M;
        c0 = bj * M;
        return r0 < rows && bj < nbc;
    }
    __device__ __forceinline__ bool holds_quad(int64_t r, int64_t c) const {
        return r >= 0 && r < rows && c >= 0 && c + 4 <= cols;
    }
};

// ---------------------------------------------------------------------------
// Unit loaders: COLS columns (from slot `slot0` on) of the unit's M rows into shared memory
// (dst: row stride WS), coalesced, vector loads when the addresses allow it.  A lane keeps its
// column(s) and walks down the rows, BATCH of them in flight: the position, and the entries of the
// column vector, are worked out once.  Aligned sources have loops of their own with many
// loads in flight; the others share one that is unrolled less, because the instruction cache is
// what the warps of an SM, spread over all phases of the kernel, compete for.  Return non-zero if
// this lane saw a non-finite score, respectively a NaN key.
// ---------------------------------------------------------------------------
template <class G, int COLS, int BATCH, class Column, class Load>
__device__ __forceinline__ void load_unit(const UnitMap<G::M>& um, int slot0, int lane, float* __restrict__ dst,
                                          Column column, Load load) {
    constexpr int M = G::M;
    constexpr int QW = (COLS / 4 < 32) ? COLS / 4 : 32;     // quads of a row that the warp takes at once
    constexpr int RPI = 32 / QW, STEPS = M / RPI;           // rows it takes at once
    constexpr int B = (BATCH < STEPS) ? BATCH : STEPS;
    static_assert(M % RPI == 0 && STEPS % B == 0, "whole batches");
#pragma unroll 1
    for (int cs = 0; cs < COLS / (4 * QW); ++cs) {
        const int c = (lane % QW + cs * QW) * 4;
        int64_t r0, c0;
        const bool there = um.locate(slot0 + c / M, r0, c0);
        r0 += lane / QW;
        c0 += c % M;
        float* d = dst + (lane / QW) * G::WS + c;
        if (there) column(c0);
#pragma unroll 1
        for (int i0 = 0; i0 < STEPS; i0 += B, r0 += B * RPI, d += B * RPI * G::WS) {
            float4 v[B];
#pragma unroll
            for (int i = 0; i < B; ++i) {
                v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (there && TS_CHECK(um.holds_quad(r0 + i * RPI, c0))) v[i] = load(r0 + i * RPI, c0);
            }
#pragma unroll
            for (int i = 0; i < B; ++i) {
                if (!TS_CHECK(lane / QW + (i0 + i) * RPI < M && c + 4 <= G::UW)) continue;
                float* const e = d + i * RPI * G::WS;
                e[0] = v[i].x; e[1] = v[i].y; e[2] = v[i].z; e[3] = v[i].w;
            }
        }
    }
}
template <class G, int COLS>
__device__ __forceinline__ int load_scores(const ScoreSrc& S, const UnitMap<G::M>& um, int slot0, int lane,
                                           float* __restrict__ dst) {
    float nan = 0.0f;     // 0 x is a NaN for a non-finite x
    const auto seen = [&](const float4& v) {
        nan = fmaf(v.x, 0.0f, fmaf(v.y, 0.0f, fmaf(v.z, 0.0f, fmaf(v.w, 0.0f, nan))));
        return v;
    };
    float4 cv = make_float4(1.f, 1.f, 1.f, 1.f);
    const auto no_column = [](int64_t) {};
    const auto column = [&](int64_t c) { cv = load_colvec_quad(S, c); };
    const auto scaled = [&](const float4& v) {      // |w| 1 is |w|
        return seen(make_float4(__fmul_rn(fabsf(v.x), cv.x), __fmul_rn(fabsf(v.y), cv.y),
                                __fmul_rn(fabsf(v.z), cv.z), __fmul_rn(fabsf(v.w), cv.w)));
    };
    const float* const w32 = static_cast<const float*>(S.w);
    const unsigned short* const w16 = static_cast<const unsigned short*>(S.w);
    if (S.kind == SC_ABS && !S.w_is_bf16 && S.vec_w) {
        load_unit<G, COLS, 8>(um, slot0, lane, dst, no_column, [&](int64_t r, int64_t c) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(w32 + r * S.ld + c));
            return seen(make_float4(fabsf(v.x), fabsf(v.y), fabsf(v.z), fabsf(v.w)));
        });
    } else if ((S.kind == SC_ABS || S.kind == SC_COLMUL) && S.vec_w && S.w_is_bf16) {
        load_unit<G, COLS, 8>(um, slot0, lane, dst, column, [&](int64_t r, int64_t c) {
            const uint2 q = __ldg(reinterpret_cast<const uint2*>(w16 + r * S.ld + c));
            return scaled(widen_bf16(q.x, q.y));
        });
    } else if (S.kind == SC_COLMUL && S.vec_w) {
        load_unit<G, COLS, 4>(um, slot0, lane, dst, column, [&](int64_t r, int64_t c) {
            return scaled(__ldg(reinterpret_cast<const float4*>(w32 + r * S.ld + c)));
        });
    } else if (S.kind == SC_ADMM && S.vec_w && S.vec_v && !S.w_is_bf16) {
        load_unit<G, COLS, 4>(um, slot0, lane, dst, no_column, [&](int64_t r, int64_t c) {
            const float4 w = __ldg(reinterpret_cast<const float4*>(w32 + r * S.ld + c));
            const float4 v = __ldg(reinterpret_cast<const float4*>(S.v + r * S.ld_v + c));
            return seen(make_float4(score_of(SC_ADMM, w.x, v.x, S.scalar, 1.f), score_of(SC_ADMM, w.y, v.y, S.scalar, 1.f),
                                    score_of(SC_ADMM, w.z, v.z, S.scalar, 1.f), score_of(SC_ADMM, w.w, v.w, S.scalar, 1.f)));
        });
    } else if (S.kind == SC_COLDIV && S.vec_w && !S.w_is_bf16) {
        load_unit<G, COLS, 4>(um, slot0, lane, dst, column, [&](int64_t r, int64_t c) {
            const float4 w = __ldg(reinterpret_cast<const float4*>(w32 + r * S.ld + c));
            return seen(make_float4(fabsf(__fdiv_rn(w.x, cv.x)), fabsf(__fdiv_rn(w.y, cv.y)),
                                    fabsf(__fdiv_rn(w.z, cv.z)), fabsf(__fdiv_rn(w.w, cv.w))));
        });
    } else {
        load_unit<G, COLS, 2>(um, slot0, lane, dst, column,
                              [&](int64_t r, int64_t c) { return seen(load_score_quad(S, r, c, cv)); });
    }
    return nan != 0.0f;
}
// |w| in fp32 at any alignment (rounding alone has no other source).
template <class G>
__device__ __forceinline__ int load_plain_scores(const ScoreSrc& S, const UnitMap<G::M>& um, int lane,
                                                 float* __restrict__ dst) {
    float nan = 0.0f;
    load_unit<G, G::UW, 4>(um, 0, lane, dst, [](int64_t) {}, [&](int64_t r, int64_t c) {
        const float4 v = load_float_quad(static_cast<const float*>(S.w) + r * S.ld + c, S.vec_w != 0);
        nan = fmaf(v.x, 0.0f, fmaf(v.y, 0.0f, fmaf(v.z, 0.0f, fmaf(v.w, 0.0f, nan))));
        return make_float4(fabsf(v.x), fabsf(v.y), fabsf(v.z), fabsf(v.w));
    });
    return nan != 0.0f;
}
// The aligned |scores| and keys of a unit together (rounding alone): one wait for memory, not two.
template <class G>
__device__ __forceinline__ int load_scores_and_keys(const ScoreSrc& S, const float* __restrict__ keys, int64_t ld,
                                                    const UnitMap<G::M>& um, int lane, float* __restrict__ w,
                                                    float* __restrict__ k) {
    constexpr int M = G::M, QW = (G::UW / 4 < 32) ? G::UW / 4 : 32, RPI = 32 / QW, STEPS = M / RPI;
    constexpr int B = (STEPS < 4) ? STEPS : 4;
    static_assert(M % RPI == 0 && STEPS % B == 0, "whole batches");
    int bad = 0;
    float nan = 0.0f;     // 0 x is a NaN for a non-finite x
#pragma unroll 1
    for (int cs = 0; cs < G::UW / (4 * QW); ++cs) {
        const int c = (lane % QW + cs * QW) * 4;
        int64_t r0, c0;
        const bool there = um.locate(c / M, r0, c0);
        c0 += c % M;
#pragma unroll 1
        for (int i0 = lane / QW; i0 < M; i0 += B * RPI) {
            float4 a[B], b[B];
#pragma unroll
            for (int i = 0; i < B; ++i) {
                const int64_t r = r0 + i0 + i * RPI;
                a[i] = b[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (there && TS_CHECK(um.holds_quad(r, c0))) {
                    a[i] = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(S.w) + r * S.ld + c0));
                    b[i] = __ldg(reinterpret_cast<const float4*>(keys + r * ld + c0));
                }
            }
#pragma unroll
            for (int i = 0; i < B; ++i) {
                nan = fmaf(a[i].x, 0.0f, fmaf(a[i].y, 0.0f, fmaf(a[i].z, 0.0f, fmaf(a[i].w, 0.0f, nan))));
                bad |= any_nan(b[i]);
                if (!TS_CHECK(i0 + i * RPI < M && c + 4 <= G::UW)) continue;
                float* const e = w + (i0 + i * RPI) * G::WS + c;
                float* const f = k + (i0 + i * RPI) * G::WS + c;
                e[0] = fabsf(a[i].x); e[1] = fabsf(a[i].y); e[2] = fabsf(a[i].z); e[3] = fabsf(a[i].w);
                f[0] = b[i].x; f[1] = b[i].y; f[2] = b[i].z; f[3] = b[i].w;
            }
        }
    }
    return bad | (nan != 0.0f);
}
template <class G>
__device__ __forceinline__ int load_keys(const float* __restrict__ src, int64_t ld, const UnitMap<G::M>& um,
                                         bool vec_ok, int lane, float* __restrict__ dst) {
    int bad = 0;
    load_unit<G, G::UW, 4>(um, 0, lane, dst, [](int64_t) {}, [&](int64_t r, int64_t c) {
        const float4 v = load_float_quad(src + r * ld + c, vec_ok);
        bad |= any_nan(v);          // infinite keys have a place in the order; NaN keys are flagged
        return v;
    });
    return bad;
}

// ---------------------------------------------------------------------------
// Rounding stage (Algorithm 2).  A group of M lanes owns one block; lane i of
// the group plays row i and column i at once.
// ---------------------------------------------------------------------------
// Tables of the rounding stage: for every line (row or column) of a block the
// M prefix sets of its sorted order, prefix p = bit mask of the positions of its
// p+1 best entries (uint32 words for M = 32, uint16 otherwise).  Each lane only
// ever reads the two tables of its own row and column.  The row tables (and for
// M <= 16 the column tables too) are written over the block's own key cells once
// both sorts have consumed the keys: key row i (M floats = 4M bytes) becomes
//   M = 32 :  [0,4M) row prefixes of row i          (column prefixes: SmemLayout::cpre)
//   M <= 16:  [0,2M) row prefixes of row i, [2M,4M) column prefixes of column i
constexpr int CPRE_STRIDE = 33;   // words per column-prefix table at M = 32 (odd: conflict-free)

// The strict order "key descending, index ascending": ascending words of the key; NaN orders as
// -inf, -0 as +0.
__device__ __forceinline__ unsigned order_word(float key) {
    if (!(key == key)) key = __int_as_float(0xff800000);
    key += 0.0f;
    const unsigned u = __float_as_uint(key);
    return (u & 0x80000000u) ? u : ~(u | 0x80000000u);
}

// That order packed into one ascending 32-bit word: order_word with its five low bits replaced by
// the index.  Dropping those bits is harmless unless two keys of the line agree in the 27 bits kept
// ("same bucket"): the network then leaves them side by side in index order, and sort_line puts
// them right by their full keys.  Keys that are exactly zero (the capped entries of a plan: up to
// half of a line) are the one common case of equal keys; each of them gets a bucket of its own,
// ZERO_BUCKET + index (zeros order among themselves by index), and the positive keys are shifted
// down by the 32 buckets this takes.
constexpr unsigned ZERO_BUCKET = 0x03ffffe0u;
__device__ __forceinline__ unsigned sort_word_packed(float key, unsigned idx) {
    if (!(key == key)) key = __int_as_float(0xff800000);
    key += 0.0f;
    const unsigned b = __float_as_uint(key);
    unsigned hi;
    if (b & 0x80000000u) hi = b;                               // negative: larger magnitude later
    else if (b == 0u) hi = (ZERO_BUCKET + idx) << 5;
    else hi = 0x7fffffffu - b - (32u * 32u + 31u);             // positive: larger first, all before the zeros
    return (hi & ~31u) | idx;
}
// The same word for a key that is known to be <= 0 and not NaN (every entry of a capped log-plan).
__device__ __forceinline__ unsigned sort_word_capped(float key, unsigned idx) {
    const unsigned hi = (key == 0.0f) ? (ZERO_BUCKET + idx) << 5 : __float_as_uint(key);
    return (hi & ~31u) | idx;
}

// Batcher's odd-even merge sort as a fully unrolled network (191 compare-exchanges for 32
// keys, 63 for 16, 19 for 8, 5 for 4), ascending.  Indices are template constants so that the
// keys stay in registers.  A compare-exchange is a min and a max.
template <int I, int J, int M> __device__ __forceinline__ void cmp_swap(unsigned (&v)[M]) {
    const unsigned a = v[I], b = v[J];
    v[I] = min(a, b);
    v[J] = max(a, b);
}
template <int LO, int N, int R, int I, int M> __device__ __forceinline__ void oem_chain(unsigned (&v)[M]) {
    if constexpr (I + R < LO + N) {
        cmp_swap<I, I + R, M>(v);
        oem_chain<LO, N, R, I + 2 * R, M>(v);
    }
}
// merges the two sorted halves of the subsequence LO, LO+R, LO+2R, ... of v[LO .. LO+N)
template <int LO, int N, int R, int M> __device__ __forceinline__ void oem_merge(unsigned (&v)[M]) {
    if constexpr (2 * R < N) {
        oem_merge<LO, N, 2 * R, M>(v);
        oem_merge<LO + R, N, 2 * R, M>(v);
        oem_chain<LO, N, R, LO + R, M>(v);
    } else {
        cmp_swap<LO, LO + R, M>(v);
    }
}
template <int LO, int N, int M> __device__ __forceinline__ void oem_sort(unsigned (&v)[M]) {
    if constexpr (N > 1) {
        oem_sort<LO, N / 2, M>(v);
        oem_sort<LO + N / 2, N / 2, M>(v);
        oem_merge<LO, N, 1, M>(v);
    }
}

// Sorts one line, given its keys in registers and its place in shared memory (stride `st`
// floats): on return the low five bits of w[p] are the position of the p-th best entry.
// capped: the keys are known to be <= 0 and not NaN.
template <int M>
__device__ __forceinline__ void sort_line(const float (&key)[M], const float* line, int st, bool capped,
                                          unsigned (&w)[M]) {
    if (capped) {
#pragma unroll
        for (int k = 0; k < M; ++k) w[k] = sort_word_capped(key[k], k);
    } else {
#pragma unroll
        for (int k = 0; k < M; ++k) w[k] = sort_word_packed(key[k], k);
    }
    oem_sort<0, M, M>(w);
    unsigned closest = 0xffffffffu;     // smallest difference pattern of two neighbours
#pragma unroll
    for (int p = 0; p + 1 < M; ++p) closest = min(closest, w[p] ^ w[p + 1]);
    // Rare: two non-zero keys of a line within 2^-18 of each other.  Passes of neighbour exchanges
    // among the entries of a bucket, by full key, until nothing moves: a bucket of L entries is
    // in order after at most L - 1 of them (entries of different buckets, and equal keys, stay as
    // they are).  A sixth of the code of a second network on 64-bit words, and a fifth of its time.
    bool more = closest < 32u;
#pragma unroll 1
    for (int pass = 0; pass < M && __any_sync(FULL, more); ++pass) {
        bool moved = false;
#pragma unroll
        for (int p = 0; p + 1 < M; ++p) {
            if (more && (w[p] ^ w[p + 1]) < 32u) {
                const unsigned a = w[p], b = w[p + 1];
                if (order_word(line[(b & 31u) * st]) < order_word(line[(a & 31u) * st])) {
                    w[p] = b;
                    w[p + 1] = a;
                    moved = true;
                }
            }
        }
        more = moved;
    }
}
// Prefix sets of a sorted line, for M <= 16 two to a word: pre[p] = positions of the p+1 best.
template <int M> __device__ __forceinline__ void prefix_sets(const unsigned (&w)[M], unsigned (&pre)[M / 2]) {
    unsigned acc = 0u;
#pragma unroll
    for (int p = 0; p < M; ++p) {
        acc |= 1u << (w[p] & 31u);
        if (p % 2 == 0) pre[p / 2] = acc;
        else pre[p / 2] |= acc << 16;
    }
}

// Prefix p of a stored table (tab points to the table's first byte).
template <int M> __device__ __forceinline__ unsigned prefix_at(const void* tab, int p) {
    if (!TS_CHECK(p >= 0 && p < M)) return 0u;
    if (M == 32) return static_cast<const unsigned*>(tab)[p];
    return static_cast<const unsigned short*>(tab)[p];
}

// The first `cap` entries of `avail` (a set of positions of one line) in the line's sorted
// order, or all of them if there are no more than `cap`: binary search for the shortest
// prefix of the order that holds `cap` available entries.  For the lane's row and its column at
// once and without branches: the two searches are chains of dependent shared-memory reads, and a
// round of the greedy selection waits for them.
template <int M>
__device__ __forceinline__ void first_available(unsigned& setR, int capR, const void* tabR, unsigned& setC, int capC,
                                                const void* tabC) {
    int p = 0, q = 0;
#pragma unroll
    for (int b = M / 2; b > 0; b >>= 1) {
        const unsigned r = prefix_at<M>(tabR, p + b - 1), c = prefix_at<M>(tabC, q + b - 1);
        p += (__popc(setR & r) < capR) ? b : 0;
        q += (__popc(setC & c) < capC) ? b : 0;
    }
    const unsigned r = prefix_at<M>(tabR, p), c = prefix_at<M>(tabC, q);
    setR &= (__popc(setR) <= capR) ? 0xffffffffu : r;
    setC &= (__popc(setC) <= capC) ? 0xffffffffu : c;
}

// Transpose of the M x M bit matrix whose row i is held by lane i of a group of M lanes
// (bit j of x = element (i, j)): recursive exchange of the off-diagonal blocks.
template <int M> __device__ __forceinline__ unsigned transpose_bits(unsigned x, int i) {
#pragma unroll
    for (int s = M / 2; s > 0; s >>= 1) {
        // positions whose bit s is clear
        const unsigned lo = (s == 16) ? 0x0000ffffu : (s == 8) ? 0x00ff00ffu : (s == 4) ? 0x0f0f0f0fu
                          : (s == 2) ? 0x33333333u : 0x55555555u;
        const unsigned y = __shfl_xor_sync(FULL, x, s);
        const bool up = (i & s) != 0;
        const unsigned keep = up ? ~lo : lo;
        const unsigned z = up ? (y >> s) : (y << s);
        x = (x & keep) | (z & ~keep);
    }
    return x;
}

// Greedy selection + local search for the block of this lane's group.
//   ks, ws: shared-memory pointers to element (0,0) of the block's keys and
//   |scores| (row stride WS); the key cells are overwritten.  cpre: this
//   lane's column-prefix table when it does not fit in the key cells (M = 32).
//   active: group has a block.  capped: the keys are known to be <= 0.  before_search: called
//   by the whole warp, once the tables are done with, if ws is going to be read.
// Returns this lane's row of the mask (M bits).  flags accumulates DEV_* bits.
template <class G, class BeforeSearch>
__device__ __forceinline__ unsigned round_block(float* ks, const float* ws, unsigned* cpre, int lane, bool active,
                                                bool capped, int N, int ls_steps, int& flags,
                                                BeforeSearch before_search) {
    constexpr int M = G::M;
    constexpr int WS = G::WS;
    constexpr unsigned GM = (M == 32) ? 0xffffffffu : ((1u << (M & 31)) - 1u);
    const int i = lane % M;            // my row, and my column
    const int gsh = (lane / M) * M;    // first lane of my group

    // ---- sorted orders of my row and of my column (Algorithm 2 line 2), kept as prefix sets
    unsigned char* const rtab = reinterpret_cast<unsigned char*>(ks + i * WS);
    unsigned char* const ctab = (M == 32) ? reinterpret_cast<unsigned char*>(cpre) : rtab + 2 * M;
    if constexpr (M == 32) {
        // One sort body for both sides: the network is some 900 instructions long and the warps of an
        // SM are spread over the whole kernel, so what counts is that its code stays in the cache.
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            float key[M];
            unsigned w[M];
            if (side == 0) {
#pragma unroll
                for (int k = 0; k < M; ++k) key[k] = ks[k * WS + i];
            } else {
#pragma unroll
                for (int k = 0; k < M; ++k) key[k] = ks[i * WS + k];
            }
            sort_line<M>(key, side ? ks + i * WS : ks + i, side ? 1 : WS, capped, w);
            __syncwarp();                   // side 1: every lane is done reading keys
            unsigned* const tab = reinterpret_cast<unsigned*>(side ? rtab : ctab);
            unsigned acc = 0u;
#pragma unroll
            for (int p = 0; p < M; ++p) {
                acc |= 1u << (w[p] & 31u);
                tab[p] = acc;
            }
        }
    } else {
        unsigned pc[M / 2], pr[M / 2];
        {
            float key[M];
            unsigned w[M];
#pragma unroll
            for (int k = 0; k < M; ++k) key[k] = ks[k * WS + i];
            sort_line<M>(key, ks + i, WS, capped, w);
            prefix_sets<M>(w, pc);
#pragma unroll
            for (int k = 0; k < M; ++k) key[k] = ks[i * WS + k];
            sort_line<M>(key, ks + i * WS, 1, capped, w);
            prefix_sets<M>(w, pr);
        }
        __syncwarp();                       // every lane is done reading keys
#pragma unroll
        for (int w = 0; w < M / 2; ++w) {
            reinterpret_cast<unsigned*>(rtab)[w] = pr[w];
            reinterpret_cast<unsigned*>(ctab)[w] = pc[w];
        }
    }
    __syncwarp();

    // ---- greedy selection (lines 3-6) in synchronous rounds.  An available
    // entry (not taken, row and column not full) that is among the first
    // capR available entries of its row and the first capC of its column
    // (cap = remaining capacity) is taken by the sequential scan whatever
    // happens elsewhere, so all such entries are taken at once; the first
    // available entry in the global order always qualifies, hence every round
    // makes progress and the fixed point is the sequential result.  availR:
    // available columns of my row; availC: available rows of my column.
    unsigned availR = active ? GM : 0u, availC = availR;
    int capR = active ? N : 0, capC = capR;
    unsigned sel = 0u, selC = 0u;
    for (int round = 0; round < M * M; ++round) {
        if (!__any_sync(FULL, availR != 0u)) break;
        if (round == M * M - 1) flags |= DEV_INTERNAL;
        unsigned pickR = availR, pickC = availC;
        first_available<M>(pickR, capR, rtab, pickC, capC, ctab);
        // an entry picked from both sides is taken: takenR columns in my row, takenC rows in my
        // column.  (Both picks are transposed, not takenR a second time: two chains of five
        // exchanges side by side, or one for M <= 16, where both fit into one word.)
        unsigned takenR, takenC;
        if (M == 32) {
            takenR = pickR & transpose_bits<M>(pickC, i);
            takenC = pickC & transpose_bits<M>(pickR, i);
        } else {
            const unsigned tt = transpose_bits<M>(pickC | (pickR << 16), i);
            takenR = pickR & tt;
            takenC = pickC & (tt >> 16);
        }
        sel |= takenR;
        selC |= takenC;
        capR -= __popc(takenR);
        capC -= __popc(takenC);
        // lines that just filled up drop out, and so do their entries
        const unsigned fullR = (__ballot_sync(FULL, capR == 0) >> gsh) & GM;
        const unsigned fullC = (__ballot_sync(FULL, capC == 0) >> gsh) & GM;
        availR = (capR == 0) ? 0u : (availR & ~takenR & ~fullC);
        availC = (capC == 0) ? 0u : (availC & ~takenC & ~fullR);
    }

    // ---- local search (lines 7-13, Eq. 6).  sel: my row of the mask (bits over columns);
    // selC: my column (bits over rows).  Lane j' scans the rows i' that can form a valid
    // triple with it: S[i'][j'] = 1 and S[i'][j] = 0, provided S[i][j'] = 0.
    if (ls_steps != 0 && __any_sync(FULL, capR > 0)) before_search();
    bool stopped = !active;
    int steps = 0;
    for (int it = 0; it <= M * N; ++it) {
        const unsigned rdef = (__ballot_sync(FULL, capR > 0) >> gsh) & GM;
        const unsigned cdef = (__ballot_sync(FULL, capC > 0) >> gsh) & GM;
        const bool work = !stopped && rdef != 0u && cdef != 0u && (ls_steps < 0 || steps < ls_steps);
        if (!__any_sync(FULL, work)) break;
        if (it == M * N) { flags |= DEV_INTERNAL; break; }
        const int di = work ? __ffs(rdef) - 1 : 0;   // lowest unsaturated row
        const int dj = work ? __ffs(cdef) - 1 : 0;   // lowest unsaturated column
        const int jp = i;                            // my candidate column j'
        const bool lines_ok = TS_CHECK(di >= 0 && di < M && dj >= 0 && dj < M);
        const unsigned col_dj = __shfl_sync(FULL, selC, lines_ok ? dj : 0, M);   // rows that hold column j
        unsigned cand = (work && lines_ok && !((selC >> di) & 1u)) ? (selC & ~col_dj & GM) : 0u;
        float best = __int_as_float(0xff800000);
        int bi = 0x7fffffff;
        const float w_ijp = lines_ok ? ws[di * WS + jp] : 0.0f;
        // Ascending i': ties keep the smallest.  Four candidates a turn, so that their scores are read
        // together: one at a time, the chain of reads was most of a step.  (A column of a 4 x 4 block
        // has one or two: rounding |W| at 4096 x 4096 takes 115 us with four, 111 with two.)
        constexpr int TURN = (M == 4) ? 2 : 4;
        while (cand) {
            int ip[TURN];
            float sc[TURN];
            bool is[TURN];
#pragma unroll
            for (int k = 0; k < TURN; ++k) {
                is[k] = cand != 0u;
                ip[k] = is[k] ? __ffs(cand) - 1 : 0;
                cand &= cand - 1u;                   // 0 stays 0
                is[k] = is[k] && TS_CHECK(ip[k] < M);
                sc[k] = is[k] ? __fsub_rn(__fadd_rn(w_ijp, ws[ip[k] * WS + dj]), ws[ip[k] * WS + jp]) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < TURN; ++k)
                if (is[k] && sc[k] > best) { best = sc[k]; bi = ip[k]; }
        }
        int bflat = (bi == 0x7fffffff) ? 0x7fffffff : bi * M + jp;
        if constexpr (M == 32) {     // the largest score of the warp, then the smallest index that has it
            const unsigned u = __float_as_uint(best + 0.0f);                      // -0 -> +0
            const unsigned mine = (u & 0x80000000u) ? ~u : (u | 0x80000000u);     // ascending
            const unsigned top = __reduce_max_sync(FULL, mine);
            bflat = (int)__reduce_min_sync(FULL, (mine == top) ? (unsigned)bflat : 0x7fffffffu);
            best = __uint_as_float((top & 0x80000000u) ? top & 0x7fffffffu : ~top);
        } else {
#pragma unroll
            for (int off = M / 2; off > 0; off >>= 1) {
                const float ob = __shfl_xor_sync(FULL, best, off, M);
                const int of = __shfl_xor_sync(FULL, bflat, off, M);
                if (ob > best || (ob == best && of < bflat)) { best = ob; bflat = of; }
            }
        }
        if (work) {
            if (bflat == 0x7fffffff) {            // no valid triple: only with non-finite scores
                stopped = true;
            } else if (ls_steps >= 0 && !(best > 0.0f)) {
                stopped = true;                   // paper-strict loop: improving swaps only
            } else if (!TS_CHECK(bflat >= 0 && bflat < M * M)) {
                stopped = true;
            } else {
                const int ip = bflat / M, jq = bflat % M;
                if (i == ip) sel = (sel & ~(1u << jq)) | (1u << dj);
                if (i == di) { sel |= 1u << jq; --capR; }
                if (i == jq) selC = (selC & ~(1u << ip)) | (1u << di);
                if (i == dj) { selC |= 1u << ip; --capC; }
                ++steps;
            }
        }
    }
    if (active && (capR != 0 || capC != 0)) flags |= DEV_UNDERFILLED;
    return sel;
}

// The mask rows of the (up to) 32 / M blocks a warp has just rounded: lane i of group grp holds
// row i of the block at (r0, c0).  In a slab every block's rows have words of their own; else the
// blocks share the words of their M rows.
template <int M>
__device__ __forceinline__ void write_mask_rows(uint32_t* bits, int64_t wpr, int64_t rows, int64_t nbp, int64_t r0,
                                                int64_t c0, int lane, bool active, unsigned sel) {
    const int grp = lane / M, i = lane % M;
    if (nbp == 1) {
        if (active && TS_CHECK(r0 + i < rows)) bits[(r0 + i) * wpr] = sel;
        return;
    }
    unsigned word = sel << (grp * M % 32);
#pragma unroll
    for (int s = M; s < 32; s <<= 1) word |= __shfl_xor_sync(FULL, word, s);
    if (grp == 0 && active && TS_CHECK(r0 + i < rows && c0 / 32 < wpr)) bits[(r0 + i) * wpr + c0 / 32] = word;
}

// ---------------------------------------------------------------------------
// "Simple" rounding (Appendix B.2): the N best keys of every row, then the N best survivors of
// every column.  A warp takes one mask word's width of blocks, a lane one row and one column, and
// both passes are read off the sorted order of the line (the same networks as the greedy
// selection's).  Bound by the ALU work of the sorts.  2048 x 2048, 8:16: 112 us for ranks by counting
// (M compares per key, from shared memory), 16 us this way.
// ---------------------------------------------------------------------------
constexpr int SIMPLE_WARPS = 4;   // per CTA; independent of one another
template <int M>
__device__ __forceinline__ void simple_round_unit(const float* __restrict__ key, int64_t ld, const UnitMap<M>& um,
                                                  int64_t wpr, int vec, int N, uint32_t* bits, int lane, float* ks) {
    using G = Geom<M, (M < 32) ? 1 : 0>;
    static_assert(G::UW == 32 && G::PASSES == 1, "one mask word wide");
    const int i = lane % M;
    load_keys<G>(key, ld, um, vec != 0, lane, ks);
    __syncwarp();
    const float* const blk = ks + lane / M * M;
    unsigned kept = 0u;              // row pass: my row's columns; column pass: my column's rows
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const float* const line = side ? blk + i : blk + i * G::WS;
        const int st = side ? G::WS : 1;
        float k[M];
        unsigned w[M];
#pragma unroll
        for (int j = 0; j < M; ++j) k[j] = line[j * st];
        sort_line<M>(k, line, st, false, w);
        const unsigned avail = side ? transpose_bits<M>(kept, i) : 0xffffffffu;
        int left = N;
        kept = 0u;
#pragma unroll
        for (int p = 0; p < M; ++p) {
            const unsigned bit = 1u << (w[p] & 31u);
            const bool take = left > 0 && (avail & bit) != 0u;
            kept |= take ? bit : 0u;
            left -= take ? 1 : 0;
        }
    }
    int64_t r0, c0;
    const bool active = um.locate(lane / M, r0, c0);
    const unsigned row = transpose_bits<M>(kept, i);
    write_mask_rows<M>(bits, wpr, um.rows, um.nbp, r0, c0, lane, active, active ? row : 0u);
}
template <int M>
__global__ void __launch_bounds__(32 * SIMPLE_WARPS)
simple_round_kernel(const float* __restrict__ key, int64_t ld, int64_t rows, int64_t cols, int64_t wpr, int64_t nbp,
                    int64_t units, int vec, int N, uint32_t* bits) {
    using G = Geom<M, (M < 32) ? 1 : 0>;
    __shared__ float ks[SIMPLE_WARPS][M * G::WS];
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int64_t unit = (int64_t)blockIdx.x * SIMPLE_WARPS + warp;
    bounds_begin();
    if (unit < units)                // (not a return: the checked flavour ends in a barrier)
        simple_round_unit<M>(key, ld, UnitMap<M>(rows, cols, nbp, unit * G::BPW), wpr, vec, N, bits, lane, ks[warp]);
    bounds_end();
}

// ---------------------------------------------------------------------------
// Fused kernel.  MODE 0: whole method; 1: Algorithm 1 only (plan to global);
// 2: Algorithm 2 only (keys from global).
// ---------------------------------------------------------------------------
struct Params {
    ScoreSrc src;
    const float* keys;   int64_t ld_keys;
    float* plan;         int64_t ld_plan; int plan_is_log;
    uint32_t* bits;      int64_t wpr;
    int64_t rows, cols;
    int64_t nbp;                   // slots of a block row (see UnitMap)
    int N; float Nf, log2N;
    InvN inv_N;
    float c_hi, c_lo;              // tau * log2(e), split in two floats
    int per_block_tau;             // tau is divided by each block's own largest score
    int iters, ls_steps;
    float ee_eps;                  // > 0: stopping test of Algorithm 1 (non-parity mode)
    unsigned long long* iter_sum;  // optional: iterations run, summed over the blocks
    int32_t* status;
    int vec_keys, vec_plan;
};

// The plan of a unit from shared memory to the matrix, whole rows of the unit at a time.
template <class G>
__device__ __forceinline__ void store_plan(const Params& P, const UnitMap<G::M>& um, int lane, const float* src) {
    constexpr int M = G::M;
    constexpr int QW = (G::UW / 4 < 32) ? G::UW / 4 : 32, RPI = 32 / QW;
#pragma unroll 1
    for (int cs = 0; cs < G::UW / (4 * QW); ++cs) {
        const int c = (lane % QW + cs * QW) * 4;
        int64_t r0, c0;
        if (!um.locate(c / M, r0, c0)) continue;
#pragma unroll 2
        for (int r = lane / QW; r < M; r += RPI) {
            if (!TS_CHECK(c + 4 <= G::UW && um.holds_quad(r0 + r, c0 + c % M))) continue;
            const float* const k = src + r * G::WS + c;
            float4 v = make_float4(k[0], k[1], k[2], k[3]);
            if (P.plan_is_log) {
                v.x *= 0.6931471805599453f; v.y *= 0.6931471805599453f;
                v.z *= 0.6931471805599453f; v.w *= 0.6931471805599453f;
            } else {
                v = make_float4(exp2f(v.x), exp2f(v.y), exp2f(v.z), exp2f(v.w));
            }
            float* const d = P.plan + (r0 + r) * P.ld_plan + c0 + c % M;
            if (P.vec_plan) *reinterpret_cast<float4*>(d) = v;
            else { d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w; }
        }
    }
}

// ---------------------------------------------------------------------------
// Algorithm 1 in the twin layout (M < 32, small matrices): the scores of the unit's blocks from
// `panel` to the capped log-plan in `k` (same row stride).  Lane i of a block's M lanes keeps row i
// of the linear iterate (Vr) and, a second time, column i (Vc) with the factors of all rows (Ra); both
// copies see the same operations and stay equal bit for bit.  A row sum and a column sum are then a
// lane's own, and an iteration is two exchanges long: rho to the lanes of the block (one store, M / 4
// broadcast loads of 16 bytes), kap likewise (here 1 / s and kap, and the new thresholds beside 1 / s).  What bounds it is that chain: sum, reciprocal,
// exchange, sum, reciprocal, exchange.  The stash of t0 is the M x 32 matrix in `k` itself, read by
// rows and by columns.  pot: 64 float2 for the owned potentials, then 96 floats for the exchange.
// The numbers are those of dykstra_iterate, whose comments apply; only the order of the sums differs.
// A lone warp takes 143 / 168 / 225 clocks an iteration for M = 4 / 8 / 16, where a block spread over M
// lanes in sub-tiles took 181 / 229 / 267 and the throughput layout takes 134 / 210 / 244 (but leaves one
// warp several blocks to round): 512 x 512 4:8 43.5 -> 37.6 us, 512 x 512 8:16 53.9 -> 46.1 us,
// 256 x 264 2:4 31.9 -> 26.4 us.
// ---------------------------------------------------------------------------
// A buffer is written again only after a barrier that follows its reads: in an iteration the other
// exchange's.
template <int M> __device__ __forceinline__ void fetch(const float* buf, int lane, float2 (&all)[M / 2]) {
    const float4* const src = reinterpret_cast<const float4*>(buf + lane / M * M);
#pragma unroll
    for (int q = 0; q < M / 4; ++q) {
        const float4 v = src[q];
        all[2 * q] = make_float2(v.x, v.y);
        all[2 * q + 1] = make_float2(v.z, v.w);
    }
}
template <int M> __device__ __forceinline__ void exchange(float* buf, int lane, float mine, float2 (&all)[M / 2]) {
    buf[lane] = mine;
    __syncwarp();
    fetch<M>(buf, lane, all);
}
template <int M> __device__ __forceinline__ float sum_line(const float2 (&v)[M / 2]) {
    float2 a = v[0], b = v[1];               // two chains
#pragma unroll
    for (int j = 2; j < M / 2; j += 2) {
        a = __fadd2_rn(a, v[j]);
        b = __fadd2_rn(b, v[j + 1]);
    }
    a = __fadd2_rn(a, b);
    return a.x + a.y;
}
template <int M, bool DELTA>
__device__ __forceinline__ float twin_step(float2 (&Vr)[M / 2], float2 (&Vc)[M / 2], float2 (&Ra)[M / 2], float& r,
                                           float& pc, float* ex, int lane, float Nf, const InvN& iN) {
    constexpr bool THR = ByThreshold<M>::value;
    float2 e[M / 2], f[M / 2], x[M / 2], thr[M / 2];
#pragma unroll
    for (int j = 0; j < M / 2; ++j)
        e[j] = THR ? make_float2(min_nan(Vr[j].x, r), min_nan(Vr[j].y, r))
                   : make_float2(__saturatef(Vr[j].x * r), __saturatef(Vr[j].y * r));
    const float s = sum_line<M>(e);
    const float delta_r = DELTA ? fabsf((THR ? s * rcp_approx(r) : s) - Nf) : 0.0f;
    if (THR) {
        r = iN.times(s);
        ex[64 + lane] = r;               // (published by the barrier in the next line)
        exchange<M>(ex, lane, rcp_approx(s), x);
        fetch<M>(ex + 64, lane, thr);
    } else {
        const float rho = Nf * rcp_approx(s);
        exchange<M>(ex, lane, rho, x);
        r *= rho;
    }
#pragma unroll
    for (int i = 0; i < M / 2; ++i) {
        f[i] = THR ? make_float2(min_nan(Vc[i].x, Ra[i].x), min_nan(Vc[i].y, Ra[i].y))
                   : make_float2(__saturatef(Vc[i].x * Ra[i].x), __saturatef(Vc[i].y * Ra[i].y));
        Ra[i] = THR ? thr[i] : __fmul2_rn(Ra[i], x[i]);
    }
    float2 a = __fmul2_rn(f[0], x[0]), b = __fmul2_rn(f[1], x[1]);
#pragma unroll
    for (int i = 2; i < M / 2; i += 2) {
        a = __ffma2_rn(f[i], x[i], a);
        b = __ffma2_rn(f[i + 1], x[i + 1], b);
    }
    a = __fadd2_rn(a, b);
    const float c = a.x + a.y;
    const float kap = THR ? rcp_approx(c) : Nf * rcp_approx(c);
    exchange<M>(ex + 32, lane, kap, x);
    pc *= kap;
#pragma unroll
    for (int j = 0; j < M / 2; ++j) {
        Vr[j] = __fmul2_rn(Vr[j], x[j]);
        Vc[j] = __fmul2_rn(Vc[j], make_float2(kap, kap));
    }
    return DELTA ? fmaxf(delta_r, fabsf((THR ? Nf * c : c) - Nf)) : 0.0f;
}
template <class G, bool EE>
__device__ __forceinline__ int twin_plan(const Params& P, const float* panel, float* k, float2* pot, int lane) {
    constexpr int M = G::M, WS = G::WS, H = M / 2;
    const int i = lane % M;
    const float* const score_row = panel + i * WS + (lane - i);      // row i of my block
    float* const row = k + i * WS + (lane - i);
    const float* const col = k + lane;                               // column i of my block
    if (!TS_CHECK((M - 1) * WS + lane < M * WS && i * WS + (lane - i) + M <= M * WS)) return 0;
    float* const ex = reinterpret_cast<float*>(pot + 64);
    float2* const fpot = pot + lane;
    float2* const gpot = pot + 32 + lane;
    float t[M];
    float mx = 0.0f;
#pragma unroll
    for (int j = 0; j < M; ++j) {
        t[j] = score_row[j];
        mx = fmaxf(mx, t[j]);
    }
    float c_hi = P.c_hi, c_lo = P.c_lo;
    if (P.per_block_tau) {   // tau of this block = tau_rel / its largest score
        float bm = mx;
#pragma unroll
        for (int s = 1; s < M; s <<= 1) bm = fmaxf(bm, __shfl_xor_sync(FULL, bm, s));
        c_hi = (bm > 0.0f) ? __fdiv_rn(P.c_hi, bm) : 0.0f;
        c_lo = (bm > 0.0f) ? __fdiv_rn(fmaf(-c_hi, bm, P.c_hi) + P.c_lo, bm) : 0.0f;
    }
    if (P.iters <= 0) {
#pragma unroll
        for (int j = 0; j < M; ++j) row[j] = fmaf(t[j], c_lo, t[j] * c_hi);
        __syncwarp();
        return 0;
    }
    const float sh = mx * c_hi;
#pragma unroll
    for (int j = 0; j < M; ++j) {
        t[j] = fmaf(t[j], c_lo, fmaf(t[j], c_hi, -sh));
        row[j] = t[j];
    }
    float r = 1.0f, pc = 1.0f;               // products of rho (or 1 / them) and of kap since the rebuild
    constexpr float SIGN = ByThreshold<M>::value ? -1.0f : 1.0f;
    float2 x[H], y[H];
    {   // iteration 0, log domain
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < M; ++j) s += ex2_approx(t[j]);
        const float F = P.log2N - lg2_approx(s);
        *fpot = make_float2(F, 0.f);
        exchange<M>(ex, lane, F, x);             // (its barrier also publishes t0)
        float cm = -3.4028234e38f, cp = 0.f;
#pragma unroll
        for (int a = 0; a < M; ++a) {
            t[a] = col[a * WS] + ((a % 2) ? x[a / 2].y : x[a / 2].x);
            cm = (a == 0) ? t[0] : fmaxf(cm, t[a]);
        }
#pragma unroll
        for (int a = 0; a < M; ++a) cp += ex2_approx(t[a] - cm);
        *gpot = make_float2((P.log2N - cm) - lg2_approx(cp), 0.f);
    }
    int it = 1, iters = P.iters;
    float2 Vr[H], Vc[H], Ra[H];
#pragma unroll 1
    while (it < iters) {
        const float F = add_potential(fpot, r, SIGN), Gc = add_potential(gpot, pc);
        __syncwarp();                            // every lane has read the exchange before
        exchange<M>(ex, lane, F, x);
        exchange<M>(ex + 32, lane, Gc, y);
#pragma unroll
        for (int j = 0; j < H; ++j) {
            const float2 a = __fadd2_rn(__fadd2_rn(make_float2(row[2 * j], row[2 * j + 1]), make_float2(F, F)), y[j]);
            const float2 b = __fadd2_rn(__fadd2_rn(make_float2(col[2 * j * WS], col[(2 * j + 1) * WS]), x[j]),
                                        make_float2(Gc, Gc));
            Vr[j] = make_float2(ex2_approx(a.x), ex2_approx(a.y));
            Vc[j] = make_float2(ex2_approx(b.x), ex2_approx(b.y));
            Ra[j] = make_float2(1.0f, 1.0f);
        }
        r = pc = 1.0f;
        const int run_end = (iters - it > MAXRUN) ? it + MAXRUN : iters;
        bool wide = false;
#pragma unroll 1
        while (!wide && it + CHECK <= run_end) {
#pragma unroll
            for (int u = 0; u < CHECK - 1; ++u) twin_step<M, false>(Vr, Vc, Ra, r, pc, ex, lane, P.Nf, P.inv_N);
            const float delta = twin_step<M, EE>(Vr, Vc, Ra, r, pc, ex, lane, P.Nf, P.inv_N);
            it += CHECK;
            if (EE && __all_sync(FULL, delta < P.ee_eps)) {   // every block of the warp has converged
                iters = it;
                wide = true;                                  // skips the remainder loop as well
                break;
            }
            wide = __any_sync(FULL, out_of_window(r) || out_of_window(pc));
        }
        if (!wide) {   // fewer than CHECK iterations left (end of the last run only)
#pragma unroll 1
            for (; it < run_end; ++it) twin_step<M, false>(Vr, Vc, Ra, r, pc, ex, lane, P.Nf, P.inv_N);
        }
    }
    // final potentials, t = t0 + F + G and x = min(t, 0)
    const float F = add_potential<true>(fpot, r, SIGN), Gc = add_potential<true>(gpot, pc);
    __syncwarp();                                // every lane has read the exchange before
    exchange<M>(ex + 32, lane, Gc, y);           // (its barrier: no column of t0 is read any more)
#pragma unroll
    for (int j = 0; j < M; ++j) row[j] = fminf((row[j] + F) + ((j % 2) ? y[j / 2].y : y[j / 2].x), 0.0f);
    __syncwarp();
    return iters;
}

template <class G, int MODE, bool EE> struct SmemLayout {   // of one warp
    static constexpr int M = G::M;
    // The score panel is kept beside the key panel for the local search, except that the whole
    // method at M = 32 reads the scores of a block again when it needs them (RELOAD): the panel would
    // cost the SM 4 of its 20 warps (14336 x 4096, 16:32: 3.13 ms with it, 3.03 without).  The stopping test
    // keeps it: a dozen iterations leave nothing to hide the second read behind, and its loop does not fit in
    // the 96 registers of 20 warps (84 bytes spilled; Student scores 656 us with RELOAD, 606 without).
    static constexpr bool RELOAD = (M == 32 && MODE == 0 && G::V == 0 && !EE);
    static constexpr bool HAS_W = MODE != 1 && !RELOAD;
    static constexpr int POT = (MODE == 2) ? 0 : 64 * (G::RO + G::CO) + (G::TWIN ? (ByThreshold<M>::value ? 96 : 64) : 0);
    static constexpr int CPRE = (M == 32 && MODE != 1) ? 32 * CPRE_STRIDE : 0;
    static constexpr int AUX = (POT > CPRE) ? POT : CPRE;
    alignas(16) float k[M * G::WS];     // scores, stash of t0, keys, row prefix tables in turn
    float w[HAS_W ? M * G::WS : 1];
    alignas(16) float aux[AUX ? AUX : 1];   // potentials (and the twin layout's exchange), then the
                                            // column-prefix tables of M = 32
};
// Resident warps per SM the register allocation aims for: 20 where the loop fits in 96 registers (see
// RELOAD for the stopping test), 12 for the latency layout, where registers count for more.
template <int M, int V, bool EE> struct MinWarps {
    static constexpr int value = (V == 1) ? 12 : (M >= 16 && V == 0 && !EE) ? 20 : 16;
};
// Warps per CTA.  One: 3 to 25 % faster than four on ragged widths (finer tail), except where much of the
// time goes into code that runs once, as at M = 32 with blocks that converge early: four warps that go
// through it together (barriers after the loader and before the rounding stage) share what they fetch of it
// (14336 x 4096, Student scores: 1,420 us apart, 1,310 together; Gaussian ones 2.95 ms both ways; two warps
// 1,415, five 1,290 and 3.02.  Stopping test: 663 and 606 us; Gaussian 3.00 and 3.07 ms).
template <int M, int V, bool EE> struct CtaWarps { static constexpr int value = (M == 32 && V == 0) ? 4 : 1; };

// Cells of a lane's sub-tile in a shared-memory panel.
template <class G> struct SubTile {
    int r0, gr, c0, gc;
    __device__ __forceinline__ explicit SubTile(int lane) {
        using T = typename G::T;
        const int g = lane % G::LPB, lr = g / T::PC, lc = g % T::PC;   // lane inside its block
        r0 = lr * T::MR; gr = xor_perm<T::MR, T::PC>(lc);
        c0 = lane / G::LPB * G::M + lc * T::MC; gc = xor_perm<T::MC, T::PR>(lr);
    }
    __device__ __forceinline__ int row(int a) const { return r0 + (a ^ gr); }
    __device__ __forceinline__ int col(int b) const { return c0 + (b ^ gc); }
};

template <int M, int MODE, int V, bool EE>
__global__ void __launch_bounds__(32 * CtaWarps<M, V, EE>::value, MinWarps<M, V, EE>::value / CtaWarps<M, V, EE>::value)
tsenor_kernel(const Params P) {
    using G = Geom<M, V>;
    using T = typename G::T;
    using L = SmemLayout<G, MODE, EE>;
    [[maybe_unused]] constexpr int MR = T::MR, MC = T::MC, PR = T::PR, PC = T::PC;
    constexpr int WPC = CtaWarps<M, V, EE>::value;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x % 32;
    L& sm = reinterpret_cast<L*>(smem_raw)[threadIdx.x / 32];
    bounds_begin();
    int flags = 0;

    // ---- block loader
    float* const panel = L::HAS_W ? sm.w : sm.k;
    {
        const UnitMap<M> um(P.rows, P.cols, P.nbp, this_unit<WPC>() * G::BPW);
        if constexpr (MODE == 2) {   // (tsenor_round: the scores are plain |W|)
            if (P.src.vec_w && P.vec_keys) {
                if (load_scores_and_keys<G>(P.src, P.keys, P.ld_keys, um, lane, panel, sm.k)) flags |= DEV_NONFINITE;
            } else {
                if (load_plain_scores<G>(P.src, um, lane, panel)) flags |= DEV_NONFINITE;
                if (load_keys<G>(P.keys, P.ld_keys, um, P.vec_keys != 0, lane, sm.k)) flags |= DEV_NONFINITE;
            }
        } else {
            if (load_scores<G, G::UW>(P.src, um, 0, lane, panel)) flags |= DEV_NONFINITE;
        }
    }
    if (WPC > 1) __syncthreads();
    else __syncwarp();

    // ---- Algorithm 1
    if constexpr (MODE != 2 && G::TWIN) {
        const int ran = twin_plan<G, EE>(P, panel, sm.k, reinterpret_cast<float2*>(sm.aux), lane);
        if (P.iter_sum && P.iters > 0) {
            const UnitMap<M> um(P.rows, P.cols, P.nbp, this_unit<WPC>() * G::BPW);
            int64_t r0, c0;
            const bool there = um.locate(lane / M, r0, c0);
            const int nact = __popc(__ballot_sync(FULL, there && lane % M == 0));
            if (lane == 0 && nact) atomicAdd(P.iter_sum, (unsigned long long)ran * nact);
        }
    } else if constexpr (MODE != 2) {
        float t[MR][MC];
        float mx[MR];
        const SubTile<G> st0(lane);
#pragma unroll
        for (int a = 0; a < MR; ++a) {
            float m = 0.f;
#pragma unroll
            for (int b = 0; b < MC; ++b) {
                const int cell = st0.row(a) * G::WS + st0.col(b);
                t[a][b] = TS_CHECK(st0.row(a) < M && st0.col(b) < G::UW) ? panel[cell] : 0.0f;
                m = fmaxf(m, t[a][b]);
            }
            mx[a] = m;
        }
        float c_hi = P.c_hi, c_lo = P.c_lo;
        if (P.iters > 0 || P.per_block_tau) {
            reduce_scatter<MR, PC>(mx, 1, OpMax());
            all_gather<MR, PC>(mx, 1);
        }
        if (P.per_block_tau) {   // tau of this block = tau_rel / its largest score
            float bm = mx[0];
#pragma unroll
            for (int a = 1; a < MR; ++a) bm = fmaxf(bm, mx[a]);
#pragma unroll
            for (int s = 0; (1 << s) < PR; ++s) bm = fmaxf(bm, __shfl_xor_sync(FULL, bm, PC << s));
            if (bm > 0.0f) {
                c_hi = __fdiv_rn(P.c_hi, bm);
                c_lo = __fdiv_rn(fmaf(-c_hi, bm, P.c_hi) + P.c_lo, bm);
            } else {
                c_hi = 0.0f; c_lo = 0.0f;
            }
        }
        __syncwarp();            // the score panel is read: its cells may become the stash
        if (P.iters > 0) {
#pragma unroll
            for (int a = 0; a < MR; ++a) {
                const float sh = mx[a] * c_hi;
#pragma unroll
                for (int b = 0; b < MC; ++b) t[a][b] = fmaf(t[a][b], c_lo, fmaf(t[a][b], c_hi, -sh));
            }
            const int ran = dykstra_iterate<G, EE>(t, sm.k, reinterpret_cast<float2*>(sm.aux), lane, P.Nf, P.inv_N, P.log2N,
                                                   P.iters, P.ee_eps);
            if (P.iter_sum) {   // one add per warp: iterations x blocks of the warp that exist
                const UnitMap<M> um(P.rows, P.cols, P.nbp, this_unit<WPC>() * G::BPW);
                int64_t r0, c0;
                const bool there = um.locate(lane / G::LPB, r0, c0);
                const int nact = __popc(__ballot_sync(FULL, there && lane % G::LPB == 0));
                if (lane == 0 && nact) atomicAdd(P.iter_sum, (unsigned long long)ran * nact);
            }
#pragma unroll
            for (int a = 0; a < MR; ++a)
#pragma unroll
                for (int b = 0; b < MC; ++b) t[a][b] = fminf(t[a][b], 0.0f);   // x = min(x + q, 0)
        } else {
#pragma unroll
            for (int a = 0; a < MR; ++a)
#pragma unroll
                for (int b = 0; b < MC; ++b) t[a][b] = fmaf(t[a][b], c_lo, t[a][b] * c_hi);
        }
        __syncwarp();            // sm.k served as stash until here; now it takes the keys
        int l = lane;            // tied to the result of the iterations, so that the addresses of the
        asm("" : "+r"(l), "+f"(t[0][0]));   // cells are worked out again and not kept over the loop
        const SubTile<G> st(l);
#pragma unroll
        for (int a = 0; a < MR; ++a)
#pragma unroll
            for (int b = 0; b < MC; ++b)
                if (TS_CHECK(st.row(a) < M && st.col(b) < G::UW)) sm.k[st.row(a) * G::WS + st.col(b)] = t[a][b];
        __syncwarp();
    }
    if (MODE == 1)               // ---- plan writer
        store_plan<G>(P, UnitMap<M>(P.rows, P.cols, P.nbp, this_unit<WPC>() * G::BPW), lane, sm.k);

    if (MODE == 0 && WPC > 1) __syncthreads();
    // ---- Algorithm 2 and the mask writer: the blocks of one mask word (GPW M = 32 columns) a pass
    if (MODE != 1) {
        const int grp = lane / M;
        const auto unit_map = [&]() { return UnitMap<M>(P.rows, P.cols, P.nbp, this_unit<WPC>() * G::BPW); };
        const UnitMap<M> um = unit_map();
#pragma unroll 1
        for (int pass = 0; pass < G::PASSES; ++pass) {
            const int slot0 = pass * G::GPW, c = (slot0 + grp) * M;
            int64_t r0, c0;
            const bool active = um.locate(slot0 + grp, r0, c0);
            if (!TS_CHECK(c + M <= G::UW)) continue;     // warp-uniform up to the group
            const unsigned sel = round_block<G>(
                sm.k + c, (L::RELOAD ? sm.k : sm.w) + c, reinterpret_cast<unsigned*>(sm.aux) + lane * CPRE_STRIDE,
                lane, active, MODE == 0 && P.iters > 0, P.N, P.ls_steps, flags, [&]() {
                    if (L::RELOAD) {
                        __syncwarp();
                        load_scores<G, 32>(P.src, unit_map(), slot0, lane, sm.k + slot0 * M);
                        __syncwarp();
                    }
                });
            if (M == 32) unit_map().locate(slot0 + grp, r0, c0);   // worked out again: one pass, few registers
            write_mask_rows<M>(P.bits, P.wpr, P.rows, P.nbp, r0, c0, lane, active, sel);
            __syncwarp();
        }
    }
    flags |= bounds_end();
    flags = __reduce_or_sync(FULL, flags);
    if (flags && lane == 0 && P.status) atomicOr(P.status, flags);
}

}  // namespace tsenor
