// Negacyclic number-theoretic transform over 64-bit RNS residues (the "NTT kernels" the paper's
// FHE backend relies on, Sec. 4.2), batched over polynomials and primes.
//
// Forward: merged-twiddle Cooley-Tukey, natural order in, bit-reversed order out:
//   position i holds a(psi^(2*brev(i)+1)).  Inverse: Gentleman-Sande, bit-reversed in, natural out.
// The internal order never leaves the library: pointwise products do not care, and automorphisms
// are applied as index gathers that account for it.
//
// A transform of N = R*C points runs as two launches.  The strided pass transforms the R rows
// (stride C) of a tile of adjacent columns; the contiguous pass transforms chunks of C adjacent
// points.  Inside a pass every thread keeps a closed set of up to 8 points in registers for up to
// three butterfly stages, and sets are exchanged through shared memory between stage groups.
#include "bf_host.h"

#include <type_traits>

namespace bf {

cudaEvent_t Profiler::get() {
    if (!pool.empty()) {
        cudaEvent_t e = pool.back();
        pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

ProfScope::ProfScope(Profiler* prof, int c, cudaStream_t st) : p(prof), cat(c), s(st) {
    if (!p) return;
    p->launches[cat]++;
    if (p->timing) {
        a = p->get();
        cudaEventRecord(a, s);
    }
}

ProfScope::~ProfScope() {
    if (!p || !a) return;
    cudaEvent_t b = p->get();
    cudaEventRecord(b, s);
    p->recs.push_back({cat, a, b});
}

struct LoadConsts {
    u64 q, mu, lift_mod, lift_red;
    double qd, qinv, c30, c30q, k59;      // (LOAD_I64_MONT: c30 = 2^96 mod q, k59 = the offset for -2^127)
    double c64d, c64q;                     // LOAD_I64_MONT: 2^64 mod q
    bool wide;          // target prime of 2^41 or more: values must stay in [0, 4q); otherwise they are signed
    bool src_small;     // LOAD_REDUCE: every source word is below 1.5 q already (block-uniform)
    bool src_fp;        // LOAD_REDUCE: every source word is below 2^51
    bool staged_fp;     // the staged source holds the bits of integer-valued doubles
                        //   (LOAD_I64_MONT: all below 2^40; src_small, src_fp: no factor 2^64, q from 2^39 or below)
};

template <int LOAD>
__device__ __forceinline__ u64 load_src(const void* src, size_t idx, const LoadConsts& c) {
    if (LOAD == LOAD_PLAIN) return ((const u64*)src)[idx];
    if (LOAD == LOAD_REDUCE) {
        u64 t = ((const u64*)src)[idx];
        if (c.staged_fp) t = d2u(__longlong_as_double((long long)t));
        return c.src_small ? (t >= c.q ? t - c.q : t) : barrett64(t, c.q, c.mu);
    }
    if (LOAD == LOAD_I64_MONT && c.staged_fp) {             // |v| < 2^40 < q
        const i64 v = d2i(((const double*)src)[idx]);
        const u64 m = mul_shoup(v < 0 ? (u64)(-v) : (u64)v, c.lift_mod, c.lift_red, c.q);
        return v < 0 && m != 0 ? c.q - m : m;
    }
    if (LOAD == LOAD_I64 || LOAD == LOAD_I64_MONT) {
        i64 v = ((const i64*)src)[idx];
        u64 a = v < 0 ? (u64)(-v) : (u64)v;
        u64 m = barrett64(a, c.q, c.mu);
        m = (v < 0 && m != 0) ? c.q - m : m;
        if (LOAD == LOAD_I64_MONT) m = mul_shoup(m, c.lift_mod, c.lift_red, c.q);   // (2^64 mod q, its Shoup companion)
        return m;
    }
    // LOAD_CENTRED: the word is t' + 2^59 with t' the centred lift of a residue modulo lift_mod
    const u64 T = ((const u64*)src)[idx];
    const bool neg = T < (1ull << 59);
    const u64 t = neg ? T + c.lift_mod - (1ull << 59) : T - (1ull << 59);      // back to [0, lift_mod)
    u64 m = barrett64(t, c.q, c.mu);
    if (neg) m = sub_mod(m, c.lift_red, c.q);
    return m;
}

// The same loads for a modulus on the fp64 path: the result is an integer-valued double congruent to the
// source, of magnitude below 3.6 q (lazy: the butterflies reduce); non-negative for primes of 2^41 or more.
template <int LOAD>
__device__ __forceinline__ double load_src_fp(const void* src, size_t idx, const LoadConsts& c) {
    if (LOAD == LOAD_REDUCE) {
        const u64 t = ((const u64*)src)[idx];
        const double td = c.staged_fp ? __longlong_as_double((long long)t) : u2d(t);
        if (c.src_small) return td;
        if (c.src_fp) {                                  // t - round(t / q) q, plus q where values must not be negative
            const double v = fp_centre(td, c.qd, c.qinv);
            return c.wide ? __dadd_rn(v, c.qd) : v;
        }
        return u2d(barrett64(t, c.q, c.mu));
    }
    if (LOAD == LOAD_CENTRED) {
        // t' + 2^59 = hi 2^30 + lo, so t' = hi (2^30 mod q) + lo - (2^59 mod q)  (mod q); with the product
        // centred in (-0.75 q, 0.75 q), lo < 2^30 and k59 = 2q - (2^59 mod q) the sum is positive
        const u64 T = ((const u64*)src)[idx];
        const double hi = u2d(T >> 30), lo = u2d(T & ((1ull << 30) - 1));
        return __dadd_rn(__dadd_rn(fp_mul_centred(hi, c.c30, c.c30q, c.qd), lo), c.k59);   // (k59: see LoadConsts)
    }
    if (LOAD == LOAD_I64_MONT && c.staged_fp) {
        // |v| < 2^40: as it is where plaintexts carry no factor and that is below 2q, else centred, or times 2^64 mod q
        // (a centred product, within 0.51q; plus q where values must not be negative)
        const double v = ((const double*)src)[idx];
        if (c.src_small) return v;
        if (c.src_fp) return fp_centre(v, c.qd, c.qinv);
        const double m = fp_mul_centred_signed(v, c.c64d, c.c64q, c.qd);
        return c.wide ? __dadd_rn(m, c.qd) : m;
    }
    if (LOAD == LOAD_I64_MONT) {
        // v = (hi' - 2^31) 2^32 + lo with hi' = (v >> 32) + 2^31 in [0, 2^32); two centred products (each
        // within 0.75 q, 0.51 q for primes below 2^41) plus the offset: magnitude below 1.6 q, or within
        // (0, 4q) for the primes whose values must stay non-negative
        const uint2 w = ((const uint2*)src)[idx];
        const double hi = __uint2double_rn(w.y ^ 0x80000000u), lo = __uint2double_rn(w.x);
        return __dadd_rn(__dadd_rn(fp_mul_centred(hi, c.c30, c.c30q, c.qd), fp_mul_centred(lo, c.c64d, c.c64q, c.qd)), c.k59);
    }
    return u2d(load_src<LOAD>(src, idx, c));
}

// How a modulus is transformed.
//   PATH_DP    primes below 2^41: signed integer-valued doubles, reduced lazily
//   PATH_WIDE  primes from 2^41 up to 2^50: integer-valued doubles in [0, 4q) (forward) or [0, 2q) (inverse)
//   PATH_INT   larger primes: 64-bit integers below 16q (forward) or 4q (inverse), Shoup products with a short quotient
enum Path : int { PATH_INT = 0, PATH_WIDE = 1, PATH_DP = 2 };
__device__ __forceinline__ int path_of(const RingDev& R, u32 mod) { return !R.fp_ok[mod] ? PATH_INT : (R.q[mod] >> 41) ? PATH_WIDE : PATH_DP; }
template <int PATH> struct Elem { typedef double T; };
template <> struct Elem<PATH_INT> { typedef u64 T; };
__device__ __forceinline__ void from_u64(u64& dst, u64 v) { dst = v; }
__device__ __forceinline__ void from_u64(double& dst, u64 v) { dst = u2d(v); }

struct ModConsts {
    u64 q;
    double qd, qinv;
    u32 mu;             // floor(2^64 / q), PATH_INT (q above 2^50: below 2^14)
    __device__ __forceinline__ ModConsts(const RingDev& R, u32 mod) : q(R.q[mod]), qd(R.qd[mod]), qinv(R.qinv_d[mod]), mu((u32)R.mu[mod]) {}
};

// x * w - h q for any 64-bit x and a constant w < q < 2^60 with companion ws = floor(w 2^64 / q): h is the high word of x * ws short
// of what its low parts would carry in, i.e. by less than 3, so the result is congruent to x * w and in [0, 4q).  (Three wide
// multiplications instead of four and their carries.)
__device__ __forceinline__ u64 mul_shoup_short(u64 x, u64 w, u64 ws, u64 q) {
    const u32 x0 = (u32)x, x1 = (u32)(x >> 32), s0 = (u32)ws, s1 = (u32)(ws >> 32);
    const u64 h = (u64)x1 * s1 + __umulhi(x1, s0) + __umulhi(x0, s1);
    return x * w - h * q;
}
// any 64-bit x, in particular any below 16q, minus a multiple of q, q above 2^50: in [0, 3q).  The quotient floor(x_hi mu / 2^32) is short of x / q
// by less than 1 + 2^-18 + x / 2^64.
__device__ __forceinline__ u64 reduce_16q(u64 x, const ModConsts& c) { return x - (u64)__umulhi((u32)(x >> 32), c.mu) * c.q; }

// 32 bytes at once (the widest global access of sm_100)
__device__ __forceinline__ void ldg4(const double* p, double& a, double& b, double& c, double& d) {
    asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a), "=d"(b), "=d"(c), "=d"(d) : "l"(p));
}
__device__ __forceinline__ void stg4(u64* p, u64 a, u64 b, u64 c, u64 d) {
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

// The 2^ST twiddles of one stage of a register-resident set: entries idx .. idx + 2^ST - 1 (idx a multiple of 2^ST) of the
// prime's table.  PATH_DP reads a table of plain doubles (half the bytes of the other paths' (w, companion) pairs: the
// transforms are limited by what passes through L1 as much as by arithmetic) and makes w / q with one multiplication,
// within 2^-52 relative.  SM: the table is a copy in shared memory.
template <int ST, bool SM>
__device__ __forceinline__ void load_twiddles(const double* tab, u32 idx, double (&w)[1 << ST]) {
    const double* p = tab + idx;
    if constexpr (ST == 0) {
        w[0] = SM ? *p : __ldg(p);
    } else if constexpr (ST == 1 || SM) {
#pragma unroll
        for (int i = 0; i < (1 << ST); i += 2) {
            const double2 v = SM ? *(const double2*)(p + i) : __ldg((const double2*)(p + i));
            w[i] = v.x;
            w[i + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < (1 << ST); i += 4) ldg4(p + i, w[i], w[i + 1], w[i + 2], w[i + 3]);
    }
}

// Butterflies of one register-resident set of 2^K points (e[OFF ..]) over K consecutive stages.  base = (blocks at the
// group's first forward stage) + the set's block: stage st, sub-block sub uses twiddle (base << st) + sub.
//
// PATH_DP forward: (X, Y) -> (X + s, X - s), s = Y*w centred in (-0.54q, 0.54q): magnitudes grow by at most 0.54q per
// stage, from at most 3.6q after the load functors to below 13q after log2 N <= 16 stages; one reduction at the very
// end.  Inverse: (a, b) -> (a + b, (a - b)*w centred): the sums double per stage, the product takes |a - b| < 2^47, i.e.
// magnitudes below 32q; see centre_sums.
// PATH_WIDE: the centred product lies in (-0.75q, 0.75q) and values must stay below 4q < 2^52, so the forward butterfly
// keeps Harvey's invariant [0, 4q) with one conditional subtraction: (X, Y) -> (X~ + T, X~ - T + 2q), X~ = X reduced
// below 2q, T = Y*w + q in (0.25q, 1.75q); the inverse is (a, b) -> (a + b reduced below 2q, (a - b + 2q)*w + q in
// (0.25q, 1.75q)): values in [0, 2q).
// PATH_INT: products come back below 4q (see mul_shoup_short).  Forward, (X, Y) -> (X + T, X - T + 4q): any 64-bit Y will do, X
// grows by 4q per stage, and where a group starts the X of its first stage are brought below 3q: K <= 3 stages end below 15q.
// Inverse, (a, b) -> (a + b, (a - b + 4q) w): every second stage, and the last of a group, brings its sums below 3q; the stage
// before leaves them below 8q, so that its successor's differences take an offset of 8q.
// (768 -> 2304 on 2^13, two of whose five moduli are 60-bit primes: 234.2 us with products below 2q, which a conditional
// subtraction per butterfly keeps, 230.9 us like this; 64 x 64 on 2^12: 59.8 and 59.4 us.)
template <int ST, int K, bool FWD, int PATH, bool SM, int OFF, typename T>
__device__ __forceinline__ void stage_butterflies(T (&e)[8], const void* __restrict__ tab, u32 base, const ModConsts& c) {
    constexpr int d = (1 << K) >> (ST + 1);
    const u32 idx = base << ST;
    if constexpr (PATH == PATH_DP) {
        double w[1 << ST];
        load_twiddles<ST, SM>((const double*)tab, idx, w);
#pragma unroll
        for (int sub = 0; sub < (1 << ST); ++sub) {
            const double wq = __dmul_rn(w[sub], c.qinv);
#pragma unroll
            for (int off = 0; off < d; ++off) {
                const int i = OFF + sub * 2 * d + off;
                if (FWD) {
                    const double sv = fp_mul_centred_signed(e[i + d], w[sub], wq, c.qd);
                    const double x = e[i];
                    e[i] = __dadd_rn(x, sv);
                    e[i + d] = __dsub_rn(x, sv);
                } else {
                    const double a = e[i], b = e[i + d];
                    e[i] = __dadd_rn(a, b);
                    e[i + d] = fp_mul_centred_signed(__dsub_rn(a, b), w[sub], wq, c.qd);
                }
            }
        }
    } else {
        const double q2d = __dadd_rn(c.qd, c.qd);
#pragma unroll
        for (int sub = 0; sub < (1 << ST); ++sub) {
            const ulonglong2 wb = SM ? ((const ulonglong2*)tab)[idx + sub] : __ldg((const ulonglong2*)tab + idx + sub);
#pragma unroll
            for (int off = 0; off < d; ++off) {
                const int i = OFF + sub * 2 * d + off;
                if constexpr (PATH == PATH_WIDE) {
                    const double w = __longlong_as_double((long long)wb.x), wq = __longlong_as_double((long long)wb.y);
                    if (FWD) {
                        double x = e[i];
                        if (x >= q2d) x = __dsub_rn(x, q2d);
                        const double t = __dadd_rn(fp_mul_centred(e[i + d], w, wq, c.qd), c.qd);
                        e[i] = __dadd_rn(x, t);
                        e[i + d] = __dadd_rn(__dsub_rn(x, t), q2d);
                    } else {
                        const double a = e[i], b = e[i + d];
                        double s2 = __dadd_rn(a, b);
                        if (s2 >= q2d) s2 = __dsub_rn(s2, q2d);
                        e[i] = s2;
                        e[i + d] = __dadd_rn(fp_mul_centred(__dadd_rn(__dsub_rn(a, b), q2d), w, wq, c.qd), c.qd);
                    }
                } else if (FWD) {
                    const u64 x = ST == 0 ? reduce_16q(e[i], c) : e[i];
                    const u64 t = mul_shoup_short(e[i + d], wb.x, wb.y, c.q);
                    e[i] = x + t;
                    e[i + d] = x - t + 4 * c.q;
                } else {
                    constexpr int POS = K - 1 - ST;             // (stages of the group before this one)
                    const u64 a = e[i], b = e[i + d];
                    e[i] = POS % 2 == 1 || ST == 0 ? reduce_16q(a + b, c) : a + b;
                    e[i + d] = mul_shoup_short(a - b + (POS % 2 == 1 ? 8 : 4) * c.q, wb.x, wb.y, c.q);
                }
            }
        }
    }
}
template <int K, bool FWD, int PATH, bool SM, int OFF = 0, typename T>
__device__ __forceinline__ void set_butterflies(T (&e)[8], const void* __restrict__ tab, u32 base, const ModConsts& c) {
    if constexpr (FWD) {
        stage_butterflies<0, K, FWD, PATH, SM, OFF>(e, tab, base, c);
        if constexpr (K > 1) stage_butterflies<1, K, FWD, PATH, SM, OFF>(e, tab, base, c);
        if constexpr (K > 2) stage_butterflies<2, K, FWD, PATH, SM, OFF>(e, tab, base, c);
    } else {
        if constexpr (K > 2) stage_butterflies<2, K, FWD, PATH, SM, OFF>(e, tab, base, c);
        if constexpr (K > 1) stage_butterflies<1, K, FWD, PATH, SM, OFF>(e, tab, base, c);
        stage_butterflies<0, K, FWD, PATH, SM, OFF>(e, tab, base, c);
    }
}
// After an inverse group the points that were sums to the end have grown: point 0 by 2^K, point 1 to 2^(K-1) fresh
// products (0.54q each), point 2 and 3 to 2^(K-2) of them, and so on.  Centring point 0 leaves every point within 2.2q, so
// that a group of at most three stages that starts there stays below 18q < 2^47.  (The contiguous pass starts from canonical
// residues and does not centre after its first group of two stages: the second starts below 4q and stays below 16q.)
template <int K, int PATH, int OFF = 0, typename T>
__device__ __forceinline__ void centre_sums(T (&e)[8], const ModConsts& c) {
    if constexpr (PATH == PATH_DP) {
        e[OFF] = fp_centre(e[OFF], c.qd, c.qinv);
    }
}

constexpr int LOG_C = 8;              // contiguous pass: chunks of 256 points

// Between the two passes of a transform the data sit in dst as lazily reduced values: 64-bit
// integers for the integer path, fp64 bit patterns for the fp64 path (the modulus decides, so both
// passes agree).

// Geometry of the strided pass over 2^LOG_R rows (stride 256) of 2^LOG_LANES adjacent columns: up to three groups of at most
// three stages, eight points a thread.  (Sixteen points and two groups execute a sixth fewer instructions, but half the
// threads hide less latency and the integer path's blocks, which every launch waits for, take twice as long: the four calls
// of a 0.6B decoder layer took 8 % longer.)
__host__ __device__ constexpr int n_groups(int log_len) { return log_len <= 3 ? 1 : (log_len <= 6 ? 2 : 3); }
__host__ __device__ constexpr int group_k(int log_len, int gi) {
    // 2:{2} 3:{3} 4:{2,2} 5:{3,2} 6:{3,3} 7:{3,2,2} 8:{3,3,2}
    return log_len <= 3 ? log_len
         : log_len == 4 ? 2
         : log_len == 5 ? (gi == 0 ? 3 : 2)
         : log_len == 6 ? 3
         : log_len == 7 ? (gi == 0 ? 3 : 2)
         : (gi == 2 ? 2 : 3);
}
// log2 of the point spacing of group gi's sets (forward order index)
__host__ __device__ constexpr int group_log_step(int log_len, int gi) {
    int done = 0;
    for (int i = 0; i <= gi; ++i) done += group_k(log_len, i);
    return log_len - done;
}
template <int LOG_R, int LOG_LANES>
struct StridedGeo {
    static constexpr int LEN = 1 << LOG_R, LANES = 1 << LOG_LANES, POINTS = LEN * LANES;
    static constexpr int NT = LOG_R == 4 ? POINTS / 4 : POINTS / 8 < 32 ? 32 : POINTS / 8;       // (4 points a thread where groups have 2 stages)
    static constexpr int BLOCKS = NT >= 512 ? 2 : NT >= 256 ? 4 : 8;       // resident blocks per SM
    static constexpr int TILES = (1 << LOG_C) / LANES;
    static constexpr int TW_WORDS = 2 * LEN;                               // (w, companion) pairs, or half of it
};

__device__ __forceinline__ const void* twiddle_table(const RingDev& R, bool fwd, int path, u32 mod) {
    return path == PATH_DP ? (const void*)((fwd ? R.tw8_fwd : R.tw8_inv) + (size_t)mod * R.N)
                           : (const void*)((fwd ? R.tw_fwd : R.tw_inv) + (size_t)mod * R.N);
}

// A thread's share of the first 2^LOG_R twiddles of a prime, fetched early and put into shared memory later.
template <int LOG_R>
struct StridedTwiddles {
    ulonglong2 mine;
    __device__ __forceinline__ void fetch(const RingDev& R, bool fwd, int path, u32 mod) {
        mine = make_ulonglong2(0, 0);
        if (threadIdx.x < (1 << LOG_R)) {
            const void* tab = twiddle_table(R, fwd, path, mod);
            if (path == PATH_DP) mine.x = __ldg((const u64*)tab + threadIdx.x);
            else mine = __ldg((const ulonglong2*)tab + threadIdx.x);
        }
    }
    __device__ __forceinline__ void put(u64* tws, int path) const {
        if (threadIdx.x < (1 << LOG_R)) {
            if (path == PATH_DP) tws[threadIdx.x] = mine.x;
            else ((ulonglong2*)tws)[threadIdx.x] = mine;
        }
    }
};

template <int LOAD>
__device__ __forceinline__ LoadConsts load_consts(const RingDev& R, const PolyBatch& B, u32 o, u32 mod) {
    LoadConsts lc;
    const u64 q = R.q[mod], mu = R.mu[mod];
    lc.q = q;
    lc.mu = mu;
    lc.lift_red = (LOAD == LOAD_CENTRED) ? barrett64(B.lift_mod, q, mu) : (LOAD == LOAD_I64_MONT) ? R.c64s[mod] : 0;
    lc.lift_mod = (LOAD == LOAD_I64_MONT) ? R.c64[mod] : B.lift_mod;
    lc.qd = R.qd[mod];
    lc.qinv = R.qinv_d[mod];
    lc.c30 = R.c30_d[mod];
    lc.c30q = R.c30_q[mod];
    lc.c64d = lc.c64q = 0.0;
    lc.wide = (q >> 41) != 0;
    // wide: 2q - (2^59 mod q) keeps the lifted value positive; otherwise the offset is just -(2^59 mod q)
    lc.k59 = lc.wide ? R.k59_d[mod] : __dsub_rn(R.k59_d[mod], __dadd_rn(lc.qd, lc.qd));
    if (LOAD == LOAD_I64_MONT) {
        const double* ec = R.enc_consts + (size_t)mod * ENC_CONSTS;
        lc.c30 = __ldg(ec);
        lc.c30q = __ldg(ec + 1);
        lc.c64d = __ldg(ec + 2);
        lc.c64q = __ldg(ec + 3);
        lc.k59 = __ldg(ec + 4);
    }
    u64 qs = ~(u64)0;
    if (LOAD == LOAD_REDUCE && B.src_digits) {      // the prime the source digit belongs to
        u32 s_hi, s_lo;
        split_index(o, R.r, B.o_div == R.r ? B.o_div_magic : 0u, s_hi, s_lo);
        qs = R.q[s_lo];
    }
    lc.src_small = LOAD == LOAD_I64_MONT ? R.dp[mod] && (q >> 39) : qs <= q + (q >> 1);
    lc.src_fp = LOAD == LOAD_I64_MONT ? R.dp[mod] != 0 : qs < (1ull << 51);
    lc.staged_fp = false;
    return lc;
}

template <bool TAIL>
__device__ __forceinline__ u64* batch_dst(const PolyBatch& B, u32 o, u32 m) {
    if (TAIL && B.tail_m && m >= B.tail_m) return B.tail_dst + (size_t)o * B.tail_so + (size_t)(m - B.tail_m) * B.dst_sm;
    return B.dst + (size_t)o * B.dst_so + (size_t)m * B.dst_sm;
}
// the same for a source of an ingest batch (PolyBatch::ingest) and its target m
__device__ __forceinline__ u64* ingest_dst(const RingDev& R, const PolyBatch& B, u32 o_hi, u32 o_lo, u32 m) {
    const size_t set = (size_t)(o_hi >> 1) * R.r + o_lo;
    return o_hi & 1 ? B.dst + set * B.dst_so + (size_t)m * B.dst_sm : B.tail_dst + set * R.N;
}

// Rows of the exchange buffer of a strided tile.  Tiles of 8 columns (64 bytes a row) swap the rows of a pair by bit 2 of the
// row number, so that the two rows a half-warp touches never share banks, whether they are neighbours or 4 apart.  Row base +
// i * step of a set then lies at (i odd ? odd : even) + i * step: two numbers per set, the rest are immediate offsets.
template <int LOG_LANES>
__device__ __forceinline__ void exchange_rows(int base, int log_step, int& even, int& odd) {
    even = odd = base;
    if (LOG_LANES != 3) return;
    if (log_step > 2) even = odd = base ^ ((base >> 2) & 1);        // (bit 2 does not depend on i)
    else if (log_step == 2) odd = base ^ 1;                         // (bit 2 of the row is bit 0 of i)
    else { even += (base >> 2) & 1; odd -= (base >> 2) & 1; }       // (sets of 4 adjacent rows)
}

// Strided pass: transforms the 2^LOG_R rows (stride 256) of a tile of adjacent columns.  Forward: first pass (reads the
// batch source through the load functor, or from `staged`, [row][column], where several target primes of the same block
// read it).  Inverse: second pass (in place, scales by N^{-1}).  tws: the prime's first 2^LOG_R twiddles, in shared memory.
template <bool FWD, int LOAD, int LOG_R, int LOG_LANES, int PATH, bool STAGED = false, bool INGEST = false>
__device__ __forceinline__ void strided_body(const RingDev& R, const PolyBatch& B, u64* sm_raw, u64* tws, u32 o,
                                             u32 m, u32 mod, u32 tile, const LoadConsts& lc, const u64* staged,
                                             const StridedTwiddles<LOG_R>& tw) {
    typedef StridedGeo<LOG_R, LOG_LANES> G;
    typedef typename Elem<PATH>::T T;
    constexpr int LEN = G::LEN, LANES = G::LANES, NT = G::NT, NG = n_groups(LOG_R);
    T* sm = (T*)sm_raw;
    const ModConsts c(R, mod);
    u64* dst = nullptr;
    if constexpr (INGEST) {
        u32 o_hi, o_lo;
        split_index(o, B.o_div, B.o_div_magic, o_hi, o_lo);
        dst = ingest_dst(R, B, o_hi, o_lo, m) + tile * LANES;
    } else {
        dst = batch_dst<!FWD>(B, o, m) + tile * LANES;
    }
    const char* src = nullptr;
    if constexpr (FWD && !STAGED) {
        u32 o_hi = 0, o_lo = o;
        if (B.o_div) split_index(o, B.o_div, B.o_div_magic, o_hi, o_lo);
        const size_t src_off = B.o_div ? (size_t)o_hi * B.src_so2 + (size_t)o_lo * B.src_so : (size_t)o * B.src_so;
        src = (const char*)B.src + (src_off + (size_t)m * B.src_sm + tile * LANES) * 8;
    }
    const int tid = threadIdx.x;
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) {
        const int fg = FWD ? gi : NG - 1 - gi;                 // group index in forward order
        const int K = group_k(LOG_R, fg);
        const int log_step = group_log_step(LOG_R, fg), step = 1 << log_step;
        const u32 base0 = (u32)(LEN >> (log_step + K));        // blocks at the group's first forward stage
        const int nsets = (LEN * LANES) >> K;
        const bool g_first = (gi == 0), g_last = (gi == NG - 1);
#pragma unroll
        for (int w0 = 0; w0 < nsets; w0 += NT) {
            const int w = w0 + tid;
            if (NT > nsets && w >= nsets) break;
            const int lane = w & (LANES - 1), u = w >> LOG_LANES;
            const int blk = u >> log_step, off = u & (step - 1);
            const int base = (blk << (log_step + K)) + off;
            int even, odd;
            exchange_rows<LOG_LANES>(base, log_step, even, odd);
            T* const sm_even = sm + even * LANES + lane;
            T* const sm_odd = sm + odd * LANES + lane;
            T e[8];
#pragma unroll
            for (int i = 0; i < (1 << K); ++i) {
                const int row = base + i * step;
                if (g_first) {
                    const size_t gidx = ((size_t)row << LOG_C) + lane;
                    if (FWD) {
                        const void* from = STAGED ? (const void*)staged : (const void*)src;
                        const size_t at = STAGED ? (size_t)(row * LANES + lane) : gidx;
                        if constexpr (PATH != PATH_INT) e[i] = load_src_fp<LOAD>(from, at, lc);
                        else e[i] = load_src<LOAD>(from, at, lc);
                    } else {
                        e[i] = ((const T*)dst)[gidx];
                    }
                } else {
                    e[i] = (i & 1 ? sm_odd : sm_even)[i * step * LANES];
                }
            }
            if (!STAGED && g_first && w0 == 0) {    // (the first sweep of the first group is full for every geometry)
                static_assert(NT <= (G::POINTS >> group_k(LOG_R, FWD ? 0 : NG - 1)), "first sweep must be full");
                tw.put(tws, PATH);
                __syncthreads();
            }
            if (K == 3) set_butterflies<3, FWD, PATH, true>(e, tws, base0 + blk, c);
            else if (K == 2) set_butterflies<2, FWD, PATH, true>(e, tws, base0 + blk, c);
            else set_butterflies<1, FWD, PATH, true>(e, tws, base0 + blk, c);
            if (!FWD && !g_last) centre_sums<1, PATH>(e, c);
#pragma unroll
            for (int i = 0; i < (1 << K); ++i) {
                const int row = base + i * step;
                if (g_last) {
                    const size_t gidx = ((size_t)row << LOG_C) + lane;
                    if (FWD) {
                        ((T*)dst)[gidx] = e[i];                 // lazy; the contiguous pass finishes
                    } else {                                    // scale by N^{-1}, to [0, q)
                        const bool mont = B.from_mont != 0;
                        u64 out;
                        if constexpr (PATH != PATH_INT) {
                            const double nv = mont ? R.ninvm_d[mod] : R.ninv_d[mod];
                            const double nq = mont ? R.ninvm_q[mod] : R.ninv_q[mod];
                            double v;
                            if (PATH == PATH_WIDE) {
                                v = __dadd_rn(fp_mul_centred(e[i], nv, nq, c.qd), c.qd);
                                if (v >= c.qd) v = __dsub_rn(v, c.qd);
                                if (v >= c.qd) v = __dsub_rn(v, c.qd);  // (the product can touch 2q for the 50-bit prime)
                            } else {
                                v = fp_mul_centred_signed(e[i], nv, nq, c.qd);
                                if (v < 0.0) v = __dadd_rn(v, c.qd);
                            }
                            out = d2u(v);
                        } else {
                            out = mul_shoup(e[i], mont ? R.ninv_m[mod] : R.ninv[mod], mont ? R.ninv_ms[mod] : R.ninvs[mod], c.q);
                        }
                        if (B.store_centred == 1 || (B.store_centred == 2 && mod == R.r))
                            out = (out > (c.q - 1) / 2 ? out - c.q : out) + (1ull << 59);
                        dst[gidx] = out;
                    }
                } else {
                    (i & 1 ? sm_odd : sm_even)[i * step * LANES] = e[i];
                }
            }
        }
        if (!g_last) __syncthreads();
    }
}

// Blocks are dealt out in grid order: the last slot (the special prime, where a batch has it, on the long integer path) goes
// first, so that nothing waits for its blocks at the end of the launch.
__device__ __forceinline__ u32 slot_of_block(u32 y, u32 n_m) { return n_m - 1 - y; }
// modulus index of slot m of a batch (n_m <= 2 * mod_wrap in every batch that wraps)
template <bool TAIL>
__device__ __forceinline__ u32 batch_modulus(const RingDev& R, const PolyBatch& B, u32 m) {
    if (TAIL && B.tail_m && m >= B.tail_m) return R.r;
    return B.mod0 + ((B.mod_wrap && m >= B.mod_wrap) ? m - B.mod_wrap : m) * B.mod_step;
}
// a digit in its own prime (o = set * r + digit with digit == mod), which ModUp does not transform
__device__ __forceinline__ bool own_prime(const RingDev& R, const PolyBatch& B, u32 o, u32 mod) {
    if (!B.skip_diag || mod >= R.r) return false;
    u32 hi, lo;
    split_index(o, R.r, B.o_div == R.r ? B.o_div_magic : 0u, hi, lo);
    return lo == mod;
}

// a residue in the form the inner products read (see RingDev::dp)
__device__ __forceinline__ u64 operand_word(const RingDev& R, u32 mod, u64 v) {
    return R.dp[mod] ? (u64)__double_as_longlong(u2d(v)) : v;
}

// grid: x = tile, y = slot m, z = outer index.
template <bool FWD, int LOAD, int LOG_R, int LOG_LANES>
__global__ void __launch_bounds__(StridedGeo<LOG_R, LOG_LANES>::NT, StridedGeo<LOG_R, LOG_LANES>::BLOCKS)
ntt_strided(const RingDev R, const PolyBatch B, u32 n_outer) {
    typedef StridedGeo<LOG_R, LOG_LANES> G;
    __shared__ __align__(16) u64 sm[n_groups(LOG_R) > 1 ? G::POINTS : 1];
    __shared__ __align__(16) u64 tws[G::TW_WORDS];
    grid_dependency_enter();
    const u32 m = slot_of_block(blockIdx.y, B.n_m), mod = batch_modulus<!FWD>(R, B, m);
    const int path = path_of(R, mod);
    StridedTwiddles<LOG_R> tw;
    tw.fetch(R, FWD, path, mod);
    for (u32 o = blockIdx.z; o < n_outer; o += gridDim.z) {
        if (FWD && own_prime(R, B, o, mod)) continue;
        const LoadConsts lc = load_consts<LOAD>(R, B, o, mod);
        if (path == PATH_DP) strided_body<FWD, LOAD, LOG_R, LOG_LANES, PATH_DP>(R, B, sm, tws, o, m, mod, blockIdx.x, lc, nullptr, tw);
        else if (path == PATH_WIDE) strided_body<FWD, LOAD, LOG_R, LOG_LANES, PATH_WIDE>(R, B, sm, tws, o, m, mod, blockIdx.x, lc, nullptr, tw);
        else strided_body<FWD, LOAD, LOG_R, LOG_LANES, PATH_INT>(R, B, sm, tws, o, m, mod, blockIdx.x, lc, nullptr, tw);
        if (o + gridDim.z < n_outer) __syncthreads();
    }
}

// Forward strided pass of a batch whose n_m target primes all read the same source polynomial (ModUp digits,
// the P-residues of ModDown): a block stages the source tile in shared memory once and transforms it
// into targets m_begin .. m_begin + m_count - 1, so the source crosses L2 once per block instead of once per
// target (and a digit is made, or converted to fp64, once).  grid: x = tile, y = outer index o, z = slice of the targets.
template <int LOAD_MODE, int LOG_R, int LOG_LANES>
__global__ void __launch_bounds__(StridedGeo<LOG_R, LOG_LANES>::NT, StridedGeo<LOG_R, LOG_LANES>::BLOCKS)
ntt_strided_shared_src(const RingDev R, const PolyBatch B, u32 m_per_block) {
    constexpr bool INGEST = LOAD_MODE == LOAD_INGEST;
    constexpr int LOAD = INGEST ? LOAD_REDUCE : LOAD_MODE;
    typedef StridedGeo<LOG_R, LOG_LANES> G;
    constexpr int LANES = G::LANES, POINTS = G::POINTS, NT = G::NT;
    extern __shared__ __align__(16) u64 shared_src_smem[];
    u64* staged = shared_src_smem;                  // [POINTS] source: doubles where staged_fp, else raw words
    u64* sm = shared_src_smem + POINTS;             // [POINTS] exchange between stage groups
    u64* tws = sm + POINTS;                         // [2][TW_WORDS] twiddles of the current and the next target
    grid_dependency_enter();
    const u32 o = blockIdx.y, tile = blockIdx.x;
    u32 o_hi = 0, o_lo = o;
    if (B.o_div) split_index(o, B.o_div, B.o_div_magic, o_hi, o_lo);
    u32 m_begin = slot_of_block(blockIdx.z, gridDim.z) * m_per_block;
    u32 m_end = min(B.n_m, m_begin + m_per_block);
    if (INGEST && !(o_hi & 1)) {                  // component 0: into its own prime only
        if (o_lo < m_begin || o_lo >= m_end) return;
        m_begin = o_lo;
        m_end = o_lo + 1;
    }
    StridedTwiddles<LOG_R> tw;
    tw.fetch(R, true, path_of(R, batch_modulus<false>(R, B, m_begin)), batch_modulus<false>(R, B, m_begin));
    // digits of primes on the fp64 path are staged as doubles
    bool staged_fp = LOAD == LOAD_REDUCE && B.src_digits && B.o_div == R.r && R.fp_ok[o_lo];
    {
        const size_t src_off = B.o_div ? (size_t)o_hi * B.src_so2 + (size_t)o_lo * B.src_so : (size_t)o * B.src_so;
        const u64* src = (const u64*)B.src + src_off + tile * LANES;
        auto at = [&](int w) { return ((size_t)(w / LANES) << LOG_C) + (w % LANES); };
        if (B.div_t) {
            // the digit is a division by P away: (source - t) * P^{-1} modulo the digit's own prime, t the centred lift
            // of the polynomial's residue modulo P (exact: same value as dividing in the transform domain)
            const u32 i = o_lo;
            LoadConsts dc;
            dc.q = R.q[i];
            dc.mu = R.mu[i];
            dc.lift_mod = R.q[R.r];
            const u64* tp = B.div_t + (size_t)o_hi * B.div_so + tile * LANES;
            if (R.fp_ok[i]) {
                // in fp64 (every value an exact integer): t lazily reduced by the load functor, the difference times
                // P^{-1} as a centred product, brought to [0, q) -- the digit must be the canonical residue, since it is
                // reduced into the other primes next
                const double qd = R.qd[i], pv = R.pinv_d[i], pq = R.pinv_q[i];
                dc.qd = qd;
                dc.c30 = R.c30_d[i];
                dc.c30q = R.c30_q[i];
                dc.wide = (dc.q >> 41) != 0;
                dc.k59 = dc.wide ? R.k59_d[i] : __dsub_rn(R.k59_d[i], __dadd_rn(qd, qd));
                const double q3 = __dadd_rn(__dadd_rn(qd, qd), qd);
#pragma unroll 4
                for (int k = 0; k < POINTS / NT; ++k) {
                    const int w = threadIdx.x + k * NT;
                    const double t = load_src_fp<LOAD_CENTRED>(tp, at(w), dc);     // (-1.75q, 0.76q), or (0.25q, 2.76q) when wide
                    const double x = __dsub_rn(u2d(src[at(w)]), t);
                    double s2 = dc.wide ? fp_mul_centred(__dadd_rn(x, q3), pv, pq, qd) : fp_mul_centred_signed(x, pv, pq, qd);
                    if (s2 < 0.0) s2 = __dadd_rn(s2, qd);
                    staged[w] = staged_fp ? (u64)__double_as_longlong(s2) : d2u(s2);
                }
            } else {
                dc.lift_red = barrett64(dc.lift_mod, dc.q, dc.mu);
                const u64 pinv = R.pinv[i], pinvs = R.pinvs[i];
                for (int w = threadIdx.x; w < POINTS; w += NT) {
                    const u64 t = load_src<LOAD_CENTRED>(tp, at(w), dc);
                    staged[w] = mul_shoup(sub_mod(src[at(w)], t, dc.q), pinv, pinvs, dc.q);
                }
            }
        } else if constexpr (LOAD == LOAD_I64_MONT) {
            // encoded coefficients: 64-bit integers, or 32-bit ones (src32).  Nearly all are small: a tile whose largest is
            // below 2^40 is staged as doubles, which the primes below that take as they are
            i64 v[POINTS / NT];
            bool big = false;
            if (B.src32) {
                const int* src4 = (const int*)B.src + src_off + tile * LANES;
#pragma unroll
                for (int k = 0; k < POINTS / NT; ++k) v[k] = src4[at(threadIdx.x + k * NT)];
            } else {
#pragma unroll
                for (int k = 0; k < POINTS / NT; ++k) v[k] = (i64)src[at(threadIdx.x + k * NT)];
#pragma unroll
                for (int k = 0; k < POINTS / NT; ++k) big = big || (u64)(v[k] + (1ll << 40)) >> 41;
                big = __syncthreads_or(big) != 0;
            }
            staged_fp = !big;
#pragma unroll
            for (int k = 0; k < POINTS / NT; ++k) staged[threadIdx.x + k * NT] = big ? (u64)v[k] : (u64)__double_as_longlong(i2d(v[k]));
        } else {
            u64 v[POINTS / NT];
#pragma unroll
            for (int k = 0; k < POINTS / NT; ++k) v[k] = src[at(threadIdx.x + k * NT)];
#pragma unroll
            for (int k = 0; k < POINTS / NT; ++k) staged[threadIdx.x + k * NT] = staged_fp ? (u64)__double_as_longlong(u2d(v[k])) : v[k];
        }
    }
    u32 buf = 0;
    for (u32 m = m_begin; m < m_end; ++m) {
        const u32 mod = batch_modulus<false>(R, B, m);
        const int path = path_of(R, mod);
        u64* tw_now = tws + buf * G::TW_WORDS;
        tw.put(tw_now, path);
        __syncthreads();            // (also: the source is staged, and the exchange buffer is free again)
        if (m + 1 < m_end) tw.fetch(R, true, path_of(R, batch_modulus<false>(R, B, m + 1)), batch_modulus<false>(R, B, m + 1));
        buf ^= 1;
        if (own_prime(R, B, o, mod)) continue;      // (its transform exists already)
        LoadConsts lc = load_consts<LOAD>(R, B, o, mod);
        lc.staged_fp = staged_fp;
        if (path == PATH_DP) strided_body<true, LOAD, LOG_R, LOG_LANES, PATH_DP, true, INGEST>(R, B, sm, tw_now, o, m, mod, tile, lc, staged, tw);
        else if (path == PATH_WIDE) strided_body<true, LOAD, LOG_R, LOG_LANES, PATH_WIDE, true, INGEST>(R, B, sm, tw_now, o, m, mod, tile, lc, staged, tw);
        else strided_body<true, LOAD, LOG_R, LOG_LANES, PATH_INT, true, INGEST>(R, B, sm, tw_now, o, m, mod, tile, lc, staged, tw);
    }
}

// Shared-memory index swizzle for a 256-point chunk of 64-bit words: makes the three access
// patterns of the contiguous pass (spacing 32, spacing 4 and 4 adjacent points per thread) free of
// bank conflicts without padding.
__host__ __device__ constexpr int swz(int i) { return i ^ ((i >> 4) & 3) ^ (((i >> 5) & 3) << 2); }

// The swizzle is linear over GF(2): swz(t ^ k) = swz(t) ^ swz(k).  Every access of the contiguous pass has
// index t ^ k with t depending on the thread and k on the unrolled loop counter, in disjoint bit fields, so
// its byte address is (A ^ 8 * (swz(k) & 15)) + 8 * (swz(k) & ~15) with A = slice base + 8 * swz(t) computed
// once per group: one logic operation and an immediate offset per access.  (The swizzle only changes the low
// four index bits, and t has no bits where swz(k) & ~15 has any.)  The slice base is 128-byte aligned.
template <int K_INDEX>
__device__ __forceinline__ void swz_store(u32 a_thread, u64 v) {
    constexpr int S = swz(K_INDEX);
    asm volatile("st.shared.b64 [%0+%1], %2;" ::"r"(a_thread ^ (u32)(8 * (S & 15))), "n"(8 * (S & ~15)), "l"(v));
}
template <int K_INDEX>
__device__ __forceinline__ void swz_store(u32 a_thread, double v) {
    swz_store<K_INDEX>(a_thread, (u64)__double_as_longlong(v));
}
template <int K_INDEX>
__device__ __forceinline__ void swz_load(u32 a_thread, u64& v) {
    constexpr int S = swz(K_INDEX);
    asm volatile("ld.shared.b64 %0, [%1+%2];" : "=l"(v) : "r"(a_thread ^ (u32)(8 * (S & 15))), "n"(8 * (S & ~15)));
}
template <int K_INDEX>
__device__ __forceinline__ void swz_load(u32 a_thread, double& v) {
    u64 bits;
    swz_load<K_INDEX>(a_thread, bits);
    v = __longlong_as_double((long long)bits);
}
// e[i] <-> slice[swz(t ^ (i << SHIFT))] for i < COUNT
template <int COUNT, int SHIFT, typename T, int I = 0>
__device__ __forceinline__ void swz_store_set(u32 a_thread, const T (&e)[8]) {
    if constexpr (I < COUNT) {
        swz_store<(I << SHIFT)>(a_thread, e[I]);
        swz_store_set<COUNT, SHIFT, T, I + 1>(a_thread, e);
    }
}
template <int COUNT, int SHIFT, typename T, int I = 0>
__device__ __forceinline__ void swz_load_set(u32 a_thread, T (&e)[8]) {
    if constexpr (I < COUNT) {
        swz_load<(I << SHIFT)>(a_thread, e[I]);
        swz_load_set<COUNT, SHIFT, T, I + 1>(a_thread, e);
    }
}

// Contiguous pass: a warp, or a block of 64 threads, transforms one chunk of 256 adjacent points (8 or 4 per thread, see
// contig_forward_far); the chunk lives in a swizzled slice of shared memory between groups.
// What bounds it: nothing alone.  In a launch of 1024 transforms modulo primes below 2^41 a chunk takes 255 cycles of an SM,
// with 691 warp instructions (68 % of the issue slots), 324 of them fp64 (64 % of that pipe) and about 165 wavefronts of the
// L1 pipe (65 %); small launches are bound by the latency of one chunk.
// Forward: second pass (final reduction to [0, q), then the store functors).  Inverse: first pass
// (reads the batch source: plain residues or tiled/limb-split plaintexts).
// TILED: the transform-domain side of the batch lives in the tile-major plaintext cache (B.tile_ptr).
// EPI: 0 = none; 1 = division by P per rotation (see ModDownEpilogue); 4 = output assembly (see OutputAssembly); 5 = ingest
// (see PolyBatch): the digits into the operand array (lazy doubles modulo primes of class OP_DP), component c of the inputs times P into lift_ptr.
struct NoEpilogue {};
struct RotationDivision {
    ModDownEpilogue e;
    RotBatch rb;
};
template <int EPI> struct EpiArg { typedef NoEpilogue T; };
template <> struct EpiArg<1> { typedef RotationDivision T; };
template <> struct EpiArg<4> { typedef OutputAssembly T; };
constexpr int CONTIG_THREADS = 128, CONTIG_WARPS = CONTIG_THREADS / 32;
// Forward launches of up to that many chunks: see ntt_contig_short.  Plain forward launches over 6 primes of 40 bits, one of 50 and
// one of 60 (N = 2^15), with 4 and with 8 points a thread: 7168 chunks 15.1 and 15.0 us, 10240 19.0 and 18.4, 13312 22.8 and 21.3,
// 17408 27.1 and 25.8, 23552 33.3 and 31.4; on a ring of 2^12 8000 17.3 and 18.2, 10944 21.0 and 21.1, 13952 25.1 and 24.6.
// Whole calls do not tell lines from 7000 to 40000 apart (within 1 % but for 768 -> 2304 without flags: 477, 485, 485 us).
constexpr size_t CONTIG_SHORT_CHUNKS = 12000;

__device__ __forceinline__ u64 word_of(u64 v) { return v; }
__device__ __forceinline__ u64 word_of(double v) { return (u64)__double_as_longlong(v); }
// a point of the forward transform, brought to [0, q)
template <int PATH, typename T>
__device__ __forceinline__ u64 canonical(T x, const ModConsts& c) {
    if constexpr (PATH == PATH_WIDE) {
        return d2u(fp_reduce(x, c.qd, c.qinv));
    } else if constexpr (PATH == PATH_DP) {
        return d2u(fp_canonical(x, c.qd, c.qinv));
    } else {
        x = reduce_16q(x, c);
        if (x >= 2 * c.q) x -= 2 * c.q;
        return x >= c.q ? x - c.q : x;
    }
}

// v * P modulo q_m, v in [0, q_m)
__device__ __forceinline__ u64 times_p(const RingDev& R, u32 m, u64 v) {
    u64 hi = 0, lo = 0;
    mac128(hi, lo, v, R.pmod[m]);
    return reduce128(hi, lo, R.q[m], R.mu[m], R.c64[m], R.c64s[m]);
}

// All but the last group of the forward pass over one chunk; the chunk is left in its slice for the last, whose sets are the
// 4 adjacent points at swizzled index 4 (lane + 32 it).
// THREADS threads a chunk: 32 with 8 points each and groups {3,3,2}, or 64 with 4 points and groups of 2.
template <int PATH, int THREADS = 32, typename T>
__device__ __forceinline__ void contig_forward_far(const T* gsrc, u32 slice, int lane, const void* tw, u32 mult, const ModConsts& c) {
    if constexpr (THREADS == 64) {
        const u32 a0 = slice + 8u * (u32)swz(lane), a1 = slice + 8u * (u32)swz((lane >> 4) * 64 + (lane & 15)),
                  a2 = slice + 8u * (u32)swz((lane >> 2) * 16 + (lane & 3));
        T e[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) e[i] = gsrc[lane + 64 * i];
        set_butterflies<2, true, PATH, false>(e, tw, mult, c);
        swz_store_set<4, 6>(a0, e);
        __syncthreads();
        swz_load_set<4, 4>(a1, e);
        set_butterflies<2, true, PATH, false>(e, tw, 4u * mult + (lane >> 4), c);
        swz_store_set<4, 4>(a1, e);
        __syncthreads();
        swz_load_set<4, 2>(a2, e);
        set_butterflies<2, true, PATH, false>(e, tw, 16u * mult + (lane >> 2), c);
        swz_store_set<4, 2>(a2, e);
        __syncthreads();
        return;
    }
    const u32 a_far = slice + 8u * (u32)swz(lane);                                    // points lane + 32 i
    const u32 a_mid = slice + 8u * (u32)swz((lane >> 2) * 32 + (lane & 3));           // points base + 4 i
    T e[8];
    // group 0: K = 3, spacing 32
#pragma unroll
    for (int i = 0; i < 8; ++i) e[i] = gsrc[lane + 32 * i];
    set_butterflies<3, true, PATH, false>(e, tw, mult, c);
    swz_store_set<8, 5>(a_far, e);
    __syncwarp();
    // group 1: K = 3, spacing 4
    swz_load_set<8, 2>(a_mid, e);
    set_butterflies<3, true, PATH, false>(e, tw, 8u * mult + (lane >> 2), c);
    swz_store_set<8, 2>(a_mid, e);
    __syncwarp();
}

// (THREADS: see contig_forward_far; the inverse pass always has 64)
template <bool FWD, int EPI, int PATH, bool TILED, int THREADS>
__device__ __forceinline__ void contig_body(const RingDev& R, const PolyBatch& B, u64* sm_raw, u32 o, u32 m, u32 mod,
                                            u32 chunk, int lane, const typename EpiArg<EPI>::T& epi) {
    typedef typename Elem<PATH>::T T;
    constexpr int LEN = 1 << LOG_C;
    T* sm = (T*)sm_raw;
    const ModConsts c(R, mod);
    const u64 q = c.q;
    const void* tw = twiddle_table(R, FWD, PATH, mod);
    u64* dst = EPI == 5 && m > R.r ? B.tail_dst + (size_t)o * R.N : batch_dst<EPI == 4>(B, o, m);
    const u64* src = FWD ? dst : (const u64*)B.src + (size_t)o * B.src_so + (size_t)m * B.src_sm;
    const u32 mult = (R.N >> LOG_C) + chunk;                   // twiddle index multiplier of this chunk
    const u64* gsrc = src + (size_t)chunk * LEN;
    u64* gdst = dst + (size_t)chunk * LEN;
    T e[8];
    const bool dp = R.dp[mod] != 0;         // (the operand arrays hold this prime's words as doubles)
    (void)dp;
    // where the thread's words lie in the tile-major plaintext cache: points 4 lane.., and 128 further on
    unsigned char* tile_stage = nullptr;
    size_t tile_step = 0;
    u32 tile_at = 0, tile_fmt = 0, tile_high = 0;
    if constexpr (TILED) {
        const u32 d = B.o_base + o, pj_all = d / B.tile.n_terms, term = d - pj_all * B.tile.n_terms, pj = pj_all - B.tile_pj0;
        const u32 n = chunk * LEN + 4 * lane;
        tile_stage = (unsigned char*)B.tile_ptr + tile_stage_of_word(B.tile, pj, term, mod, n);
        tile_fmt = tile_format(B.tile, mod);
        tile_at = tile_word_offset(B.tile, tile_fmt, pj, term, n);
        tile_high = tile_high_offset(B.tile, pj, term, n);
        tile_step = (size_t)((128u >> B.tile.log_tn) * B.tile.G * B.tile.C) * tile_stage_bytes(B.tile, tile_fmt);
    }
    // byte addresses (shared window) of the thread's base points
    const u32 slice = (u32)__cvta_generic_to_shared(sm);
    const u32 a_near = slice + 8u * (u32)swz(4 * lane);                               // points 4 (lane + 32 it) + i
    if (FWD) {
        contig_forward_far<PATH, THREADS>((const T*)gsrc, slice, lane, tw, mult, c);
        // last group: K = 2, adjacent points; two sets per thread
#pragma unroll
        for (int it = 0; it < 64 / THREADS; ++it) {
            const int s = lane + 32 * it;
            swz_load_set<4, 0>(a_near + (u32)(it * 8 * swz(128)), e);      // (swz(128) = 128: above the bits of 4 * lane)
            // the epilogue's operands do not depend on the transform: ask for them before the last butterflies
            u64 uu[4] = {0, 0, 0, 0}, cc[4] = {0, 0, 0, 0};
            u32 pp[4] = {0, 0, 0, 0};
            if constexpr (EPI == 1) {
                const u32 rot = o >> 1, comp = o & 1, ip = mod, nb = R.r + 1;
                const size_t n = (size_t)chunk * LEN + 4 * s;
                const u64* up = epi.e.u + ((size_t)o * nb + ip) * R.N + n;
                const ulonglong2 u0 = *(const ulonglong2*)up, u1 = *(const ulonglong2*)(up + 2);
                uu[0] = u0.x; uu[1] = u0.y; uu[2] = u1.x; uu[3] = u1.y;
                if (comp == 0) {
                    const u64* cp = epi.e.c0_base + (size_t)epi.rb.c0[rot] * epi.e.c0_stride + (size_t)ip * R.N + n;
                    const ulonglong2 c0 = *(const ulonglong2*)cp, c1 = *(const ulonglong2*)(cp + 2);
                    cc[0] = c0.x; cc[1] = c0.y; cc[2] = c1.x; cc[3] = c1.y;
                }
                const uint4 pv = *(const uint4*)(epi.e.pinv + (size_t)epi.rb.key[rot] * R.N + n);
                pp[0] = pv.x; pp[1] = pv.y; pp[2] = pv.z; pp[3] = pv.w;
            }
            set_butterflies<2, true, PATH, false>(e, tw, 64u * mult + s, c);
            // (what is stored as doubles stays lazy: see LAZY_DIGITS)
            u64 v4[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) v4[i] = EPI == 5 && PATH == PATH_DP ? word_of(e[i]) : canonical<PATH>(e[i], c);
            if constexpr (EPI == 5 && PATH == PATH_DP) {
                if (!dp) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v4[i] = canonical<PATH>(e[i], c);
                }
            }
            if constexpr (EPI == 5) {
                const u32 n = chunk * LEN + 4 * s, nbp = R.r + 1;
                u32 q_in, j;
                split_index(o, B.dtile_div, B.dtile_magic, q_in, j);
                if (m <= R.r) stg4(B.dtile_ptr + ks_tile_base(R.N, nbp, R.r, q_in, j, m) + (size_t)(n / KS_TILE) * R.r * KS_TILE + n % KS_TILE, v4[0], v4[1], v4[2], v4[3]);
                if (mod == j) {             // its own prime: the un-rotated input, times P
                    u64 p4[4];                  // (the multiply-accumulate, which reads them, takes doubles where it takes digits as such)
                    const double pd = u2d(R.pmod[mod]), pq = __dmul_rn(pd, c.qinv);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        p4[i] = dp ? (u64)__double_as_longlong(fp_mul_centred_signed(__longlong_as_double((long long)v4[i]), pd, pq, c.qd)) : times_p(R, mod, v4[i]);
                    stg4(B.lift_ptr + (size_t)q_in * B.lift_so + ((size_t)(m <= R.r ? nbp : 0u) + mod) * R.N + n, p4[0], p4[1], p4[2], p4[3]);
                }
                continue;
            }
            if constexpr (EPI == 1) {
                const u32 rot = o >> 1, comp = o & 1, ip = mod, r = R.r;
                u64* op = epi.e.out_base + (size_t)epi.rb.out[rot] * epi.e.out_stride + ((size_t)comp * r + ip) * R.N;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    u64 v = mul_shoup(sub_mod(uu[i], v4[i], q), R.pinv[ip], R.pinvs[ip], q);
                    v = add_mod(v, cc[i], q);
                    op[pp[i]] = v;
                }
                continue;
            }
            if constexpr (TILED) {   // tile-major plaintext cache; 4 adjacent coefficients never straddle a tile (tiles hold >= 16)
                unsigned char* stage = tile_stage + (size_t)it * tile_step;
                const u32 at = tile_at, fmt = tile_fmt;
                if (fmt == TILE_W64) {
                    const u32 L = q >> 50 ? LIMB_WIDE : B.split_bits;
                    stg4((u64*)(stage + at), limb_split(v4[0], L), limb_split(v4[1], L), limb_split(v4[2], L), limb_split(v4[3], L));
                } else {
                    *(uint4*)(stage + at) = make_uint4((u32)v4[0], (u32)v4[1], (u32)v4[2], (u32)v4[3]);
                    if (fmt == TILE_W40) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) stage[tile_high + 4 * i] = (unsigned char)(v4[i] >> 32);
                    }
                }
                continue;
            }
            if (B.lift_ptr) {   // P times the value, into the extended-basis copy of the un-rotated inputs
                const u32 comp = (B.mod_wrap && m >= B.mod_wrap) ? 1u : 0u, nbp = R.r + 1;    // (n_m <= 2 * mod_wrap)
                u64* xp = B.lift_ptr + (size_t)o * B.lift_so + ((size_t)comp * nbp + mod) * R.N + (size_t)chunk * LEN + 4 * s;
                u64 p4[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) p4[i] = times_p(R, mod, v4[i]);
                ((ulonglong2*)xp)[0] = make_ulonglong2(p4[0], p4[1]);
                ((ulonglong2*)xp)[1] = make_ulonglong2(p4[2], p4[3]);
                if (B.lift_zero && mod == 0) {     // the residue modulo P of P * ct is zero
                    u64* zp = B.lift_ptr + (size_t)o * B.lift_so + ((size_t)comp * nbp + R.r) * R.N + (size_t)chunk * LEN + 4 * s;
                    ((ulonglong2*)zp)[0] = make_ulonglong2(0, 0);
                    ((ulonglong2*)zp)[1] = make_ulonglong2(0, 0);
                }
            }
            if (B.scatter) {    // rotation keys: permuted by their automorphism, in the form the inner products read
                const u32* sc = B.scatter + (size_t)(o / B.scatter_div) * R.N + chunk * LEN + 4 * s;
#pragma unroll
                for (int i = 0; i < 4; ++i) key_store(R, B.dtile_ptr, o / B.scatter_div, m, o % B.scatter_div, sc[i], v4[i]);
                continue;
            }
            ulonglong2* gp = (ulonglong2*)(gdst + 4 * s);
            gp[0] = make_ulonglong2(v4[0], v4[1]);
            gp[1] = make_ulonglong2(v4[2], v4[3]);
        }
    } else {
        // inverse: groups in the opposite order
#pragma unroll
        for (int it = 0; it < 64 / THREADS; ++it) {
            const int s = lane + 32 * it;
            u64 v4[4];
            if constexpr (EPI == 4) {   // see OutputAssembly
                const u32 g1 = epi.g1, rows = epi.ext ? R.r + 1 : R.r, nu = epi.n_u();
                const size_t n = (size_t)chunk * LEN + 4 * s;
                u32 comp = 0, ju_lo = 1, ju_hi = 0, jc_lo = 1, jc_hi = 0;     // u of giant steps ju_lo..ju_hi, rotated c0 parts of jc_lo..jc_hi
                bool ident = false;
                if (mod < R.r) {
                    comp = m / R.r; ident = true; ju_hi = g1;
                    if (comp == 0) jc_hi = g1;
                } else if (m - B.tail_m < nu) {
                    const u32 mt = m - B.tail_m;
                    comp = mt & 1;
                    if (epi.each) ju_lo = ju_hi = 1 + mt / 2;
                    else ju_hi = g1;
                } else {
                    const u32 mt = m - B.tail_m - nu;
                    if (mt < 2) { comp = mt; ident = true; }
                    else jc_lo = jc_hi = mt - 1;
                }
                v4[0] = v4[1] = v4[2] = v4[3] = 0;
                // (the producers stored every rotated term through its rotation already: plain loads; the words of
                // three giant steps are requested together)
                auto add_terms = [&](const u64* base, size_t step, u32 count) {
                    for (u32 j0 = 0; j0 < count; j0 += 3) {
                        ulonglong2 a2[3], b2[3];
#pragma unroll
                        for (u32 h = 0; h < 3; ++h)
                            if (j0 + h < count) {
                                const u64* p = base + (size_t)(j0 + h) * step;
                                a2[h] = *(const ulonglong2*)p;
                                b2[h] = *(const ulonglong2*)(p + 2);
                            }
#pragma unroll
                        for (u32 h = 0; h < 3; ++h)
                            if (j0 + h < count) {
                                v4[0] = add_mod(v4[0], a2[h].x, q); v4[1] = add_mod(v4[1], a2[h].y, q);
                                v4[2] = add_mod(v4[2], b2[h].x, q); v4[3] = add_mod(v4[3], b2[h].y, q);
                            }
                    }
                };
                const u64* ap = epi.a + (size_t)o * epi.a_stride + n;
                if (ident) add_terms(ap + ((size_t)comp * rows + mod) * R.N, 0, 1);
                const size_t c_step = (size_t)epi.n_out * epi.a_stride;
                add_terms(ap + (size_t)mod * R.N + jc_lo * c_step, c_step, jc_hi + 1 - jc_lo);
                if (!epi.ext && mod < R.r) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) v4[i] = times_p(R, mod, v4[i]);
                }
                const size_t u_step = (size_t)epi.n_out * 2 * (R.r + 1) * R.N;
                add_terms(epi.u + (((size_t)o * 2 + comp) * (R.r + 1) + mod) * R.N + n + (ju_lo - 1) * u_step, u_step, ju_hi + 1 - ju_lo);
            } else if constexpr (TILED) {  // read back from the tile-major plaintext cache
                const unsigned char* stage = tile_stage + (size_t)it * tile_step;
                const u32 at = tile_at, fmt = tile_fmt;
                if (fmt == TILE_W64) {
                    const ulonglong2* gp = (const ulonglong2*)(stage + at);
                    const ulonglong2 a = gp[0], b = gp[1];
                    v4[0] = a.x; v4[1] = a.y; v4[2] = b.x; v4[3] = b.y;
                    const u32 L = q >> 50 ? LIMB_WIDE : B.split_bits;
#pragma unroll
                    for (int i = 0; i < 4; ++i) v4[i] = limb_join(v4[i], L);
                } else {
                    const uint4 lo = *(const uint4*)(stage + at);
                    v4[0] = lo.x; v4[1] = lo.y; v4[2] = lo.z; v4[3] = lo.w;
                    if (fmt == TILE_W40) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) v4[i] |= (u64)stage[tile_high + 4 * i] << 32;
                    }
                }
            } else {
                const ulonglong2* gp = (const ulonglong2*)(gsrc + 4 * s);
                const ulonglong2 a = gp[0], b = gp[1];
                v4[0] = a.x; v4[1] = a.y; v4[2] = b.x; v4[3] = b.y;
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) from_u64(e[i], v4[i]);
            set_butterflies<2, false, PATH, false>(e, tw, 64u * mult + s, c);
            swz_store_set<4, 0>(a_near + (u32)(it * 8 * swz(128)), e);
        }
        const u32 a0 = slice + 8u * (u32)swz(lane), a1 = slice + 8u * (u32)swz((lane >> 4) * 64 + (lane & 15)),
                  a2 = slice + 8u * (u32)swz((lane >> 2) * 16 + (lane & 3));
        __syncthreads();
        swz_load_set<4, 2>(a2, e);
        set_butterflies<2, false, PATH, false>(e, tw, 16u * mult + (lane >> 2), c);
        centre_sums<2, PATH>(e, c);
        swz_store_set<4, 2>(a2, e);
        __syncthreads();
        swz_load_set<4, 4>(a1, e);
        set_butterflies<2, false, PATH, false>(e, tw, 4u * mult + (lane >> 4), c);
        centre_sums<2, PATH>(e, c);
        swz_store_set<4, 4>(a1, e);
        __syncthreads();
        swz_load_set<4, 6>(a0, e);
        set_butterflies<2, false, PATH, false>(e, tw, mult, c);
        centre_sums<2, PATH>(e, c);
#pragma unroll
        for (int i = 0; i < 4; ++i) ((T*)gdst)[lane + 64 * i] = e[i];      // lazy; the strided pass finishes
    }
}

// grid: x = group of 2^log_wo outer indices, y = slot m, z = group of chunks.
template <int EPI, bool TILED>
__global__ void __launch_bounds__(CONTIG_THREADS, 8) ntt_contig(const RingDev R, const PolyBatch B, u32 n_outer, u32 log_wo,
                                                              const typename EpiArg<EPI>::T epi) {
    __shared__ __align__(128) u64 sm_all[CONTIG_WARPS << LOG_C];
    grid_dependency_enter();
    const u32 m = slot_of_block(blockIdx.y, B.n_m);
    u32 mod = batch_modulus<false>(R, B, m);
    const u32 warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const u32 o = (blockIdx.x << log_wo) + (warp & ((1u << log_wo) - 1)), chunk = blockIdx.z * (CONTIG_WARPS >> log_wo) + (warp >> log_wo);
    if (o >= n_outer || chunk >= (R.N >> LOG_C)) return;    // (whole warps leave)
    if (EPI == 5 && m > R.r) mod = o % R.r;         // (component 0, in the prime it is a residue of)
    if (own_prime(R, B, o, mod)) return;
    u64* sm = sm_all + (warp << LOG_C);
    const int path = path_of(R, mod);
    if (path == PATH_DP) contig_body<true, EPI, PATH_DP, TILED, 32>(R, B, sm, o, m, mod, chunk, lane, epi);
    else if (path == PATH_WIDE) contig_body<true, EPI, PATH_WIDE, TILED, 32>(R, B, sm, o, m, mod, chunk, lane, epi);
    else contig_body<true, EPI, PATH_INT, TILED, 32>(R, B, sm, o, m, mod, chunk, lane, epi);
}

// The same with a block of 64 threads per chunk, 4 points a thread: the inverse pass, and forward launches too small to run
// in many rounds, whose time is that of one chunk, and of the integer path's in particular.  (Forward launches of up to 12000
// chunks and all inverse ones: the calls of a 0.6B layer 1362 -> 1327 us, a 64 x 64 product on a ring of 2^12 70 -> 61 us.
// Inverse launches of a LLaMA-3-8B layer, up to 36000 chunks: 549 -> 477 us.  Forward launches of 200000 chunks: 783 us with
// 8 points, 938 us with 4, for an exchange through shared memory more.)  grid: x = outer index, y = slot m, z = chunk.
// (the output assembly runs on a few polynomials per launch and holds the operands of three giant steps at once: it trades
// resident blocks for registers)
template <bool FWD, int EPI, bool TILED>
__global__ void __launch_bounds__(64, EPI == 4 ? 10 : 16) ntt_contig_short(const RingDev R, const PolyBatch B,
                                                                        const typename EpiArg<EPI>::T epi) {
    __shared__ __align__(128) u64 sm[1 << LOG_C];
    grid_dependency_enter();
    const u32 m = slot_of_block(blockIdx.y, B.n_m), o = blockIdx.x, chunk = blockIdx.z;
    u32 mod = batch_modulus<EPI == 4>(R, B, m);
    if (EPI == 5 && m > R.r) mod = o % R.r;         // (component 0, in the prime it is a residue of)
    if (FWD && own_prime(R, B, o, mod)) return;
    const int path = path_of(R, mod), lane = threadIdx.x;
    if (path == PATH_DP) contig_body<FWD, EPI, PATH_DP, TILED, 64>(R, B, sm, o, m, mod, chunk, lane, epi);
    else if (path == PATH_WIDE) contig_body<FWD, EPI, PATH_WIDE, TILED, 64>(R, B, sm, o, m, mod, chunk, lane, epi);
    else contig_body<FWD, EPI, PATH_INT, TILED, 64>(R, B, sm, o, m, mod, chunk, lane, epi);
}

// Key-switch products (Sec. 4.2 "key-switching primitives"): the contiguous pass of the digits' transforms and their inner
// product with the rotation keys in one kernel.
//   u'[rot][comp][m][n] = sum_j NTT_m(digit j of set dig(rot))[n] * key'[key(rot)][j][comp][m][n]
// The rotation keys are stored pre-permuted by their automorphism, so the product runs in the un-rotated index space with
// coalesced operands, and the automorphism is applied once, as a scatter, when the result is stored (pinv) or when the
// rotated ciphertext is assembled.
//
// A block owns one run of rotations of the same digit set, one modulus m and cb chunks of 256 coefficients: a warp transforms
// digit w % r of chunk w / r (w = its number, then 8 more) into its slice of shared memory, then every thread takes a coefficient, multiplies the r digits
// with the 2r key words of each rotation of the run (straight from global memory: read once, coalesced) and reduces once per
// output word.  The transformed digits, r (r+1) polynomials per set, never reach memory.
// What bounds it: the key stream where the run is long (baby steps), the fp64 pipe and the latency of the transform elsewhere.
// Measured over the giant steps of the four calls of a 0.6B decoder layer (N = 2^15, r = 7, 19 rotations): 302 us, where a
// contiguous pass and an inner product of their own took 218 + 210 us; a projection's 15 baby and 9 giant rotations without
// double hoisting: 291 us instead of 110 + 224 us.
// grid: x = run, y = group of chunks, z = m: the runs that share a key's tile are adjacent.
// (three blocks of 80 registers an SM instead of four of 64: 334 instead of 302 us)
// An instance for every digit count: the key words of a component are all requested before the first is used, at immediate
// offsets.  (A loop over the digits instead, four of them at a time, on a projection of 1024 -> 2048 with N = 2^15 without
// double hoisting: 435 us for 6 digits, 800 for 10, 1394 for 15; with instances 356, 628, 1135.)  Eight warps for ten digits
// and more: as many warps as digits leave fewer blocks to an SM (15 digits, loop: 1801 us).
template <int RC>
struct InnerGeo {
    static constexpr int WARPS = RC == 9 ? 9 : 8;                           // (few digits leave room for several chunks)
    static constexpr int BLOCKS = RC == 9 ? 3 : 4;
};
template <int CLS, int RC>
__device__ __forceinline__ void inner_products(const RingDev& R, const RotBatch& rb, u32 first, u32 cnt, u32 m, u32 n, const u64* sd,
                                               const void* __restrict__ keys, u64* u, u64* xext,
                                               const u32* __restrict__ pinv, u64 pol) {
    const u32 N = R.N, r = RC, nb = r + 1;
    const u32 at = (u32)swz((int)(n & 255u));
    const size_t out_words = (size_t)2 * nb * N;
    for (u32 rot = first; rot < first + cnt; ++rot) {
        const KeyTile<CLS> kt(key_tile(R, keys, (u32)rb.key[rot], m, n / KS_TILE), n % KS_TILE, r);
        u32 dest = n;
        u64 pc0 = 0;
        if (pinv) dest = __ldg(&pinv[(size_t)rb.key[rot] * N + n]);
        if (xext) pc0 = xext[(size_t)rb.c0[rot] * out_words + (size_t)m * N + n];
        // (one component at a time: with the key words of both in registers fewer blocks fit an SM)
        u32 high[(2 * RC + 3) / 4];
#pragma unroll
        for (int h = 0; h < (2 * RC + 3) / 4; ++h) high[h] = kt.high(h, pol);
        auto component = [&](u32 comp) -> u64 {
            DigitDot<CLS> dot;
            u32 k0[RC], k1[RC];
#pragma unroll
            for (int j = 0; j < RC; ++j) kt.word(2 * j + comp, pol, k0[j], k1[j]);
#pragma unroll
            for (int j = 0; j < RC; ++j) {
                KeyTile<CLS>::cut(2 * j + comp, high[j / 2], k0[j], k1[j]);
                dot.mac(*(const uint2*)&sd[(j << LOG_C) + at], k0[j], k1[j]);
            }
            return dot.reduce(R, m, RC > LAZY_DIGITS);
        };
        const u64 v0 = component(0), v1 = component(1);
        // xext (double hoisting): the rotated input in the extended basis is (P*c0 + u0, u1) moved through the rotation's
        // permutation; P*c0 (zero modulo P) was stored as the un-rotated term
        u64* up = xext ? xext + (size_t)rb.out[rot] * out_words + (size_t)m * N + dest : u + (size_t)rb.out[rot] * out_words + (size_t)m * N + dest;
        up[0] = xext ? add_mod(v0, pc0, R.q[m]) : v0;
        up[(size_t)nb * N] = v1;
    }
}

template <int RC>
__global__ void __launch_bounds__(32 * InnerGeo<RC>::WARPS, InnerGeo<RC>::BLOCKS)
ntt_contig_inner(const RingDev R, const PolyBatch B, const RotBatch rb, const void* __restrict__ keys, u64* u, u64* xext,
                 const u32* __restrict__ pinv, u32 cb) {
    extern __shared__ __align__(128) u64 sm_all[];          // [cb][r] slices
    grid_dependency_enter();
    const u32 N = R.N, r = RC, nb = r + 1;
    const u32 m = slot_of_block(blockIdx.z, nb), chunk0 = blockIdx.y * cb;
    const u32 first = rb.grp_first[blockIdx.x], cnt = rb.grp_cnt[blockIdx.x], set = (u32)rb.dig[first];
    const u32 warps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31;
    const int path = path_of(R, m);
    const ModConsts c(R, m);
    const bool dp = R.dp[m] != 0;
    if (threadIdx.x < cb * 2 && chunk0 + threadIdx.x / 2 < (N >> LOG_C)) {      // the first rotation's keys, on their way to L2
        const unsigned char* kp = key_tile(R, keys, (u32)rb.key[first], m, chunk0 * 2 + threadIdx.x);
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(kp), "r"(key_tile_bytes(dp, r)) : "memory");
    }
    for (u32 w = threadIdx.x >> 5; w < cb * r; w += warps) {
        const u32 chunk = chunk0 + w / r, j = w % r;
        if (chunk >= (N >> LOG_C)) break;
        u64* sm = sm_all + (w << LOG_C);
        const u32 slice = (u32)__cvta_generic_to_shared(sm);
        if (B.skip_diag && j == m) {            // a digit in its own prime: its transform exists already
            const u64* ds = B.diag_src + (size_t)set * B.diag_so + (size_t)m * N + (chunk << LOG_C);
#pragma unroll
            for (int i = 0; i < 8; ++i) sm[swz(lane + 32 * i)] = operand_word(R, m, ds[lane + 32 * i]);
            continue;
        }
        const u64* gsrc = B.dst + (size_t)(set * r + j) * B.dst_so + (size_t)m * B.dst_sm + (chunk << LOG_C);
        const u32 mult = (N >> LOG_C) + chunk;
        const void* tw = twiddle_table(R, true, path, m);
        const u32 a_near = slice + 8u * (u32)swz(4 * lane);
        auto finish = [&](auto path_c, auto lazy_c) {
            constexpr int PATH = decltype(path_c)::value;
            constexpr bool LAZY = decltype(lazy_c)::value;          // (digits of class OP_DP stay lazy: see LAZY_DIGITS)
            typedef typename Elem<PATH>::T T;
            contig_forward_far<PATH>((const T*)gsrc, slice, lane, tw, mult, c);
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                T e[8];
                swz_load_set<4, 0>(a_near + (u32)(it * 8 * swz(128)), e);
                set_butterflies<2, true, PATH, false>(e, tw, 64u * mult + lane + 32 * it, c);
                u64 v[8];
#pragma unroll
                for (int i = 0; i < 4; ++i) v[i] = LAZY ? word_of(e[i]) : canonical<PATH>(e[i], c);
                swz_store_set<4, 0>(a_near + (u32)(it * 8 * swz(128)), v);
            }
        };
        if (dp) finish(std::integral_constant<int, PATH_DP>(), std::true_type());
        else if (path == PATH_DP) finish(std::integral_constant<int, PATH_DP>(), std::false_type());
        else if (path == PATH_WIDE) finish(std::integral_constant<int, PATH_WIDE>(), std::false_type());
        else finish(std::integral_constant<int, PATH_INT>(), std::false_type());
    }
    __syncthreads();
    const u64 pol = stream_policy();
    for (u32 i = threadIdx.x; i < (cb << LOG_C); i += blockDim.x) {
        const u32 n = (chunk0 << LOG_C) + i;
        if (n >= N) break;
        const u64* sd = sm_all + ((size_t)(i >> LOG_C) * r << LOG_C);
        if (dp) inner_products<OP_DP, RC>(R, rb, first, cnt, m, n, sd, keys, u, xext, pinv, pol);
        else if (R.q[m] >> 50) inner_products<OP_WIDE, RC>(R, rb, first, cnt, m, n, sd, keys, u, xext, pinv, pol);
        else inner_products<OP_NARROW, RC>(R, rb, first, cnt, m, n, sd, keys, u, xext, pinv, pol);
    }
}

// o / d by a reciprocal where the outer count allows it (see split_index)
static void set_magics(PolyBatch& B, u32 n_outer) {
    B.o_div_magic = B.dtile_magic = 0;
    if (n_outer > 65535u) return;
    if (B.o_div) B.o_div_magic = (u32)((((u64)1 << 32) + B.o_div - 1) / B.o_div);
    if (B.dtile_div) B.dtile_magic = (u32)((((u64)1 << 32) + B.dtile_div - 1) / B.dtile_div);
}

template <bool FWD, int LOAD, int LOG_R, int LOG_LANES>
static void launch_strided_t(const RingHost& ring, const PolyBatch& B_in, u32 n_polys, cudaStream_t stream) {
    typedef StridedGeo<LOG_R, LOG_LANES> G;
    PolyBatch B = B_in;
    const u32 n_outer = n_polys / B.n_m;
    set_magics(B, n_outer);
    const dim3 grid(G::TILES, B.n_m, n_outer < 65535u ? n_outer : 65535u);
    launch_dependent(ring, ntt_strided<FWD, LOAD, LOG_R, LOG_LANES>, grid, dim3(G::NT), 0, stream, ring.dev, B, n_outer);
}

template <int LOAD, int LOG_R, int LOG_LANES>
static void launch_shared_src_t(const RingHost& ring, const PolyBatch& B_in, u32 n_outer, cudaStream_t stream) {
    typedef StridedGeo<LOG_R, LOG_LANES> G;
    PolyBatch B = B_in;
    set_magics(B, n_outer);
    // targets per block: fewer blocks share the source better, but a launch lasts as long as its longest block and ends raggedly.
    // Cost = the work over the resident blocks, or one block where that is longer, and half a block for the end, unless another chain's
    // launches fill it (PolyBatch::beside); a block costs its targets and the staging of its source, a whole target's worth where that
    // divides by P (an ingest batch has half as many blocks and one of a single target for every other source).  us for 1, 2, 4, 8
    // targets a block, N = 2^15, r = 7, what is taken marked: digits of one ciphertext 15.2*, 15.7, 16.9, 20.5, of three 31.0, 29.0*, 30.7,
    // 31.1, of six 53.7, 49.6, 49.2*, 50.0, of 40 322, 284, 269, 261*; ingest of one input 13.1*, 12.7, 14.7, 18.0, of three 31.6, 29.9*,
    // 31.4, 34.9; for 1, 2, 5, 10, N = 2^16, r = 9: digits of one ciphertext 36.2, 33.1*, 33.1, 34.7, of six 174, 154, 146*, 146, ingest of
    // four inputs 134, 119, 114*, 117.  Whole calls whose giant steps run as two chains, the end counted and not: 768 -> 2304 without flags
    // 454 and 445 us, with double hoisting alone 392 and 389; 1024 -> 6144 with all flags 389 and 384.
    const double slots = 148.0 * G::BLOCKS, stage = B.div_t ? 1.0 : 0.5, tail = B.beside ? 0.0 : 0.5;
    u32 best = 1;
    double best_cost = 1e30;
    for (u32 per = 1; per <= B.n_m; ++per) {
        const u32 slices = (B.n_m + per - 1) / per;
        if ((B.n_m + slices - 1) / slices != per) continue;         // keep the slices balanced
        double work = (double)G::TILES * n_outer * slices * (per + stage) / slots;
        if (LOAD == LOAD_INGEST) work = work / 2 + (double)G::TILES * n_outer * 1.5 / 2 / slots;
        const double cost = (work > per + stage ? work : per + stage) + tail * (per + stage);
        if (cost <= best_cost) { best_cost = cost; best = per; }
    }
    const dim3 grid(G::TILES, n_outer, (B.n_m + best - 1) / best);
    constexpr size_t smem = (size_t)8 * (2 * G::POINTS + 2 * G::TW_WORDS);
    static bool attr_set[MAX_DEVICES] = {false};     // opt in once per device to more than 48 KB of dynamic shared memory
    if (smem > 48 * 1024 && !attr_set[device_slot(ring)]) {
        cudaFuncSetAttribute(ntt_strided_shared_src<LOAD, LOG_R, LOG_LANES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        attr_set[device_slot(ring)] = true;
    }
    launch_dependent(ring, ntt_strided_shared_src<LOAD, LOG_R, LOG_LANES>, grid, dim3(G::NT), smem, stream, ring.dev, B, best);
}

template <bool FWD, int LOAD>
static cudaError_t launch_strided(const RingHost& ring, const PolyBatch& B, u32 n_polys, cudaStream_t stream) {
    if (n_polys == 0) return cudaSuccess;
    ProfScope prof(ring.prof, FWD ? CAT_NTT_FWD_STRIDED : CAT_NTT_INV_STRIDED, stream);
    if constexpr (FWD && (LOAD == LOAD_REDUCE || LOAD == LOAD_CENTRED || LOAD == LOAD_INGEST || LOAD == LOAD_I64_MONT)) {
        const u32 n_outer = n_polys / B.n_m;
        if (B.src_sm == 0 && B.n_m > 1 && n_outer <= 65535) {
            switch (ring.dev.logN - LOG_C) {
                case 2: launch_shared_src_t<LOAD, 2, 8>(ring, B, n_outer, stream); break;
                case 3: launch_shared_src_t<LOAD, 3, 8>(ring, B, n_outer, stream); break;
                case 4: launch_shared_src_t<LOAD, 4, 5>(ring, B, n_outer, stream); break;
                case 5: launch_shared_src_t<LOAD, 5, 5>(ring, B, n_outer, stream); break;
                case 6: launch_shared_src_t<LOAD, 6, 5>(ring, B, n_outer, stream); break;
                case 7: launch_shared_src_t<LOAD, 7, 3>(ring, B, n_outer, stream); break;
                case 8: launch_shared_src_t<LOAD, 8, 3>(ring, B, n_outer, stream); break;
                default: return cudaErrorInvalidValue;
            }
            return cudaGetLastError();
        }
    }
    if constexpr (LOAD == LOAD_INGEST || LOAD == LOAD_I64_MONT) return cudaErrorInvalidValue;     // (always from a shared source)
    else
    // (tiles of 512 points on a ring of 2^12 and of 1024 on one of 2^13, not 2048: their launches are too small to fill the
    // GPU, and more and shorter blocks end sooner: 76 -> 70 us for a 64 x 64 product, 276 -> 267 us for 768 x 2304)
    switch (ring.dev.logN - LOG_C) {
        case 2: launch_strided_t<FWD, LOAD, 2, 8>(ring, B, n_polys, stream); break;
        case 3: launch_strided_t<FWD, LOAD, 3, 8>(ring, B, n_polys, stream); break;
        case 4: launch_strided_t<FWD, LOAD, 4, 5>(ring, B, n_polys, stream); break;
        case 5: launch_strided_t<FWD, LOAD, 5, 5>(ring, B, n_polys, stream); break;
        case 6: launch_strided_t<FWD, LOAD, 6, 5>(ring, B, n_polys, stream); break;
        case 7: launch_strided_t<FWD, LOAD, 7, 4>(ring, B, n_polys, stream); break;
        case 8: launch_strided_t<FWD, LOAD, 8, 4>(ring, B, n_polys, stream); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <bool FWD, int EPI = 0>
static cudaError_t launch_contig(const RingHost& ring, const PolyBatch& B_in, u32 n_polys, cudaStream_t stream,
                                 const typename EpiArg<EPI>::T& epi = {}) {
    if (n_polys == 0) return cudaSuccess;
    ProfScope prof(ring.prof, FWD ? CAT_NTT_FWD_CONTIG : CAT_NTT_INV_CONTIG, stream);
    PolyBatch B = B_in;
    const u32 n_outer = n_polys / B.n_m;
    set_magics(B, n_outer);
    const u32 chunks = ring.dev.N >> LOG_C;
    // the four warps of a block take the same chunk of four polynomials where the batch has enough of them (one fetch of the
    // chunk's twiddles serves them), else of two, else neighbouring chunks
    const u32 log_wo = n_outer % 4 == 0 || n_outer >= 16 ? 2u : n_outer % 2 == 0 || n_outer >= 7 ? 1u : 0u;
    const u32 per = CONTIG_WARPS >> log_wo;
    const dim3 grid((n_outer + (1u << log_wo) - 1) >> log_wo, B.n_m, (chunks + per - 1) / per), grid_short(n_outer, B.n_m, chunks);
    auto go = [&](auto tiled_c) {
        constexpr bool TILED = decltype(tiled_c)::value;
        if constexpr (FWD) {
            if ((size_t)n_polys * chunks > CONTIG_SHORT_CHUNKS) {
                launch_dependent(ring, ntt_contig<EPI, TILED>, grid, dim3(CONTIG_THREADS), 0, stream, ring.dev, B, n_outer, log_wo, epi);
                return;
            }
        }
        launch_dependent(ring, ntt_contig_short<FWD, EPI, TILED>, grid_short, dim3(64), 0, stream, ring.dev, B, epi);
    };
    if constexpr (EPI == 0) {
        if (B.tile_ptr) {
            go(std::integral_constant<bool, true>());
            return cudaGetLastError();
        }
    }
    go(std::integral_constant<bool, false>());
    return cudaGetLastError();
}

cudaError_t ntt_forward(const RingHost& ring, const PolyBatch& B, u32 n_outer, int load, cudaStream_t stream) {
    const u32 n_polys = n_outer * B.n_m;
    cudaError_t e;
    if (load == LOAD_PLAIN) e = launch_strided<true, LOAD_PLAIN>(ring, B, n_polys, stream);
    else if (load == LOAD_REDUCE) e = launch_strided<true, LOAD_REDUCE>(ring, B, n_polys, stream);
    else if (load == LOAD_I64) e = launch_strided<true, LOAD_I64>(ring, B, n_polys, stream);
    else if (load == LOAD_I64_MONT) e = launch_strided<true, LOAD_I64_MONT>(ring, B, n_polys, stream);
    else e = launch_strided<true, LOAD_CENTRED>(ring, B, n_polys, stream);
    if (e != cudaSuccess) return e;
    return launch_contig<true>(ring, B, n_polys, stream);
}

cudaError_t ntt_forward_ingest(const RingHost& ring, const PolyBatch& B0, u32 n_in, cudaStream_t stream) {
    const u32 r = ring.dev.r;
    PolyBatch B = B0;
    B.ingest = 1;
    B.n_m = r + 1;
    cudaError_t e = launch_strided<true, LOAD_INGEST>(ring, B, n_in * 2 * r * B.n_m, stream);
    if (e != cudaSuccess) return e;
    B.n_m = r + 2;
    return launch_contig<true, 5>(ring, B, n_in * r * B.n_m, stream);
}

cudaError_t ntt_forward_moddown(const RingHost& ring, const PolyBatch& B, u32 n_outer, const RotBatch& rb,
                                const ModDownEpilogue& epi, cudaStream_t stream) {
    const u32 n_polys = n_outer * B.n_m;
    cudaError_t e = launch_strided<true, LOAD_CENTRED>(ring, B, n_polys, stream);
    if (e != cudaSuccess) return e;
    return launch_contig<true, 1>(ring, B, n_polys, stream, RotationDivision{epi, rb});
}

// Forward transform whose final store is permuted: polynomial (o, m) ends up at
// final[(o*dst_so + m*dst_sm) + scatter[(o / scatter_div)*N + n]].  B.dst is a staging buffer of the same shape.
cudaError_t ntt_forward_split(const RingHost& ring, const PolyBatch& B0, u32 n_outer, int load, void* final_dst,
                              const u32* scatter, u32 scatter_div, cudaStream_t stream) {
    PolyBatch B = B0;
    const u32 n_polys = n_outer * B.n_m;
    cudaError_t e;
    if (load == LOAD_PLAIN) e = launch_strided<true, LOAD_PLAIN>(ring, B, n_polys, stream);
    else e = launch_strided<true, LOAD_REDUCE>(ring, B, n_polys, stream);
    if (e != cudaSuccess) return e;
    B.scatter = scatter;
    B.scatter_div = scatter_div;
    B.dtile_ptr = (u64*)final_dst;
    return launch_contig<true>(ring, B, n_polys, stream);
}

cudaError_t ntt_forward_first(const RingHost& ring, const PolyBatch& B, u32 n_outer, cudaStream_t stream) {
    return launch_strided<true, LOAD_REDUCE>(ring, B, n_outer * B.n_m, stream);
}

template <int RC>
static cudaError_t launch_contig_inner_t(const RingHost& ring, const PolyBatch& B, const RotBatch& rb, const void* keys, u64* u, u64* xext,
                                         const u32* pinv, u32 cb, cudaStream_t stream) {
    typedef InnerGeo<RC> G;
    const u32 chunks = ring.dev.N >> LOG_C;
    return launch_dependent(ring, ntt_contig_inner<RC>, dim3(rb.n_groups, (chunks + cb - 1) / cb, RC + 1), dim3(32 * G::WARPS),
                            (size_t)8 * (cb * RC << LOG_C), stream, ring.dev, B, rb, keys, u, xext, pinv, cb);
}

// (a context has 2 to MAX_MODULI - 1 digits: see bf_ctx_create)
template <int RC>
static cudaError_t launch_contig_inner(const RingHost& ring, const PolyBatch& B, const RotBatch& rb, const void* keys, u64* u, u64* xext,
                                       const u32* pinv, u32 cb, cudaStream_t stream) {
    if (ring.dev.r == RC) return launch_contig_inner_t<RC>(ring, B, rb, keys, u, xext, pinv, cb, stream);
    if constexpr (RC + 1 < MAX_MODULI) return launch_contig_inner<RC + 1>(ring, B, rb, keys, u, xext, pinv, cb, stream);
    else return cudaErrorInvalidValue;
}

cudaError_t ntt_forward_inner(const RingHost& ring, const PolyBatch& B_in, u32 n_sets, const RotBatch& rb_in, const void* keys, u64* u,
                              u64* xext, const u32* pinv, cudaStream_t stream) {
    const u32 r = ring.dev.r;
    if (rb_in.n == 0) return cudaSuccess;
    if (n_sets) {
        const cudaError_t e = ntt_forward_first(ring, B_in, n_sets * r, stream);
        if (e != cudaSuccess) return e;
    }
    // runs of consecutive rotations with the same digit set, cut into parts until the blocks fill the machine (every part
    // transforms the digits again, which costs less than idle SMs).  Three rounds of 148 SMs x 4 blocks; one where most moduli
    // are on the integer path, whose transforms cost several times as much (N = 2^15, 1024 -> 2048 without double hoisting:
    // 55-bit primes 422 us in three, 409 us in one; 40-bit primes, 3072 -> 768, 632 and 641 us)
    RotBatch rb = rb_in;
    // (as many chunks a block as digits leave warps for, fewer where a block per rotation and chunks would not fill the GPU once:
    // six rotations of three digits on a ring of 2^12 6.6 us with two chunks a block, 5.7 us with one)
    const u32 chunks = ring.dev.N >> LOG_C;
    u32 cb = r > 8 ? 1u : 8u / r;
    if (cb > chunks) cb = chunks;
    while (cb > 1 && (u32)rb.n * ((chunks + cb - 1) / cb) * (r + 1) < 592u) cb = (cb + 1) / 2;
    u32 runs = 0, n_int = 0;
    for (int t = 0; t < rb.n; ++t) runs += t == 0 || rb.dig[t] != rb.dig[t - 1];
    for (u32 m = 0; m <= r; ++m) n_int += ring.dev.fp_ok[m] ? 0u : 1u;
    const u32 blocks = runs * ((chunks + cb - 1) / cb) * (r + 1), fill = 2 * n_int > r + 1 ? 592u : 1776u;
    const u32 parts = blocks < fill ? fill / blocks : 1u;
    rb.n_groups = 0;
    for (int t = 0; t < rb.n;) {
        int end = t + 1;
        while (end < rb.n && rb.dig[end] == rb.dig[t]) ++end;
        const int len = end - t, per = (len + (int)parts - 1) / (int)parts;
        for (; t < end; t += per) {
            rb.grp_first[rb.n_groups] = (unsigned char)t;
            rb.grp_cnt[rb.n_groups++] = (unsigned char)(end - t < per ? end - t : per);
        }
        t = end;
    }
    if (ring.prof) {
        const u64 key_bytes = ring.dev.key_bytes;
        u32 distinct = 0;
        for (int t = 0; t < rb.n; ++t) {
            bool seen = false;
            for (int k = 0; k < t && !seen; ++k) seen = rb.key[k] == rb.key[t];
            distinct += seen ? 0u : 1u;
        }
        ring.prof->key_bytes_distinct += distinct * key_bytes;
        ring.prof->key_bytes_per_rotation += (u64)rb.n * key_bytes;
    }
    ProfScope prof(ring.prof, CAT_KEY_INNER, stream);
    return launch_contig_inner<2>(ring, B_in, rb, keys, u, xext, pinv, cb, stream);
}

cudaError_t ntt_inverse_assembly(const RingHost& ring, const PolyBatch& B, u32 n_outer, const OutputAssembly& as, cudaStream_t stream) {
    const u32 n_polys = n_outer * B.n_m;
    cudaError_t e = launch_contig<false, 4>(ring, B, n_polys, stream, as);
    if (e != cudaSuccess) return e;
    return launch_strided<false, LOAD_PLAIN>(ring, B, n_polys, stream);
}

// Last step of the output assembly: the inverse transforms above left, per output p and
// component, the sum of all terms modulo every q_i (in ct) and each separately rounded term's residue modulo P as a
// centred lift plus 2^59 (in T, n_t polynomials per output, indexed as OutputAssembly lists them):
//   ct[p][comp][i][n] = (ct[p][comp][i][n] - sum_terms t_term[n]) * P^{-1}  (mod q_i)
// low non-null: the rescale (Sec. 2.1) follows in the same thread, which holds all residues of its coefficient: the
// result goes to low[p][comp][r-1][N] as c'_i = (c_i - centred(c_{r-1})) * q_{r-1}^{-1} and ct only held the sums.
// the k-th of component comp's terms, as the polynomials of T are numbered, and how many there are
__device__ __forceinline__ u32 assembly_term(u32 k, u32 comp, u32 n_u) { return 2 * k < n_u ? comp + 2 * k : 2 * k == n_u ? n_u + comp : n_u + 1 + k - n_u / 2; }
__device__ __forceinline__ u32 assembly_terms(u32 comp, u32 n_u, u32 n_t) { return n_u / 2 + (n_t == n_u ? 0u : comp ? 1u : n_t - n_u - 1); }

// the centred values of terms k0 .. k0 + 7 (each below 2^59 in magnitude), requested together: two outputs of five terms at N = 2^15
// 8.6 us one after the other, 6.8 us like this
__device__ __forceinline__ i64 assembly_sum(const u64* __restrict__ tp, size_t N, u32 k0, u32 nt, u32 comp, u32 n_u) {
    u64 t[8];
#pragma unroll
    for (u32 h = 0; h < 8; ++h) t[h] = k0 + h < nt ? __ldg(tp + assembly_term(k0 + h, comp, n_u) * N) : 1ull << 59;
    i64 S = 0;
#pragma unroll
    for (u32 h = 0; h < 8; ++h) S += (i64)(t[h] - (1ull << 59));
    return S;
}

__global__ void __launch_bounds__(128, 8) finish_division_kernel(const RingDev R, u64* __restrict__ ct, long long ct_stride,
                                                              const u64* __restrict__ T, u32 n_u, u32 n_t, const RescaleConsts rc,
                                                              u64* __restrict__ low) {
    grid_dependency_enter();
    const u32 n = blockIdx.x * 128 + threadIdx.x;
    const u32 p = blockIdx.y >> 1, comp = blockIdx.y & 1;
    const u64* tp = T + (size_t)p * n_t * R.N + n;
    u64* cp = ct + (size_t)p * ct_stride + (size_t)comp * R.r * R.N + n;
    u64 v[MAX_MODULI];
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i)
        if ((u32)i < R.r) v[i] = cp[(size_t)i * R.N];
    // the centred values of this component's terms are added as integers, eight at a time (each is below 2^59 in magnitude),
    // and the sum is reduced once per prime
    const u32 nt = assembly_terms(comp, n_u, n_t);
    for (u32 k0 = 0; k0 < nt; k0 += 8) {
        const i64 S = assembly_sum(tp, R.N, k0, nt, comp, n_u);
        const bool neg = S < 0;
        const u64 a = neg ? (u64)(-S) : (u64)S;
#pragma unroll
        for (int i = 0; i < MAX_MODULI; ++i)
            if ((u32)i < R.r) {
                u64 t = barrett64(a, R.q[i], R.mu[i]);
                if (neg && t) t = R.q[i] - t;
                v[i] = sub_mod(v[i], t, R.q[i]);
            }
    }
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i)
        if ((u32)i < R.r) v[i] = mul_shoup(v[i], R.pinv[i], R.pinvs[i], R.q[i]);
    if (!low) {
#pragma unroll
        for (int i = 0; i < MAX_MODULI; ++i)
            if ((u32)i < R.r) cp[(size_t)i * R.N] = v[i];
        return;
    }
    u64 t = 0;                      // the residue that is dropped
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i) {
        u64 vi = v[i];
        asm volatile("" : "+l"(vi));    // (keeps the selection a chain of moves: as an indexed read it would put v in local memory)
        if ((u32)i == R.r - 1) t = vi;
    }
    const bool high = t > (R.q[R.r - 1] - 1) / 2;
    u64* lp = low + ((size_t)p * 2 + comp) * (R.r - 1) * R.N + n;
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i)
        if ((u32)i + 1 < R.r) {
            const u64 q = R.q[i];
            u64 tq = barrett64(t, q, R.mu[i]);
            if (high) tq = sub_mod(tq, rc.qlmod[i], q);
            lp[(size_t)i * R.N] = mul_shoup(sub_mod(v[i], tq, q), rc.inv[i], rc.invs[i], q);
        }
}

// The same in fp64 (every value an exact integer below 2^53), for rings whose ciphertext primes are all on the fp64
// path: a 64-bit modular product costs about twenty integer instructions, an exact fp64 one six on a pipe that is
// otherwise idle here.  Each term sum S = s_hi 2^30 + s_lo is reduced as s_hi (2^30 mod q) + s_lo; products come back
// centred and are brought to [0, q) only where a canonical residue is needed (the stored words, the dropped residue).
__device__ __forceinline__ double fp_times_const(double x, bool wide, double w, double wq, double q, double qinv) {
    // x an integer of magnitude below 2^50 (any sign): x * w mod q in [0, q)
    double s2;
    if (wide) s2 = fp_mul_centred(__dadd_rn(fp_centre(x, q, qinv), q), w, wq, q);     // operand in (0.5q, 1.5q)
    else s2 = fp_mul_centred_signed(x, w, wq, q);
    return s2 < 0.0 ? __dadd_rn(s2, q) : s2;
}

__global__ void __launch_bounds__(128, 8) finish_division_fp_kernel(const RingDev R, u64* __restrict__ ct, long long ct_stride,
                                                                 const u64* __restrict__ T, u32 n_u, u32 n_t, const RescaleConsts rc,
                                                                 u64* __restrict__ low) {
    grid_dependency_enter();
    const u32 n = blockIdx.x * 128 + threadIdx.x;
    const u32 p = blockIdx.y >> 1, comp = blockIdx.y & 1;
    const u64* tp = T + (size_t)p * n_t * R.N + n;
    u64* cp = ct + (size_t)p * ct_stride + (size_t)comp * R.r * R.N + n;
    double v[MAX_MODULI];
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i)
        if ((u32)i < R.r) v[i] = u2d(cp[(size_t)i * R.N]);
    const u32 nt = assembly_terms(comp, n_u, n_t);
    for (u32 k0 = 0; k0 < nt; k0 += 8) {
        const i64 S = assembly_sum(tp, R.N, k0, nt, comp, n_u);
        const i64 s_hi = S >> 30;                               // |s_hi| < 2^33
        const double lo = u2d((u64)(S & ((1ll << 30) - 1)));
        const bool sneg = s_hi < 0;
        const double ah = u2d((u64)(sneg ? -s_hi : s_hi));
#pragma unroll
        for (int i = 0; i < MAX_MODULI; ++i)
            if ((u32)i < R.r) {
                const double sm = fp_mul_centred(ah, R.c30_d[i], R.c30_q[i], R.qd[i]);      // within 0.75 q
                const double x = __dsub_rn(__dsub_rn(v[i], sneg ? -sm : sm), lo);
                v[i] = fp_centre(x, R.qd[i], R.qinv_d[i]);
            }
    }
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i)
        if ((u32)i < R.r) v[i] = fp_times_const(v[i], (R.q[i] >> 41) != 0, R.pinv_d[i], R.pinv_q[i], R.qd[i], R.qinv_d[i]);
    if (!low) {
#pragma unroll
        for (int i = 0; i < MAX_MODULI; ++i)
            if ((u32)i < R.r) cp[(size_t)i * R.N] = d2u(v[i]);
        return;
    }
    double t = 0.0;                 // the residue that is dropped (below 2^46: the launcher checked)
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i) {
        double vi = v[i];
        asm volatile("" : "+d"(vi));    // (keeps the selection a chain of moves: as an indexed read it would put v in local memory)
        if ((u32)i == R.r - 1) t = vi;
    }
    const bool high = d2u(t) > (R.q[R.r - 1] - 1) / 2;
    u64* lp = low + ((size_t)p * 2 + comp) * (R.r - 1) * R.N + n;
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i)
        if ((u32)i + 1 < R.r) {
            double tq = fp_reduce(t, R.qd[i], R.qinv_d[i]);
            if (high) tq = __dsub_rn(tq, rc.qlmod_d[i]);
            const double y = fp_times_const(__dsub_rn(v[i], tq), (R.q[i] >> 41) != 0, rc.inv_d[i], rc.inv_q[i], R.qd[i],
                                            R.qinv_d[i]);
            lp[(size_t)i * R.N] = d2u(y);
        }
}

cudaError_t finish_division(const RingHost& ring, u64* ct, long long ct_stride, const u64* T, u32 n_u, u32 n_t, u32 n_out,
                            cudaStream_t stream, const RescaleConsts* rc, u64* low) {
    RescaleConsts none;
    memset(&none, 0, sizeof(none));
    bool fp = true;
    for (u32 i = 0; i < ring.dev.r; ++i) fp = fp && ring.dev.fp_ok[i];
    if (rc && ring.q[ring.dev.r - 1] >= (1ull << 46)) fp = false;
    // (a launch for every 32767 outputs, whose polynomials the second dimension of a grid holds; a place worked out of one dimension
    // costs a short chain of launches 0.4 us: 300 -> 1000 on a ring of 2^12 46.7 -> 47.0 us)
    constexpr u32 MOST = 65535u / 2;
    const size_t N = ring.dev.N;
    for (u32 p0 = 0; p0 < n_out; p0 += MOST) {
        ProfScope prof(ring.prof, CAT_DIVIDE, stream);
        const u32 n = n_out - p0 < MOST ? n_out - p0 : MOST;
        launch_dependent(ring, fp ? finish_division_fp_kernel : finish_division_kernel, dim3(ring.dev.N / 128, n * 2), dim3(128), 0, stream, ring.dev,
                         ct + (size_t)p0 * ct_stride, ct_stride, T + (size_t)p0 * n_t * N, n_u, n_t, rc ? *rc : none,
                         rc ? low + (size_t)p0 * 2 * (ring.dev.r - 1) * N : (u64*)nullptr);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The last step of a rotation whose key-switch result u is at hand in the coefficient domain, rotated, over {q_i, P} (its residue
// modulo P as a centred lift plus 2^59): out = (u0, u1) / P + (phi(c0), 0), plus (c0, c1) where `add`.  phi moves coefficient k to
// k * gal mod 2N, with a sign beyond N.  A thread has all residues of its coefficient, so that the lift is cut once.
template <bool FP>
__global__ void __launch_bounds__(128, 8) finish_rotation_kernel(const RingDev R, const u64* __restrict__ u, const u64* __restrict__ ct,
                                                                 u64* __restrict__ out, u32 gal_inv, u32 add) {
    grid_dependency_enter();
    const u32 n = blockIdx.x * 128 + threadIdx.x, comp = blockIdx.y & 1;
    const size_t N = R.N, poly = (size_t)blockIdx.y * R.r * N;
    const u64* up = u + (size_t)blockIdx.y * (R.r + 1) * N + n;
    const u64* cp = ct + poly;
    const u32 k = (n * gal_inv) & (2 * R.N - 1), from = k & (R.N - 1);
    const bool minus = k >= R.N;
    const i64 S = (i64)(up[R.r * N] - (1ull << 59));
    const i64 s_hi = S >> 30;
    const bool neg = S < 0;
    const u64 mag = neg ? (u64)(-S) : (u64)S;
    const double lo = u2d((u64)(S & ((1ll << 30) - 1))), ah = u2d((u64)(s_hi < 0 ? -s_hi : s_hi));
#pragma unroll
    for (int i = 0; i < MAX_MODULI; ++i)
        if ((u32)i < R.r) {
            const u64 q = R.q[i];
            u64 v;
            if (FP) {
                const double sm = fp_mul_centred(ah, R.c30_d[i], R.c30_q[i], R.qd[i]);
                const double x = __dsub_rn(__dsub_rn(u2d(up[i * N]), neg ? -sm : sm), lo);
                v = d2u(fp_times_const(fp_centre(x, R.qd[i], R.qinv_d[i]), (q >> 41) != 0, R.pinv_d[i], R.pinv_q[i], R.qd[i], R.qinv_d[i]));
            } else {
                u64 t = barrett64(mag, q, R.mu[i]);
                if (neg && t) t = q - t;
                v = mul_shoup(sub_mod(up[i * N], t, q), R.pinv[i], R.pinvs[i], q);
            }
            if (comp == 0) {
                const u64 c = cp[i * N + from];
                v = minus ? sub_mod(v, c, q) : add_mod(v, c, q);
            }
            if (add) v = add_mod(v, cp[i * N + n], q);
            out[poly + i * N + n] = v;
        }
}

cudaError_t finish_rotation(const RingHost& ring, const u64* u, const u64* ct, u64* out, u32 n_ct, u32 gal_inv, bool add, cudaStream_t stream) {
    ProfScope prof(ring.prof, CAT_DIVIDE, stream);
    bool fp = true;
    for (u32 i = 0; i < ring.dev.r; ++i) fp = fp && ring.dev.fp_ok[i];
    launch_dependent(ring, fp ? finish_rotation_kernel<true> : finish_rotation_kernel<false>, dim3(ring.dev.N / 128, n_ct * 2), dim3(128), 0,
                     stream, ring.dev, u, ct, out, gal_inv, add ? 1u : 0u);
    return cudaGetLastError();
}

cudaError_t ntt_inverse(const RingHost& ring, const PolyBatch& B, u32 n_outer, cudaStream_t stream) {
    const u32 n_polys = n_outer * B.n_m;
    cudaError_t e = launch_contig<false>(ring, B, n_polys, stream);
    if (e != cudaSuccess) return e;
    return launch_strided<false, LOAD_PLAIN>(ring, B, n_polys, stream);
}

}  // namespace bf
