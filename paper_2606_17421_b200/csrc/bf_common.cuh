// Shared device-side types and modular arithmetic for the CKKS linear-layer kernels (sm_100a).
//
// Residues are 64-bit words modulo primes q < 2^60, so lazily reduced values up to 16q fit a word
// and a sum of up to 2^8 products of two residues fits 128 bits.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace bf {

typedef uint64_t u64;
typedef int64_t i64;
typedef uint32_t u32;

constexpr int MAX_MODULI = 16;    // ciphertext primes + the special prime
constexpr int ENC_CONSTS = 5;
// Per-ring constants handed to every kernel by value (lands in the constant bank).
// Modulus index r is the special prime P; 0..r-1 are the ciphertext primes q_0..q_L.
struct RingDev {
    u32 N, logN, r;
    u64 q[MAX_MODULI];
    u64 mu[MAX_MODULI];          // floor(2^64 / q)
    u64 c64[MAX_MODULI];         // 2^64 mod q
    u64 c64s[MAX_MODULI];        // Shoup companion of c64
    u64 ninv[MAX_MODULI];        // N^{-1} mod q
    u64 ninvs[MAX_MODULI];
    u64 pinv[MAX_MODULI];        // P^{-1} mod q_i (i < r)
    u64 pinvs[MAX_MODULI];
    u64 pmod[MAX_MODULI];        // P mod q_i
    u64 qneg[MAX_MODULI];        // -q^{-1} mod 2^64 (Montgomery reduction)
    u64 ninv_m[MAX_MODULI];      // N^{-1} * 2^{-64} mod q: inverse transform that also leaves Montgomery form
    u64 ninv_ms[MAX_MODULI];
    u32 fp_ok[MAX_MODULI];       // modulus below 2^50: its transforms run in fp64 (every value an exact integer below
                                 //   2^53) and its twiddle tables hold the bits of ((double)w, (double)w / q)
    double qd[MAX_MODULI];       // (double)q
    double qinv_d[MAX_MODULI];   // 1.0 / q
    double ninv_d[MAX_MODULI], ninv_q[MAX_MODULI];     // (double)N^{-1} and N^{-1} / q
    double ninvm_d[MAX_MODULI], ninvm_q[MAX_MODULI];   // the same for N^{-1} * 2^{-64} (leaving Montgomery form)
    double c30_d[MAX_MODULI], c30_q[MAX_MODULI];       // (double)(2^30 mod q) and that over q
    double k59_d[MAX_MODULI];    // 2q - (2^59 mod q): undoes the offset of a stored centred lift, keeps it positive
    double pinv_d[MAX_MODULI], pinv_q[MAX_MODULI];     // (double)(P^{-1} mod q_i) and that over q_i (i < r)
    u32 dp[MAX_MODULI];          // modulus below 2^40: operands of the inner products (cached plaintexts, rotation keys, digits)
                                 //   are kept as the bits of doubles and multiplied in fp64 (see DpAcc)
    double c40_d[MAX_MODULI], c40_q[MAX_MODULI];       // (double)(2^40 mod q) and that over q
    u64 key_base[MAX_MODULI];    // resident rotation keys (see KeyTile): byte offset of modulus m inside a key
    u64 key_bytes;               //   bytes of a key
    // encoder output (signed 64-bit coefficients) into Montgomery form on the fp64 path: the word is
    // (hi' - 2^31) 2^32 + lo, so times 2^64 it is  hi' (2^96 mod q) + lo (2^64 mod q) - (2^127 mod q).
    // Five doubles per prime, in device memory (kernel parameters stay small): (double)(2^96 mod q), that
    // over q, (double)(2^64 mod q), that over q, and the centred residue of -2^127 (plus 2q for primes of
    // 2^41 or more, whose values stay non-negative).  Primes with dp set keep plaintexts without the factor 2^64:
    // 2^32, 1 and -2^63 instead
    const double* enc_consts;    // [r+1][ENC_CONSTS]
    const ulonglong2* tw_fwd;    // [r+1][N]  (psi^brev(k), companion), merged Cooley-Tukey order
    const ulonglong2* tw_inv;    // [r+1][N]  inverses of the above, for the Gentleman-Sande inverse
    const double *tw8_fwd, *tw8_inv;   // [r+1][N]  (double)w alone, moduli below 2^41
};

// floor(x * w / 2^64)-based modular multiplication by a constant w with precomputed
// ws = floor(w * 2^64 / q).  Valid for any 64-bit x; result in [0, 2q).
__device__ __forceinline__ u64 mul_shoup_lazy(u64 x, u64 w, u64 ws, u64 q) {
    u64 hi = __umul64hi(x, ws);
    return x * w - hi * q;
}

// First statement of every kernel of a linear-layer call.  Lets the next kernel of the stream be scheduled
// as soon as all blocks of this one have started, then waits until the previous kernel has completed and
// flushed its writes.  A no-op when the launch carries no programmatic dependency.
__device__ __forceinline__ void grid_dependency_enter() {
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---- fp64 arithmetic for primes q < 2^50.  B200 issues fp64 FMAs at the rate of 32-bit integer
// multiply-adds, on a pipe of its own, while a 64x64-bit high product costs about ten integer
// multiply-add slots; and integers below 2^53 are exact in fp64.
__device__ __forceinline__ double u2d(u64 x) {          // exact for x < 2^52
    return __longlong_as_double((long long)(x | 0x4330000000000000ull)) - 4503599627370496.0;
}
__device__ __forceinline__ u64 d2u(double d) {          // d an integer in [0, 2^52)
    return (u64)__double_as_longlong(d + 4503599627370496.0) - 0x4330000000000000ull;
}
__device__ __forceinline__ double i2d(i64 v) {          // exact for |v| < 2^51
    return __longlong_as_double((long long)(v + 0x4338000000000000ll)) - 6755399441055744.0;
}
__device__ __forceinline__ i64 d2i(double d) {          // d an integer, |d| < 2^51
    return (i64)__double_as_longlong(d + 6755399441055744.0) - 0x4338000000000000ll;
}
// x * w - round(x * w / q) * q for a non-negative integer-valued x and a constant 0 <= w < q given as
// (double)w and wq = (double)w / q.  ph + pl = x*w exactly (FMA); the quotient estimate is within
// 1/2 + x * 2^-52 of x*w/q; ph - qh*q is an integer far below 2^53 and therefore exact, and so is the final
// sum.  For q < 2^41 and x < 2^46 the result lies in (-0.51q, 0.51q); for q < 2^50 and x <= 4q < 2^52 in
// (-0.75q, 0.75q).  Always congruent to x*w.
__device__ __forceinline__ double fp_mul_centred(double x, double w, double wq, double q) {
    const double magic = 4503599627370496.0;             // 2^52
    const double ph = __dmul_rn(x, w);
    const double pl = __fma_rn(x, w, -ph);
    const double qh = __dsub_rn(__fma_rn(x, wq, magic), magic);
    return __dadd_rn(__fma_rn(-qh, q, ph), pl);
}
// The same product for a signed integer-valued |x| < 2^47 and q < 2^41 (rounding constant 1.5 * 2^52, which
// is exact for quotients of either sign): congruent to x*w, |result| <= 0.532 q.
__device__ __forceinline__ double fp_mul_centred_signed(double x, double w, double wq, double q) {
    const double magic = 6755399441055744.0;             // 1.5 * 2^52
    const double ph = __dmul_rn(x, w);
    const double pl = __fma_rn(x, w, -ph);
    const double qh = __dsub_rn(__fma_rn(x, wq, magic), magic);
    return __dadd_rn(__fma_rn(-qh, q, ph), pl);
}
// v - round(v / q) q for a signed integer-valued |v| < 2^50: congruent to v, |result| <= q / 2
__device__ __forceinline__ double fp_centre(double v, double q, double qinv) {
    const double magic = 6755399441055744.0;
    const double qh = __dsub_rn(__fma_rn(v, qinv, magic), magic);
    return __fma_rn(-qh, q, v);
}
// v mod q in [0, q) for a signed integer-valued |v| < 2^50, q < 2^41: (v + 1/2) / q is at least 1 / (2q) away from any integer,
// which the error of 1/q (2^-53 of at most 2^50 / q) does not bridge, so its floor is exact
__device__ __forceinline__ double fp_canonical(double v, double q, double qinv) {
    const double magic = 6755399441055744.0;
    const double qh = __dsub_rn(__fma_rd(__dadd_rn(v, 0.5), qinv, magic), magic);
    return __fma_rn(-qh, q, v);
}
// v mod q in [0, q) for an integer-valued 0 <= v < 2^46
__device__ __forceinline__ double fp_reduce(double v, double q, double qinv) {
    const double magic = 4503599627370496.0;
    const double qh = __dsub_rn(__fma_rn(v, qinv, magic), magic);
    double r = __fma_rn(-qh, q, v);
    if (r < 0.0) r = __dadd_rn(r, q);
    return r;
}

__device__ __forceinline__ u64 mul_shoup(u64 x, u64 w, u64 ws, u64 q) {
    u64 v = mul_shoup_lazy(x, w, ws, q);
    return v >= q ? v - q : v;
}

// x mod q for any 64-bit x, mu = floor(2^64 / q).  The quotient estimate is short by at most one.
__device__ __forceinline__ u64 barrett64(u64 x, u64 q, u64 mu) {
    u64 v = x - __umul64hi(x, mu) * q;
    return v >= q ? v - q : v;
}

// (hi * 2^64 + lo) mod q:  hi * (2^64 mod q) by a Shoup product, lo by Barrett, then fold.
__device__ __forceinline__ u64 reduce128(u64 hi, u64 lo, u64 q, u64 mu, u64 c64, u64 c64s) {
    u64 a = mul_shoup_lazy(hi, c64, c64s, q);        // [0, 2q)
    u64 b = lo - __umul64hi(lo, mu) * q;             // [0, 2q)
    u64 v = a + b;                                   // [0, 4q)
    if (v >= 2 * q) v -= 2 * q;
    if (v >= q) v -= q;
    return v;
}

// acc (128-bit, as hi:lo) += a * b
__device__ __forceinline__ void mac128(u64& hi, u64& lo, u64 a, u64 b) {
    u64 pl = a * b;
    u64 ph = __umul64hi(a, b);
    lo += pl;
    hi += ph + (lo < pl ? 1ull : 0ull);
}

__device__ __forceinline__ u64 add_mod(u64 a, u64 b, u64 q) {
    u64 v = a + b;
    return v >= q ? v - q : v;
}

__device__ __forceinline__ u64 sub_mod(u64 a, u64 b, u64 q) {
    return a >= b ? a - b : a + q - b;
}

// How the first pass of a transform reads its input.
enum LoadMode : int {
    LOAD_PLAIN = 0,     // residues already modulo the target prime, in [0, q)
    LOAD_REDUCE = 1,    // any 64-bit non-negative integer (e.g. a residue of another prime): x mod q
    LOAD_I64 = 2,       // signed 64-bit integer coefficient: x mod q in [0, q)
    LOAD_CENTRED = 3,   // centred lift t' in (-M/2, M/2] of a residue of modulus M, stored as t' + 2^59: t' mod q
    LOAD_I64_MONT = 4,  // LOAD_I64, then times 2^64 mod q: the transform's output is in Montgomery form
    LOAD_INGEST = 5,    // LOAD_REDUCE for an ingest batch (see PolyBatch::ingest)
};

constexpr int MAX_ROT_BATCH = 64; // rotations handled by one key-switch launch

struct RotBatch {                     // one key-switch launch over n rotations
    int n;
    int key[MAX_ROT_BATCH];           // index of the rotation key (and of its permutation table)
    int dig[MAX_ROT_BATCH];           // which digit set the rotation reads
    int c0[MAX_ROT_BATCH];            // which source ciphertext is being rotated (its c0 is added)
    int out[MAX_ROT_BATCH];           // which output ciphertext slot receives the result
    // runs of consecutive rotations that read the same digit set (filled in by the launcher): one block takes one run
    int n_groups;
    unsigned char grp_first[MAX_ROT_BATCH], grp_cnt[MAX_ROT_BATCH];
};

// Epilogue of the division by P of a rotated input, fused into the forward transform of the lifted P-residue
// (polynomial (o, m) = (rotation*2 + component, prime i)):  instead of storing t = NTT(lift),
//   v = (u[o][i][n] - t) * P^{-1} + (component == 0 ? c0[c0(rot)][i][n] : 0)
// is scattered to out[out(rot)][component][i][pinv[key(rot)][n]].
struct ModDownEpilogue {
    const u64* u;                 // [rot][2][r+1][N]
    const u64* c0_base;
    long long c0_stride;
    const u32* pinv;              // [n_keys][N]
    u64* out_base;
    long long out_stride;
};

// Output assembly (load of an inverse transform).  Output p is a sum of the inner sum of giant step 0, the rotated c0 parts of
// the other inner sums and the key-switch results of their c1 parts, which live over {q_i, P} and are divided by P, each by
// itself or once for their sum.  The result is wanted in the coefficient domain, where that division is element-wise
// (finish_division): so the terms are summed modulo every q_i here and what is rounded by itself is transformed modulo P by
// itself; no lifted P-residue is transformed forward.  Inner sum (j, p) is a + (j*n_out + p)*a_stride, [2][r or r+1][N];
// u[((j-1)*n_out + p)*2 + comp][r+1][N] are the key-switch results of giant steps j >= 1.  What is rotated (u, and component
// 0 of the inner sums with j >= 1) was stored through rotation j's permutation by its producer.  Polynomial (o = p, m):
//   modulus i < r, m = comp*r + i:  F a[p][comp][i] + sum_j u[j][p][comp][i] + (comp == 0) F sum_j a[j][p][0][i]
//       (F = 1 where the inner sums live in the extended basis, else P)
//   modulus P, the separately rounded terms, m - 2r =
//       0, 1:                        sum_j u[j][p][comp][P]             (one division per output)
//       2 (j - 1) + comp:            u[j][p][comp][P]                   (each: one division per rotation)
//     and, n_u such terms further on, where the inner sums live in the extended basis,
//       comp:                        a[p][comp][P]
//       1 + j:                       a[j][p][0][P]
struct OutputAssembly {
    const u64 *u, *a;
    long long a_stride;
    u32 g1, n_out;                // giant steps j >= 1, outputs
    u32 ext;                      // the inner sums live in the extended basis (double hoisting)
    u32 each;                     // every key-switch result is divided by itself
    __host__ __device__ __forceinline__ u32 n_u() const { return g1 == 0 ? 0u : each ? 2u * g1 : 2u; }
    __host__ __device__ __forceinline__ u32 n_t() const { return n_u() + (ext ? g1 + 2u : 0u); }
};

// Component 0 of inner sum (j, p), j >= 1, is only ever used rotated by giant step j, so the multiply-accumulate stores it
// through that rotation (group pj0 + pj has j = (pj0 + pj) / n_out; on = 0: plain stores).
struct MacScatter {
    u32 on, n_out, pj0;
    u32 gal_inv;                        // inverse Galois element of giant step 1: step j has its j-th power
};

// Baby rotations computed inside the multiply-accumulate (double hoisting): input q's term k is its rotation by the key at key_at[k].
struct BabySteps {
    u32 n_in, b;
    u32 parts, per_part;                // how the inputs are dealt out to a block's lanes (set by the launcher)
    const void* keys;                   // resident keys
    const u64* dig;                     // digit set q of input q (tile-major, see KS_TILE)
    u64 key_at[MAX_ROT_BATCH + 1];      // byte offset of the key
    u32 gal[MAX_ROT_BATCH + 1], gal_inv[MAX_ROT_BATCH + 1];
};

// Constants of a rescale from `level` primes: q_L^{-1} mod q_i with its Shoup companion, and q_L mod q_i (i < level - 1).
struct RescaleConsts {
    u64 inv[MAX_MODULI], invs[MAX_MODULI], qlmod[MAX_MODULI];
    double inv_d[MAX_MODULI], inv_q[MAX_MODULI], qlmod_d[MAX_MODULI];   // the same as doubles; inv_q = inv / q_i
};

// Tile-major layout of cached plaintexts, chosen so that the multiply-accumulate kernel's blocks
// each stream one contiguous region:  word (group pj, term t, prime i, coefficient n) has index
//   ((pj%PL)*TS + t%TS)*TN + n%TN   inside stage   ((i, n/TN), pj/PL, t/TS)
// with TN = 2^log_tn coefficients per tile, PL = 256/TN group lanes, TS = 8 terms per stage,
// G = ceil(n_pj/PL), C = ceil(n_terms/TS); a stage holds the words of min(PL, n_pj) lanes, 2048 of them where the groups fill
// the lanes.  The stages of one prime are
// contiguous, ordered (tile, pj/PL, t/TS), and every prime stores its words in the narrowest of three
// formats its size allows, because the kernel that reads them is bound by HBM bytes:
//   TILE_W64  8 bytes per word, two limbs (16 KB per full stage)
//   TILE_W40  primes below 2^40: a lane's TS rows of low 32 bits, then two rows of high bytes, those of four terms in one
//             32-bit word: byte t%4 of word n%TN of row t%8 / 4 (10 KB per full stage)
//   TILE_W32  primes below 2^32: 32-bit words (8 KB per full stage)
// (Words of 8 bytes throughout: the four calls of a 0.6B layer stream 2.78 instead of 2.40 GB.)
enum TileFormat : u32 { TILE_W64 = 0, TILE_W40 = 1, TILE_W32 = 2 };
struct TileLayout {
    u32 log_tn, n_terms, n_pj, G, C, ntiles;
    u32 stage_words;
    u32 fmt_bits;                           // TileFormat of prime i in bits 2i, 2i+1
    u32 n_primes;                           // primes the plaintexts are held in: r, or r + 1 with double hoisting
                                            //   (the special prime last, in the format its own size asks for)
    size_t base[MAX_MODULI + 1];            // see tile_prime_base
};
constexpr u32 TILE_TS = 8;

__host__ __device__ __forceinline__ u32 tile_format(const TileLayout& t, u32 i) { return (t.fmt_bits >> (2 * i)) & 3u; }
__host__ __device__ __forceinline__ u32 tile_stage_bytes(const TileLayout& t, u32 fmt) {
    return t.stage_words * (fmt == TILE_W64 ? 8u : fmt == TILE_W40 ? 5u : 4u);
}
// byte offset of prime i's first stage (i = n_primes: total size): the primes' regions follow one another
__host__ __device__ __forceinline__ size_t tile_prime_base(const TileLayout& t, u32 i) { return t.base[i]; }
// byte offset of a stage
__host__ __device__ __forceinline__ size_t tile_stage_offset(const TileLayout& t, u32 i, u32 tile, u32 g, u32 ch) {
    return tile_prime_base(t, i) + (((size_t)tile * t.G + g) * t.C + ch) * tile_stage_bytes(t, tile_format(t, i));
}
// byte offset of a word (TILE_W40: of its low half) inside its stage
__host__ __device__ __forceinline__ u32 tile_word_offset(const TileLayout& t, u32 fmt, u32 pj, u32 term, u32 n) {
    const u32 TN = 1u << t.log_tn, PL = 256u >> t.log_tn;
    return ((pj % PL * (fmt == TILE_W40 ? TILE_TS + 2 : TILE_TS) + term % TILE_TS) * TN + (n & (TN - 1))) * (fmt == TILE_W64 ? 8 : 4);
}
// byte offset, inside its stage, of a word's high byte (TILE_W40)
__host__ __device__ __forceinline__ u32 tile_high_offset(const TileLayout& t, u32 pj, u32 term, u32 n) {
    const u32 TN = 1u << t.log_tn, PL = 256u >> t.log_tn;
    return ((pj % PL * (TILE_TS + 2) + TILE_TS + term % TILE_TS / 4) * TN + (n & (TN - 1))) * 4 + term % 4;
}
__host__ __device__ __forceinline__ size_t tile_stage_of_word(const TileLayout& t, u32 pj, u32 term, u32 i, u32 n) {
    const u32 PL = 256u >> t.log_tn;
    return tile_stage_offset(t, i, n >> t.log_tn, pj / PL, term / TILE_TS);
}

// A batch of equally sized polynomials addressed as (outer index o, slot m):
//   source  = src + o*src_so + m*src_sm      destination = dst + o*dst_so + m*dst_sm
//   modulus index of polynomial (o, m) = mod0 + m*mod_step
struct PolyBatch {
    const void* src;
    u64* dst;
    long long src_so, src_sm, dst_so, dst_sm;
    u32 n_m, mod0, mod_step;
    u32 mod_wrap;                 // > 0: modulus index = mod0 + (m % mod_wrap) * mod_step (e.g. m = component*r + prime)
    u32 o_div;                    // > 0: source = src + (o / o_div)*src_so2 + (o % o_div)*src_so + m*src_sm
    long long src_so2;
    u64 lift_mod;                 // LOAD_CENTRED: the modulus M the source residues live in
    u32 src32;                    // LOAD_I64_MONT: the source words are 32-bit integers
    u32 src_digits;               // LOAD_REDUCE: the source of outer index o is a residue modulo prime o % r
    u32 store_centred;            // inverse transform: store the centred lift of each coefficient plus 2^59
                                  //   (the form LOAD_CENTRED reads) instead of the residue in [0, q); 2: only for the
                                  //   polynomials modulo the special prime
    u32 from_mont;                // inverse transform only: input is in Montgomery form, output is not
    u64* tile_ptr;                // non-null: the NTT-domain side lives there in the tile-major layout `tile`
    TileLayout tile;              //   (forward writes its final result there, inverse reads its input there);
    u32 tile_pj0, o_base;         //   diagonal o_base + o = pj*n_terms + t; the layout's group 0 is group tile_pj0
    u32 skip_diag;                // forward only: polynomial (o, m) with m < r and o % r == m (a digit in its own prime)
    const u64* diag_src;          //   is not transformed but read from diag_src + (o / r)*diag_so + m*N, where its
    long long diag_so;            //   transform already exists
    const u32* scatter;           // forward only (rotation keys): coefficient n of the result goes to position
    u32 scatter_div;              //   scatter[(o / scatter_div) * N + n] of dtile_ptr
    u32 split_bits;               // tile-major side: 8-byte words are stored as two limbs,
                                  //   (v >> L) << 32 | (v & (2^L - 1)), L = split_bits below 2^50, else 30
    u64* lift_ptr;                // forward only, non-null (double hoisting): the transform of component comp of input o modulo
    long long lift_so;            //   q_i is also stored times P mod q_i at lift_ptr + o*lift_so + (comp*(r+1) + i)*N: the
                                  //   un-rotated input lifted to the extended basis (its residue modulo P is zero; it is only
                                  //   written where lift_zero is set)
    u32 lift_zero;
    // inverse only, tail_m > 0: slots m >= tail_m are polynomials modulo the special prime with a destination of their own,
    u32 tail_m;                   //   tail_dst + o*tail_so + (m - tail_m)*dst_sm
    u64* tail_dst;
    long long tail_so;
    // forward only, ingest = 1 (the inputs of a double-hoisted call and their digits in one go): source o = (input, component,
    // prime j).  Component 1 is transformed into every prime (digit j; n_m = r + 1 slots), component 0 into its own only, and
    // passes through tail_dst + (input * r + j) * N between the passes.  The second pass takes outer index (input, j) and
    // slots m <= r of component 1, m = r + 1 component 0; see EPI 5 of the contiguous pass
    u32 ingest;
    u64* dtile_ptr;               // ingest: the digits' transforms go there, tile-major (see
    u32 dtile_div;                //   KS_TILE, div = r); with `scatter` the resident keys
    u32 o_div_magic, dtile_magic; // ceil(2^32 / o_div), ceil(2^32 / dtile_div): o / d = umulhi(o, magic) for o < 2^16
                                  //   (set by the launchers; 0 = divide)
    const u64* div_t;             // forward from a shared source, non-null (double hoisting): the source of digit
    long long div_so;             //   i = o % o_div of set s = o / o_div is the residue modulo q_i of a polynomial in the
                                  //   extended basis, coefficient domain, and t = div_t + s*div_so holds its residue
                                  //   modulo P as a centred lift plus 2^59: the digit is (source - t) * P^{-1} mod q_i
    u32 beside;                   // forward from a shared source: digits of giant steps that run as several chains, whose launches
                                  //   overlap (for the launcher.  The lifts of baby rotations in two chains, in fewer
                                  //   blocks, do better without it: 1024 -> 512 without flags 293 us, 298 with it)
};

// The digit sets that the multiply-accumulate reads are kept tile-major, so that what a block needs of one (set, modulus,
// tile) is contiguous.  Polynomial (o, m), o = set * div + digit, div = r; coefficient n:
//   (((set * n_m + m) * (N / KS_TILE) + n / KS_TILE) * div + digit) * KS_TILE + n % KS_TILE
// (keys: see KeyTile)
constexpr u32 KS_TILE = 128;

// o / d and o % d with a host-made reciprocal (see PolyBatch::o_div_magic); magic = 0 divides
__device__ __forceinline__ void split_index(u32 o, u32 d, u32 magic, u32& hi, u32& lo) {
    hi = magic ? __umulhi(o, magic) : o / d;
    lo = o - hi * d;
}
// that index for coefficient 0 of polynomial (o = o_hi * div + o_lo, m); coefficient n then sits at
// base + (n / KS_TILE) * div * KS_TILE + n % KS_TILE
__device__ __forceinline__ size_t ks_tile_base(u32 N, u32 n_m, u32 div, u32 o_hi, u32 o_lo, u32 m) {
    return (((size_t)o_hi * n_m + m) * (N / KS_TILE) * div + o_lo) * KS_TILE;
}

__device__ __forceinline__ u64 limb_split(u64 v, u32 L) { return ((v >> L) << 32) | (v & ((1ull << L) - 1)); }
__device__ __forceinline__ u64 limb_join(u64 s, u32 L) { return ((s >> 32) << L) | (s & 0xffffffffull); }

// Montgomery reduction by two 32-bit rounds: V * 2^{-64} mod q in [0, q), for V = (H, L) < q * 2^64.
// qneg32 = -q^{-1} mod 2^32.  Six 32-bit multiplies instead of a 64x64 high product.
__device__ __forceinline__ u64 redc_2x32(u64 H, u64 L, u64 q, u32 qneg32) {
    u32 l0 = (u32)L, l1 = (u32)(L >> 32), h0 = (u32)H, h1 = (u32)(H >> 32);
    const u32 q0 = (u32)q, q1 = (u32)(q >> 32);
    // first pass: m = l0 * qneg32; (h1 h0 l1 l0) += m * (q1 q0); l0 becomes 0 and is dropped
    // second pass: the same one limb up; the result is (h1 h0)
    asm("{\n\t.reg .u32 m;\n\t"
        "mul.lo.u32 m, %0, %6;\n\t"
        "mad.lo.cc.u32 %0, m, %4, %0;\n\t"
        "madc.hi.cc.u32 %1, m, %4, %1;\n\t"
        "addc.cc.u32 %2, %2, 0;\n\t"
        "addc.u32 %3, %3, 0;\n\t"
        "mad.lo.cc.u32 %1, m, %5, %1;\n\t"
        "madc.hi.cc.u32 %2, m, %5, %2;\n\t"
        "addc.u32 %3, %3, 0;\n\t"
        "mul.lo.u32 m, %1, %6;\n\t"
        "mad.lo.cc.u32 %1, m, %4, %1;\n\t"
        "madc.hi.cc.u32 %2, m, %4, %2;\n\t"
        "addc.u32 %3, %3, 0;\n\t"
        "mad.lo.cc.u32 %2, m, %5, %2;\n\t"
        "madc.hi.u32 %3, m, %5, %3;\n\t}"
        : "+r"(l0), "+r"(l1), "+r"(h0), "+r"(h1)
        : "r"(q0), "r"(q1), "r"(qneg32));
    const u64 t = ((u64)h1 << 32) | h0;
    return t >= q ? t - q : t;
}

// A pointer kept whole in a thread's registers, so that loads around it take immediate offsets.  (Left to itself the compiler adds
// each offset to the part of the address that a warp shares: two instructions a load.)
template <typename T>
__device__ __forceinline__ const T* thread_pointer(const T* p) {
    asm("" : "+l"(p));
    return p;
}

// words that are read exactly once: not kept in L1, first to leave L2
__device__ __forceinline__ u64 stream_policy() {
    u64 pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}
__device__ __forceinline__ void ld_stream(const void* p, u64 policy, u32& lo, u32& hi) {
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v2.b32 {%0, %1}, [%2], %3;" : "=r"(lo), "=r"(hi) : "l"(p), "l"(policy));
}
__device__ __forceinline__ u32 ld_stream32(const void* p, u64 policy) {
    u32 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(v) : "l"(p), "l"(policy));
    return v;
}

// ---- Sums of products of residues, three ways.  fp64 multiply-adds and 32x32+64-bit integer ones issue at the same measured
// rate (62 and 63 per SM and clock), but a product takes four fp64 operations, on a pipe that these kernels leave idle
// otherwise, against three or four integer multiply-adds beside the cutting and adding of limbs, on the pipes that do the
// address arithmetic too: so the primes below 2^40 (all but one or two of a chain) multiply in fp64.
enum OperandClass : int { OP_DP = 0, OP_NARROW = 1, OP_WIDE = 2 };
constexpr u32 LIMB_NARROW = 25, LIMB_WIDE = 30;

// Primes below 2^40, operands integer-valued doubles.  The running sum h sits at 1.5 * 2^92, where doubles are 2^40 apart:
// h' = fma(a, b, h) adds a*b rounded to a multiple of 2^40 (exactly representable), h - h' is exact, and
// fma(a, b, h - h') is the part rounded away, an integer of magnitude at most 2^39; l collects those.  Exact while
// |sum| < 2^91 and |l| < 2^53: 2048 terms.
struct DpAcc {
    double h = 7427640235712281649394745344.0;       // 1.5 * 2^92
    double l = 0.0;
    __device__ __forceinline__ void mac(double a, double b) {
        const double h2 = __fma_rn(a, b, h);
        l = __dadd_rn(l, __fma_rn(a, b, __dsub_rn(h, h2)));
        h = h2;
    }
    // the sum modulo q as an integer-valued double, (h / 2^40) (2^40 mod q) + l: within 0.54q plus 2^39 a term.  The product takes
    // |h / 2^40| < 2^47, i.e. sums below 2^87: 128 products of residues below 2^40.  `many`: more than that, up to 2^91.
    __device__ __forceinline__ double lazy(double q, double qinv, double c40, double c40q, bool many) const {
        double hi = __fma_rn(h, 9.094947017729282379150390625e-13, -6755399441055744.0);       // (h - 1.5 * 2^92) 2^-40, exact
        if (many) hi = fp_centre(hi, q, qinv);
        return __dadd_rn(fp_mul_centred_signed(hi, c40, c40q, q), l);
    }
};

// 64-bit words cut into two limbs, 25 bits below 2^50 (NARROW), 30 bits up to 2^60 (WIDE).  NARROW: Karatsuba, three
// multiply-adds per product and no carries; a middle product is below 2^52, so the sums take 2^10 terms.  WIDE: four;
// products are below 2^60, so 15 terms fit, and the sum of up to 2^7 such sums fits 128 bits.
template <bool WIDE>
struct LimbAcc {
    u64 lo = 0, m0 = 0, m1 = 0, hi = 0;
    __device__ __forceinline__ void mac(u32 a0, u32 a1, u32 as, u32 b0, u32 b1) {      // (as = a0 + a1)
        lo += (u64)a0 * b0;
        hi += (u64)a1 * b1;
        if (WIDE) {
            m0 += (u64)a0 * b1;
            m1 += (u64)a1 * b0;
        } else {
            m0 += (u64)as * (b0 + b1);
        }
    }
    __device__ __forceinline__ unsigned __int128 value() const {
        typedef unsigned __int128 u128;
        return WIDE ? (u128)lo + ((u128)m0 << 30) + ((u128)m1 << 30) + ((u128)hi << 60)
                    : (u128)lo + ((u128)(m0 - lo - hi) << 25) + ((u128)hi << 50);
    }
    // times 2^-64, in [0, q)
    __device__ __forceinline__ u64 reduce(u64 q, u32 qneg32) const {
        const unsigned __int128 v = value();
        return redc_2x32((u64)(v >> 64), (u64)v, q, qneg32);
    }
};
__device__ __forceinline__ void cut_limbs(u32 lo, u32 hi, u32 L, u32& w0, u32& w1) {
    w0 = lo & ((1u << L) - 1u);
    w1 = __funnelshift_r(lo, hi, L);
}

// The 40-bit word of low half lo and high byte s % 4 of `high` as a double: 2^52 + the word, minus 2^52.
__device__ __forceinline__ void unpack40(u32 s, u32 high, u32& lo, u32& hi) {
    const double d = __dsub_rn(__hiloint2double((int)__byte_perm(high, 0x43300000u, 0x7650u + s % 4), (int)lo), 4503599627370496.0);
    lo = (u32)__double2loint(d);
    hi = (u32)__double2hiint(d);
}

// Resident rotation keys: [key][modulus][tile of KS_TILE coefficients], a tile holding the 2r segments s = 2 digit + component
// in turn.  The multiply-accumulate and the inner products read each key once and are bound by those bytes, so residues of
// primes below 2^40 (RingDev::dp) take five: the low 32 bits, [2r][KS_TILE] words, then the high bytes of four segments at a
// time, [(2r + 3) / 4][KS_TILE] words.  (Over the four calls of a 0.6B layer the keys are 60 % of the bytes.)  The others are
// 8-byte words with a factor 2^64.
__host__ __device__ __forceinline__ u32 key_tile_bytes(bool dp, u32 r) { return dp ? (2 * r + (2 * r + 3) / 4) * KS_TILE * 4 : 2 * r * KS_TILE * 8; }
__device__ __forceinline__ const unsigned char* key_tile(const RingDev& R, const void* keys, u32 key, u32 m, u32 tile) {
    return (const unsigned char*)keys + key * R.key_bytes + R.key_base[m] + (size_t)tile * key_tile_bytes(R.dp[m] != 0, R.r);
}
__device__ __forceinline__ void key_store(const RingDev& R, void* keys, u32 key, u32 m, u32 s, u32 n, u64 v) {      // v in [0, q)
    unsigned char* t = const_cast<unsigned char*>(key_tile(R, keys, key, m, n / KS_TILE));
    const u32 c = n % KS_TILE;
    if (R.dp[m]) {
        ((u32*)t)[s * KS_TILE + c] = (u32)v;
        t[((size_t)(2 * R.r + s / 4) * KS_TILE + c) * 4 + s % 4] = (unsigned char)(v >> 32);
    } else {
        ((u64*)t)[s * KS_TILE + c] = mul_shoup(v, R.c64[m], R.c64s[m], R.q[m]);
    }
}
// Coefficient c of a tile: the words of segments as they are stored (OP_DP: low words, and high[s / 4] with the high bytes),
// cut into the form KeyDot and DigitDot multiply.
template <int CLS>
struct KeyTile {
    const unsigned char* at;
    u32 r;
    __device__ __forceinline__ KeyTile(const unsigned char* tile, u32 c, u32 r_) : at(thread_pointer(tile + (CLS == OP_DP ? 4 : 8) * c)), r(r_) {}
    __device__ __forceinline__ u32 high(u32 group, u64 pol) const { return CLS == OP_DP ? ld_stream32(at + (2 * r + group) * KS_TILE * 4, pol) : 0u; }
    __device__ __forceinline__ void word(u32 s, u64 pol, u32& k0, u32& k1) const {
        if (CLS == OP_DP) k0 = ld_stream32(at + s * KS_TILE * 4, pol);
        else ld_stream(at + s * KS_TILE * 8, pol, k0, k1);
    }
    static __device__ __forceinline__ void cut(u32 s, u32 high, u32& k0, u32& k1) {
        if (CLS == OP_DP) {
            unpack40(s, high, k0, k1);
        } else {
            cut_limbs(k0, k1, CLS == OP_WIDE ? LIMB_WIDE : LIMB_NARROW, k0, k1);
        }
    }
};

// One output word of the key-switch inner product: digits times key words (cut), summed, in [0, q).  The keys carry a
// factor 2^64 except where the class is OP_DP; there the digits may be lazy, as a forward transform leaves them: within 13q, so
// that a sum of LAZY_DIGITS products stays below 2^87 (`many`: more of them; see DpAcc::lazy).  (Four fp64 operations and a
// conversion less for every point of a digit's transform: three rotations of 7 digits at N = 2^15 36.1 -> 34.0 us.)
constexpr u32 LAZY_DIGITS = 9;
template <int CLS>
struct DigitDot {
    static constexpr u32 L = CLS == OP_WIDE ? LIMB_WIDE : LIMB_NARROW;
    LimbAcc<CLS == OP_WIDE> a;
    __device__ __forceinline__ void mac(uint2 d, u32 k0, u32 k1) {
        u32 d0, d1;
        cut_limbs(d.x, d.y, L, d0, d1);
        a.mac(d0, d1, d0 + d1, k0, k1);
    }
    __device__ __forceinline__ u64 reduce(const RingDev& R, u32 m, bool) const { return a.reduce(R.q[m], (u32)R.qneg[m]); }
};
template <>
struct DigitDot<OP_DP> {
    DpAcc a;
    __device__ __forceinline__ void mac(uint2 d, u32 k0, u32 k1) { a.mac(__hiloint2double((int)d.y, (int)d.x), __hiloint2double((int)k1, (int)k0)); }
    __device__ __forceinline__ u64 reduce(const RingDev& R, u32 m, bool many) const {
        return d2u(fp_canonical(a.lazy(R.qd[m], R.qinv_d[m], R.c40_d[m], R.c40_q[m], many), R.qd[m], R.qinv_d[m]));
    }
};

// One output pair of the key-switch inner product: digit j (d[j * ds]) times key words (2j, 2j + 1) (k[s * ks]) summed
// over r digits, in [0, q).  The keys carry a factor 2^64 except where the class is OP_DP.
template <int CLS>
struct KeyDot {
    LimbAcc<CLS == OP_WIDE> a0, a1;
    __device__ __forceinline__ void mac(uint2 d, u32 k0, u32 k1, u32 l0, u32 l1) {     // (key limbs already cut)
        u32 d0, d1;
        cut_limbs(d.x, d.y, CLS == OP_WIDE ? LIMB_WIDE : LIMB_NARROW, d0, d1);
        a0.mac(d0, d1, d0 + d1, k0, k1);
        a1.mac(d0, d1, d0 + d1, l0, l1);
    }
    __device__ __forceinline__ void reduce(const RingDev& R, u32 m, u64& v0, u64& v1) const {
        v0 = a0.reduce(R.q[m], (u32)R.qneg[m]);
        v1 = a1.reduce(R.q[m], (u32)R.qneg[m]);
    }
};
template <>
struct KeyDot<OP_DP> {
    DpAcc a0, a1;
    __device__ __forceinline__ void mac(uint2 d, u32 k0, u32 k1, u32 l0, u32 l1) {
        const double dd = __hiloint2double((int)d.y, (int)d.x);
        a0.mac(dd, __hiloint2double((int)k1, (int)k0));
        a1.mac(dd, __hiloint2double((int)l1, (int)l0));
    }
};

}  // namespace bf
