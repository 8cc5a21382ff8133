// Multiply-accumulate over encoded diagonals (the ciphertext x plaintext product of Sec. 3.5 / 4.2),
//   A[pj][comp][i][n] = sum_{t < n_terms} Pt[pj][t][i][n] * X[t][comp][i][n]   (mod q_i),
// with the baby rotations that make X computed in the same kernel where the plan allows (BABY: double hoisting).
//
// A block owns one prime i and a tile of TN adjacent coefficients, for all output groups.  It first fills the X tile of
// all terms and both components in shared memory, then streams its contiguous region of the cached weights once.
//
// BABY: rotated input (q, k) is (P c0 + u0, u1) moved through the automorphism of its rotation, u the key-switch inner
// product of the digits of input q with key k.  In the transform's bit-reversed order an automorphism maps every
// aligned power-of-two block of positions onto another aligned block: position n holds the evaluation at exponent
// 2 brev(n) + 1, adjacent positions differ in the exponent's top bits only, and multiplying by an odd number keeps
// equal low bits equal.  So the tile of X needs exactly one tile of every key and of every digit; the block reads those
// in place, coalesced, and permutes inside the tile on the way to shared memory.  X itself (2 (r+1) N words per term) is
// never written to memory.
//
// What bounds it: the stream where one input meets the keys, issue where several do.  In one layer of a 0.6B decoder (N = 2^15, r = 7,
// 5 bytes a word modulo the primes below 2^40) 1024 -> 4096 reads 534 MB of keys and weights in 110 us, 4.9 TB/s, and 1024 -> 6144 with 31
// keys 974 MB in 187 us, 5.2 TB/s, where a plain sequential read reaches 5.5; two and three inputs 4.2 and 3.8 TB/s, with 58 to 62 % of the
// issue slots taken, 45 % of the warps resident and waits for loads ahead of every other stall.  Loads go straight to registers: a
// stream that every thread consumes in the pattern it loads needs no staging, no barriers and no producer; what hides the latency
// is the number of independent loads per thread (2r key words at a time; two batches of 8 weights, three where they are packed)
// times resident warps.
// Since issue slots come next, index arithmetic is done per warp where it can be, X is held as pairs of its two components (one
// 16-byte read per weight), and what stays in the block is only reduced as far as its next use needs: the four products of a 0.6B
// layer take 55 us less than with canonical residues, divisions for an item's place and an automorphism evaluated per
// coefficient (the layer 1373 -> 1314 us, one of an 8B model 9430 -> 9087 us).  Tiles of 16 differ in two of these: see XRow.
#pragma once
#include "bf_host.h"

#include <type_traits>

namespace bf {

constexpr int MAC_THREADS = 256;

// Position n holds the evaluation at exponent e = 2 brev(n) + 1; an automorphism X -> X^gal moves to it the one at e * gal, and
// with the inverse exponent that is where it goes.  The positions n0 + c of an aligned tile have exponents e0 + brev(c) 2^k,
// k = log2(2N / tile): their images lie in the tile whose first position is `tile`, at brev(brev(c) * gal + top) inside it.  All
// but that last step is the same for the whole tile.
template <int LOG_TN>
struct TileMove {
    u32 tile, top, gal;
    __device__ __forceinline__ TileMove(u32 n0, u32 gal_, u32 logN) : gal(gal_) {
        const u32 e = ((2u * (__brev(n0) >> (32u - logN)) + 1u) * gal) & ((2u << logN) - 1u);
        tile = (__brev(e >> 1) >> (32u - logN)) & ~((1u << LOG_TN) - 1u);
        top = e >> (logN + 1 - LOG_TN);
    }
    __device__ __forceinline__ u32 inside(u32 c_rev) const { return __brev(c_rev * gal + top) >> (32 - LOG_TN); }     // c_rev = brev(c)
};

// g^j modulo 2^32
__device__ __forceinline__ u32 power32(u32 g, u32 j) {
    u32 v = j & 1u ? g : 1u;
    while (j >>= 1) {
        g *= g;
        if (j & 1u) v *= g;
    }
    return v;
}

// Accumulator of one output word of the multiply-accumulate and the form its operands have: weights as stored (two
// 32-bit halves), the X word as it sits in shared memory (x_word: of a residue; x_stored: of a word of the un-rotated inputs, which
// are residues except modulo primes of class OP_DP, where they are doubles).
template <int CLS>
struct MacAcc {                                          // OP_NARROW
    static constexpr u32 L = LIMB_NARROW;
    LimbAcc<false> a;
    __device__ __forceinline__ void mac(u32 w0, u32 w1, u64 x) { a.mac(w0, w1, w0 + w1, (u32)x, (u32)(x >> 32)); }
    __device__ __forceinline__ void end_chunk(const RingDev&, u32, u32) {}
    __device__ __forceinline__ u64 reduce(const RingDev& R, u32 i, bool) const { return a.reduce(R.q[i], (u32)R.qneg[i]); }
    static __device__ __forceinline__ u64 x_word(u64 v) { return limb_split(v, L); }
    static __device__ __forceinline__ u64 x_stored(u64 v) { return x_word(v); }
};
template <>
struct MacAcc<OP_WIDE> {
    // a chunk of 8 terms keeps every sum below 2^64 (16 middle products below 2^60), then it is folded into 128 bits;
    // 128 terms of 120 bits fit there, and the reduction at the end wants the high half below q
    static constexpr u32 L = LIMB_WIDE;
    LimbAcc<true> a;
    unsigned __int128 v = 0;
    __device__ __forceinline__ void mac(u32 w0, u32 w1, u64 x) {
        const u32 x0 = (u32)x, x1 = (u32)(x >> 32);
        a.lo += (u64)w0 * x0;
        a.m0 += (u64)w0 * x1;
        a.m0 += (u64)w1 * x0;
        a.hi += (u64)w1 * x1;
    }
    __device__ __forceinline__ void end_chunk(const RingDev& R, u32 i, u32 chunk) {
        v += a.value();
        a = {};
        if ((chunk & 15u) == 15u) v = ((unsigned __int128)barrett64((u64)(v >> 64), R.q[i], R.mu[i]) << 64) | (u64)v;
    }
    __device__ __forceinline__ u64 reduce(const RingDev& R, u32 i, bool) const {
        return redc_2x32(barrett64((u64)(v >> 64), R.q[i], R.mu[i]), (u64)v, R.q[i], (u32)R.qneg[i]);
    }
    static __device__ __forceinline__ u64 x_word(u64 v) { return limb_split(v, L); }
    static __device__ __forceinline__ u64 x_stored(u64 v) { return x_word(v); }
};
template <>
struct MacAcc<OP_DP> {
    DpAcc a;
    __device__ __forceinline__ void mac(u32 w0, u32 w1, u64 x) {
        a.mac(__hiloint2double((int)w1, (int)w0), __longlong_as_double((long long)x));
    }
    __device__ __forceinline__ void end_chunk(const RingDev&, u32, u32) {}
    __device__ __forceinline__ u64 reduce(const RingDev& R, u32 i, bool many) const {
        return d2u(fp_canonical(a.lazy(R.qd[i], R.qinv_d[i], R.c40_d[i], R.c40_q[i], many), R.qd[i], R.qinv_d[i]));
    }
    static __device__ __forceinline__ u64 x_word(u64 v) { return (u64)__double_as_longlong(u2d(v)); }
    static __device__ __forceinline__ u64 x_stored(u64 v) { return v; }
};

// A row of the tile fills a warp: its threads share their lane, and what depends on the lane is worked out once for all of them.
__host__ __device__ constexpr bool warp_has_one_lane(int log_tn) { return log_tn >= 5; }

// The X tile: [term][TN] pairs (component 0, component 1), one 16-byte read per weight; rows of 16, [term][component][TN] words, because
// the halves of a warp read such a row alike and 8-byte reads serve both at once.  (Tiles of 16, a product of 4096 -> 1024 in 128 terms on
// 2^15, us: without rotations inside 371 with pairs and what a lane needs carried along as below, 330 like this; with them 686 and 633.)
template <int LOG_TN>
struct XRow {
    static constexpr bool PAIRS = warp_has_one_lane(LOG_TN);
    static constexpr u32 TN = 1u << LOG_TN, WORDS = PAIRS ? TN : 2 * TN;
    typedef typename std::conditional<PAIRS, ulonglong2, u64>::type Word;
    static __device__ __forceinline__ void put(Word* at, ulonglong2 v) {
        if constexpr (PAIRS) *at = v;
        else { at[0] = v.x; at[TN] = v.y; }
    }
    static __device__ __forceinline__ ulonglong2 get(const Word* at) {
        if constexpr (PAIRS) return *at;
        else return make_ulonglong2(at[0], at[TN]);
    }
};

template <int CLS, int LOG_TN, bool BABY, int RC>
__device__ __forceinline__ void mac_body(const RingDev& R, const u64* __restrict__ pt, const TileLayout& lay,
                                         const u64* __restrict__ x, u64* __restrict__ a, u32 n_terms, u32 pj_begin, u32 pj_end,
                                         u32 tile, u32 i, const MacScatter& sc, const BabySteps& bs, typename XRow<LOG_TN>::Word* xs) {
    constexpr u32 TN = 1u << LOG_TN, PL = MAC_THREADS >> LOG_TN;
    typedef MacAcc<CLS> Acc;
    typedef XRow<LOG_TN> Row;
    constexpr u32 RW = Row::WORDS;
    const u32 N = R.N, logN = R.logN;
    const u32 np = lay.n_primes;
    const u32 tid = threadIdx.x, c = tid & (TN - 1), c_rev = __brev(c) >> (32 - LOG_TN);
    u32 l = tid >> LOG_TN;
    constexpr bool ONE_LANE = warp_has_one_lane(LOG_TN);
    if constexpr (ONE_LANE) l = __shfl_sync(0xffffffffu, l, 0);
    const u32 n0 = tile << LOG_TN;
    const u64 pol = stream_policy();
    if constexpr (BABY) {
        const u32 r = RC > 0 ? (u32)RC : R.r;
        const u32 b = bs.b, n_in = bs.n_in;
        // term (q, 0): P times the un-rotated input (zero modulo P, and not stored there)
        const u64* xg = x + (size_t)i * N + c;
        const size_t comp_stride = (size_t)np * N;
        for (u32 e = l; e < n_in; e += PL) {
            const u64* xp = xg + e * 2 * comp_stride + n0;
            Row::put(xs + e * b * RW + c, i < r ? make_ulonglong2(Acc::x_stored(__ldg(xp)), Acc::x_stored(__ldg(xp + comp_stride)))
                                                : make_ulonglong2(Acc::x_word(0), Acc::x_word(0)));
        }
        // rotations: an item is a key and a part of the inputs that share it.  The tile has the exponents e0 + brev(c) 2^k; a
        // rotation reads the tile of e0 * gal, whose own first exponent is that less its top bits T, so that the word at c there
        // goes to brev((brev(c) - T) / gal) here (see TileMove)
        const u32 parts = bs.parts, per_part = bs.per_part;
        const size_t dig_stride = ks_tile_base(N, r + 1, r, 1u, 0u, 0u);
        const u64* dig0 = bs.dig + ks_tile_base(N, r + 1, r, 0u, 0u, i) + c;
        const unsigned char* key0 = (const unsigned char*)bs.keys + R.key_base[i];
        const u32 e0 = 2u * (__brev(n0) >> (32u - logN)) + 1u, tile_bytes = key_tile_bytes(CLS == OP_DP, r);
        u32 k = 1, part = l;
        const u32 step_k = PL / parts, step_part = PL % parts;      // (used by tiles of 16)
        if constexpr (!ONE_LANE) { k += l / parts; part = l % parts; }
        for (;;) {
            if constexpr (ONE_LANE) {
                while (part >= parts) { part -= parts; ++k; }
            }
            if (k >= b) break;
            const u32 e = (e0 * bs.gal[k]) & ((2u << logN) - 1u), T = e >> (logN + 1 - LOG_TN);
            const u32 src = (__brev(e >> 1) >> (32u - logN)) & ~(TN - 1), ks = src / KS_TILE, in_tile = src % KS_TILE;
            const u32 cd = __brev((c_rev - T) * bs.gal_inv[k]) >> (32 - LOG_TN);
            const KeyTile<CLS> kt(key0 + bs.key_at[k] + ks * tile_bytes, in_tile + c, r);
            const u32 q0 = part * per_part, q_end = min(n_in, q0 + per_part);
            const u64* dp = dig0 + q0 * dig_stride + ks * (r * KS_TILE) + in_tile;
            const u64* cp = xg + q0 * 2 * comp_stride + src;
            typename Row::Word* xp = xs + (q0 * b + k) * RW + cd;
            u32 k0[RC > 0 ? 2 * RC : 1], k1[RC > 0 ? 2 * RC : 1];
            if constexpr (RC > 0) {
                u32 high[(2 * RC + 3) / 4];
#pragma unroll
                for (int s = 0; s < 2 * RC; ++s) kt.word(s, pol, k0[s], k1[s]);
#pragma unroll
                for (int h = 0; h < (2 * RC + 3) / 4; ++h) high[h] = kt.high(h, pol);
#pragma unroll
                for (int s = 0; s < 2 * RC; ++s) KeyTile<CLS>::cut(s, high[s / 4], k0[s], k1[s]);
            }
            for (u32 qi = q0; qi < q_end; ++qi, dp += dig_stride, cp += 2 * comp_stride, xp += b * RW) {
                KeyDot<CLS> dot;
                const u64 pc0 = i < r ? __ldg(cp) : 0ull;
                if constexpr (RC > 0) {
                    uint2 dw[RC];
#pragma unroll
                    for (int j = 0; j < RC; ++j) dw[j] = __ldg((const uint2*)(dp + j * KS_TILE));
#pragma unroll
                    for (int j = 0; j < RC; ++j) dot.mac(dw[j], k0[2 * j], k1[2 * j], k0[2 * j + 1], k1[2 * j + 1]);
                } else {
#pragma unroll 4
                    for (u32 j = 0; j < r; ++j) {
                        uint2 ka, kb;
                        kt.word(2 * j, pol, ka.x, ka.y);
                        kt.word(2 * j + 1, pol, kb.x, kb.y);
                        const u32 high = kt.high(j / 2, pol);
                        KeyTile<CLS>::cut(2 * j, high, ka.x, ka.y);
                        KeyTile<CLS>::cut(2 * j + 1, high, kb.x, kb.y);
                        dot.mac(__ldg((const uint2*)(dp + j * KS_TILE)), ka.x, ka.y, kb.x, kb.y);
                    }
                }
                if constexpr (CLS == OP_DP) {           // (centred: what the weights multiply may have either sign)
                    const double qd = R.qd[i], qinv = R.qinv_d[i], c40 = R.c40_d[i], c40q = R.c40_q[i];
                    const double v0 = __dadd_rn(dot.a0.lazy(qd, qinv, c40, c40q, r > LAZY_DIGITS), __longlong_as_double((long long)pc0));
                    const double v1 = dot.a1.lazy(qd, qinv, c40, c40q, r > LAZY_DIGITS);
                    Row::put(xp, make_ulonglong2((u64)__double_as_longlong(fp_centre(v0, qd, qinv)), (u64)__double_as_longlong(fp_centre(v1, qd, qinv))));
                } else {
                    u64 v0, v1;
                    dot.reduce(R, i, v0, v1);
                    Row::put(xp, make_ulonglong2(Acc::x_word(add_mod(v0, pc0, R.q[i])), Acc::x_word(v1)));
                }
            }
            if constexpr (ONE_LANE) part += PL;
            else {
                k += step_k;
                part += step_part;
                if (part >= parts) { part -= parts; ++k; }
            }
        }
    } else {
        // X tile: all of a thread's words are requested in batches, one round trip each
        const u64* xg = x + (size_t)i * N + n0 + c;
        const size_t comp_stride = (size_t)np * N;
        u32 e = l;
        for (; e + 3 * PL < n_terms; e += 4 * PL) {
            u64 v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = __ldg(xg + ((size_t)(e + j / 2 * PL) * 2 + j % 2) * comp_stride);
#pragma unroll
            for (int j = 0; j < 4; ++j) Row::put(xs + (e + j * PL) * RW + c, make_ulonglong2(Acc::x_word(v[2 * j]), Acc::x_word(v[2 * j + 1])));
        }
        for (; e < n_terms; e += PL) {
            const u64* xp = xg + (size_t)e * 2 * comp_stride;
            Row::put(xs + e * RW + c, make_ulonglong2(Acc::x_word(__ldg(xp)), Acc::x_word(__ldg(xp + comp_stride))));
        }
    }
    // terms up to a whole chunk are zero, and so are the padding words of a group's last stage once they are in registers
    for (u32 e = n_terms + l; e < TILE_TS * lay.C; e += PL) Row::put(xs + e * RW + c, make_ulonglong2(0, 0));
    __syncthreads();

    // ---------------- the weight stream: a lane's words of successive stages lie one stage apart
    if (pj_begin + l >= pj_end) return;
    // (primes of class OP_DP have 4 or 5 bytes a word, the others 8: see TileLayout)
    constexpr bool PACKED = CLS == OP_DP;
    const u32 fmt = tile_format(lay, i);
    const u32 n_chunks = lay.C;
    u32 left = ((pj_end - pj_begin - l + PL - 1) / PL) * n_chunks;      // stages to go
    const u32 stage_bytes = tile_stage_bytes(lay, fmt);
    const unsigned char* stage = (const unsigned char*)pt + tile_prime_base(lay, i) +
                                 ((size_t)tile * lay.G + pj_begin / PL) * n_chunks * stage_bytes;
    stage += tile_word_offset(lay, fmt, l, 0, c);       // (the lane's words of a stage lie together)
    constexpr int TS = (int)TILE_TS, TH = PACKED ? TS / 4 : TS;
    // one stage's words of this thread, as they are stored
    auto fetch = [&](u32 (&wa)[TS], u32 (&wb)[TH]) {
        if constexpr (PACKED) {
            const u32* p = (const u32*)stage;
#pragma unroll
            for (int ts = 0; ts < TS; ++ts) wa[ts] = ld_stream32(p + ts * TN, pol);
#pragma unroll
            for (int h = 0; h < TH; ++h) wb[h] = fmt == TILE_W40 ? ld_stream32(p + (TS + h) * TN, pol) : 0u;
        } else {
            const u64* p = (const u64*)stage;
#pragma unroll
            for (int ts = 0; ts < TS; ++ts) ld_stream(p + ts * TN, pol, wa[ts], wb[ts]);
        }
        stage += stage_bytes;
    };
    Acc a0, a1;
    u32 ch = 0;
    const size_t comp1 = (size_t)np * N;                // from component 0 to component 1
    u32 pj = pj_begin + l;
    u64* ap = a + ((size_t)pj * 2 * np + i) * N;
    const typename Row::Word* xt = xs + c;
    const u32 tail = n_terms % TILE_TS;
    // the giant step of group pj and the Galois element of its rotation (see MacScatter): carried along from group to group where
    // a warp's threads share them, else (they would take registers of every thread) made when the group ends
    u32 step_rem = 0, step_gal = 1, step = 0;
    auto set_step = [&] {
        if (!sc.on) return;
        step = (sc.pj0 + pj) / sc.n_out;
        step_rem = sc.pj0 + pj - step * sc.n_out;
        step_gal = power32(sc.gal_inv, step);
    };
    if constexpr (ONE_LANE) set_step();
    auto use = [&](u32 (&wa)[TS], u32 (&wb)[TH]) {
        if constexpr (!PACKED) {        // (packed padding is a finite number times a zero of X, whatever it is)
            if (tail && ch + 1 == n_chunks) {
#pragma unroll
                for (int ts = 1; ts < TS; ++ts)
                    if ((u32)ts >= tail) wa[ts] = wb[ts] = 0;
            }
        }
#pragma unroll
        for (int ts = 0; ts < TS; ++ts) {
            u32 w0 = wa[ts], w1 = wb[PACKED ? ts / 4 : ts];
            if constexpr (PACKED) unpack40(ts, w1, w0, w1);
            const ulonglong2 xw = Row::get(xt + ts * RW);
            a0.mac(w0, w1, xw.x);
            a1.mac(w0, w1, xw.y);
        }
        a0.end_chunk(R, i, ch);
        a1.end_chunk(R, i, ch);
        xt += TS * RW;
        if (++ch == n_chunks) {
            if constexpr (!ONE_LANE) {
                set_step();
                ap = a + ((size_t)pj * 2 * np + i) * N;
                pj += PL;
            }
            u32 at0 = n0 + c;                                           // where component 0 goes (see MacScatter)
            if (step) {
                const TileMove<LOG_TN> to(n0, step_gal, logN);
                at0 = to.tile + to.inside(c_rev);
            }
            ap[at0] = a0.reduce(R, i, n_terms > 128);
            ap[comp1 + n0 + c] = a1.reduce(R, i, n_terms > 128);
            if constexpr (ONE_LANE) ap += 2 * PL * comp1;
            a0 = {};
            a1 = {};
            if (ONE_LANE && sc.on)
                for (step_rem += PL; step_rem >= sc.n_out; step_rem -= sc.n_out) {
                    step_gal *= sc.gal_inv;
                    ++step;
                }
            ch = 0;
            xt = xs + c;
        }
    };
    // batches in flight: packed words leave registers for a third
    constexpr int NB = PACKED ? 3 : 2;
    u32 wa[NB][TS], wb[NB][TH];
#pragma unroll
    for (int s = 0; s + 1 < NB; ++s)
        if (left > (u32)s) fetch(wa[s], wb[s]);
    for (;;) {
#pragma unroll
        for (int s = 0; s < NB; ++s) {
            if (left > (u32)(NB - 1)) fetch(wa[(s + NB - 1) % NB], wb[(s + NB - 1) % NB]);
            use(wa[s], wb[s]);
            if (--left == 0) return;
        }
    }
}

// grid: x = slice of the output groups * tiles * primes, primes fastest: the blocks that share an SM then work in different
// operand classes, i.e. on different pipes (4 % of the kernel against tiles fastest on a 1024 -> 6144 product).
// Four blocks an SM (64 registers, which the key part of up to 9 digits fits in tiles of 32 and more; in tiles of 16 it spills 4
// bytes at 7 digits and 196 at 9) because resident warps are what hides the latency: two,
// three and four blocks took 791, 671 and 653 us over the four products of a 0.6B decoder layer (N = 2^15, r = 7; 3.34 GB of
// keys and weights), where the separate inner product and multiply-accumulate this kernel replaces took 867 us.
template <bool NARROW, int LOG_TN, bool BABY, int RC>
__global__ void __launch_bounds__(MAC_THREADS, 4)
mac_kernel(const __grid_constant__ RingDev R, const u64* __restrict__ pt, const __grid_constant__ TileLayout lay,
           const u64* __restrict__ x, u64* __restrict__ a, u32 n_terms, u32 n_pj, u32 pj_per_block,
           const __grid_constant__ MacScatter sc, const __grid_constant__ BabySteps bs) {
    extern __shared__ __align__(128) u64 mac_xs_words[];
    typename XRow<LOG_TN>::Word* mac_xs = (typename XRow<LOG_TN>::Word*)mac_xs_words;
    grid_dependency_enter();
    const u32 tiles_log = R.logN - LOG_TN;
    const u32 i = lay.n_primes - 1 - blockIdx.x % lay.n_primes;
    const u32 tile = (blockIdx.x / lay.n_primes) & ((1u << tiles_log) - 1u), slice = (blockIdx.x / lay.n_primes) >> tiles_log;
    const u32 pj_begin = slice * pj_per_block, pj_end = min(n_pj, pj_begin + pj_per_block);
    if (R.dp[i]) mac_body<OP_DP, LOG_TN, BABY, RC>(R, pt, lay, x, a, n_terms, pj_begin, pj_end, tile, i, sc, bs, mac_xs);
    // (the class follows the words' limbs, as the tile store cuts them: 25 bits below 2^50 where every ciphertext prime is, the
    // special prime included, else 30)
    else if (NARROW && !(R.q[i] >> 50)) mac_body<OP_NARROW, LOG_TN, BABY, RC>(R, pt, lay, x, a, n_terms, pj_begin, pj_end, tile, i, sc, bs, mac_xs);
    else mac_body<OP_WIDE, LOG_TN, BABY, RC>(R, pt, lay, x, a, n_terms, pj_begin, pj_end, tile, i, sc, bs, mac_xs);
}

struct MacLaunch {
    const RingHost* ring;
    const u64* pt;
    TileLayout lay;
    const u64* x;
    u64* a;
    u32 n_pj, n_terms;
    MacScatter sc;
    BabySteps bs;
    bool baby;
    cudaStream_t stream;
};

template <bool NARROW, int LOG_TN, bool BABY, int RC>
static cudaError_t launch_mac_t(const MacLaunch& m) {
    constexpr u32 TN = 1u << LOG_TN, PL = MAC_THREADS >> LOG_TN;
    const RingHost& ring = *m.ring;
    const size_t smem = (size_t)m.lay.C * TILE_TS * 2 * TN * 8;
    if (smem > 200 * 1024) return cudaErrorInvalidValue;
    static bool attr_set[MAX_DEVICES] = {false};     // opt in once per device to the large dynamic shared-memory carve-out
    if (!attr_set[device_slot(ring)]) {
        cudaError_t e = cudaFuncSetAttribute(mac_kernel<NARROW, LOG_TN, BABY, RC>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        if (e != cudaSuccess) return e;
        attr_set[device_slot(ring)] = true;
    }
    // slices over the output groups where the tiles alone are fewer than three rounds of blocks (every slice reads the X tile
    // again, which is little beside its weights; where the block makes X it is not): the primes beyond 2^50 take several times
    // as long as the others, and one round ends with them alone (N = 2^13, 48 groups of 16 terms: 66 us in one, 50 us in three)
    const u32 tiles = (ring.dev.N >> LOG_TN) * m.lay.n_primes;
    u32 slices = BABY ? 1u : (148u * 12 + tiles - 1) / tiles;
    const u32 max_slices = (m.n_pj + PL - 1) / PL;
    if (slices > max_slices) slices = max_slices;
    if (slices < 1) slices = 1;
    u32 per = (m.n_pj + slices - 1) / slices;
    per = (per + PL - 1) / PL * PL;
    slices = (m.n_pj + per - 1) / per;
    return launch_dependent(ring, mac_kernel<NARROW, LOG_TN, BABY, RC>, dim3(tiles * slices), dim3(MAC_THREADS), smem,
                            m.stream, ring.dev, m.pt, m.lay, m.x, m.a, m.n_terms, m.n_pj, per, m.sc, m.bs);
}

template <bool NARROW, bool BABY, int RC>
static cudaError_t launch_mac_tile(const MacLaunch& m) {
    switch (m.lay.log_tn) {
        case 7: return launch_mac_t<NARROW, 7, BABY, RC>(m);
        case 6: return launch_mac_t<NARROW, 6, BABY, RC>(m);
        case 5: return launch_mac_t<NARROW, 5, BABY, RC>(m);
        default: return launch_mac_t<NARROW, 4, BABY, RC>(m);
    }
}

// The 2 r key words of a rotation in registers, asked for together and once for all inputs it is applied to: an instance for every digit
// count up to 11.  Beyond that too many are spilled (in tiles of 32 and more at most 4 bytes up to 9 digits, 172 at 10, 296 at 11, 352 at
// 12) and a loop over the digits is used, which asks for the words again for every input.  us with the loop and with an instance, one input
// and 1024 -> 2048 on 2^15: 2 digits 95 and 87, 3 125 and 113, 5 168 and 157, 6 205 and 180, 8 256 and 244, 10 363 and 338, 11 433 and
// 396, 12 441 and 452.
constexpr int MAC_MOST_DIGITS = 11;
template <bool NARROW, int RC>
static cudaError_t launch_mac_digits(const MacLaunch& m) {
    if (m.ring->dev.r == RC) return launch_mac_tile<NARROW, true, RC>(m);
    if constexpr (RC < MAC_MOST_DIGITS) return launch_mac_digits<NARROW, RC + 1>(m);
    else return launch_mac_tile<NARROW, true, 0>(m);
}

template <bool NARROW>
static cudaError_t launch_mac_ring(const MacLaunch& m) {
    if (!m.baby) return launch_mac_tile<NARROW, false, 0>(m);
    return launch_mac_digits<NARROW, 2>(m);
}

cudaError_t launch_mac_narrow(const MacLaunch& m);      // every ciphertext prime below 2^50
cudaError_t launch_mac_wide(const MacLaunch& m);

}  // namespace bf
