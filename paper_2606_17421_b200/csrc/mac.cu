// Layout of cached plaintexts and dispatch of the multiply-accumulate (kernel: mac_kernel.cuh).
#include <cstring>

#include "mac_kernel.cuh"

namespace bf {

static int bits_of(u64 v) {
    int b = 0;
    while (v) { ++b; v >>= 1; }
    return b;
}

// Tile width: the X tile (n_terms * 2 * TN words) must stay within 48 KB so that four blocks share an SM, and a small
// ring is cut finer so that its tiles fill the machine.
static u32 mac_log_tn(const RingHost& ring, u32 n_terms, u32 n_primes) {
    u32 log_tn = 7;
    while (log_tn > 4 && (size_t)((n_terms + 7) / 8) * 16 * (1u << log_tn) * 8 > 48 * 1024) --log_tn;
    while (log_tn > 5 && (ring.dev.N >> log_tn) * n_primes < 148u * 3) --log_tn;
    return log_tn;
}

TileLayout mac_tile_layout(const RingHost& ring, u32 n_pj, u32 n_terms, u32 n_primes) {
    TileLayout t;
    memset(&t, 0, sizeof(t));
    t.n_primes = n_primes ? n_primes : ring.dev.r;
    t.log_tn = mac_log_tn(ring, n_terms, t.n_primes);
    const u32 PL = 256u >> t.log_tn;
    t.n_terms = n_terms;
    t.n_pj = n_pj;
    t.G = (n_pj + PL - 1) / PL;
    t.C = (n_terms + TILE_TS - 1) / TILE_TS;
    t.ntiles = ring.dev.N >> t.log_tn;
    t.stage_words = (n_pj < PL ? n_pj : PL) * TILE_TS << t.log_tn;
    for (u32 i = 0; i < t.n_primes; ++i) {
        const u32 f = ring.q[i] < (1ull << 32) ? TILE_W32 : ring.q[i] < (1ull << 40) ? TILE_W40 : TILE_W64;
        t.fmt_bits |= f << (2 * i);
        t.base[i + 1] = t.base[i] + (size_t)tile_stage_bytes(t, f) * t.ntiles * t.G * t.C;
    }
    return t;
}

size_t mac_tile_bytes(const TileLayout& t) { return tile_prime_base(t, t.n_primes); }

// (of the groups there are: the last stages' idle lanes, at most PL - 1 groups, are left out)
size_t mac_accounted_bytes(const RingHost& ring, const TileLayout& t) {
    size_t width = 0;
    for (u32 i = 0; i < t.n_primes; ++i) {
        const u32 f = tile_format(t, i);
        width += !ring.compact_cache || f == TILE_W64 ? 8 : f == TILE_W40 ? 5 : 4;
    }
    return width * ring.dev.N * t.n_pj * t.C * TILE_TS;
}

u32 mac_split_bits(const RingHost& ring) {
    u64 qmax = 0;
    for (u32 i = 0; i < ring.dev.r; ++i) qmax = ring.q[i] > qmax ? ring.q[i] : qmax;
    return bits_of(qmax) <= 50 ? LIMB_NARROW : LIMB_WIDE;
}

cudaError_t launch_mac_narrow(const MacLaunch& m) { return launch_mac_ring<true>(m); }

cudaError_t launch_mac(const RingHost& ring, const u64* pt, const TileLayout& lay, const u64* x, u64* a, u32 n_pj,
                       u32 n_terms, cudaStream_t stream, const MacScatter& sc, const BabySteps* baby) {
    if (n_pj == 0) return cudaSuccess;
    if (lay.n_pj != n_pj || lay.n_terms != n_terms) return cudaErrorInvalidValue;
    MacLaunch m;
    m.ring = &ring;
    m.pt = pt;
    m.lay = lay;
    m.x = x;
    m.a = a;
    m.n_pj = n_pj;
    m.n_terms = n_terms;
    m.sc = sc;
    memset(&m.bs, 0, sizeof(m.bs));
    m.baby = baby != nullptr;
    if (baby) {
        m.bs = *baby;
        // a lane of a block takes one (key, part of the inputs) at a time: the inputs are cut into parts only where the
        // keys alone would leave lanes idle (few baby steps, many inputs)
        const u32 lanes = 256u >> lay.log_tn, keys = baby->b - 1;
        u32 parts = keys && keys < 2 * lanes ? (2 * lanes + keys - 1) / keys : 1u;
        if (parts > baby->n_in) parts = baby->n_in;
        if (parts < 1) parts = 1;
        m.bs.per_part = (baby->n_in + parts - 1) / parts;
        m.bs.parts = (baby->n_in + m.bs.per_part - 1) / m.bs.per_part;
        if (ring.prof) ring.prof->mac_key_bytes += (u64)(baby->b - 1) * ring.dev.key_bytes;
    }
    m.stream = stream;
    ProfScope prof(ring.prof, CAT_MAC, stream);
    return mac_split_bits(ring) == LIMB_NARROW ? launch_mac_narrow(m) : launch_mac_wide(m);
}

}  // namespace bf
