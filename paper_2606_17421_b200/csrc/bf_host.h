// Host-side structures and kernel launchers shared by the translation units of libbifrost.
#pragma once
#include <cstddef>
#include <cstdint>
#include <map>
#include <vector>

#include "bf_common.cuh"

namespace bf {

// Kernel categories for launch counting and optional per-launch event timing.
enum KernelCat : int {
    CAT_NTT_FWD_STRIDED = 0, CAT_NTT_FWD_CONTIG, CAT_NTT_INV_CONTIG, CAT_NTT_INV_STRIDED,
    CAT_KEY_INNER, CAT_MAC, CAT_RESCALE,
    CAT_ENCODE_FFT_A, CAT_ENCODE_FFT_B, CAT_POINTWISE, CAT_DIVIDE, CAT_COUNT
};

struct Profiler {
    bool timing = false;
    uint64_t launches[CAT_COUNT] = {0};
    // key-switch inner products: bytes of rotation keys counted once per distinct key of a launch (what must come
    // from HBM) and once per rotation (what the launch reads, L2 hits included)
    uint64_t key_bytes_distinct = 0, key_bytes_per_rotation = 0;
    uint64_t mac_key_bytes = 0;       // the baby keys that multiply-accumulates read, once per key and launch
    struct Rec { int cat; cudaEvent_t a, b; };
    std::vector<Rec> recs;            // event pairs recorded since the last collection
    std::vector<cudaEvent_t> pool;    // idle events
    cudaEvent_t get();
};

// Counts a launch and, when timing is on, brackets it with two events on the launch stream.
struct ProfScope {
    Profiler* p; int cat; cudaStream_t s; cudaEvent_t a = nullptr;
    ProfScope(Profiler* prof, int c, cudaStream_t st);
    ~ProfScope();
};

struct RingHost {
    RingDev dev;
    std::vector<u64> q;               // q_0..q_L, then P
    Profiler* prof = nullptr;
    bool dependent_launch = true;     // launch the kernels of a call with programmatic stream serialisation
    bool compact_cache = false;       // cached plaintexts count for the bytes of their words, not for 8 a word
    int device = 0;                   // the CUDA device of the context (kernel attributes are set once per device)
};
constexpr int MAX_DEVICES = 64;
inline int device_slot(const RingHost& ring) { return ring.device >= 0 && ring.device < MAX_DEVICES ? ring.device : 0; }

// Launch with programmatic stream serialisation: the grid may be scheduled while the previous kernel
// of the stream drains; every kernel launched this way calls grid_dependency_enter() before it touches
// global memory, which waits until that previous kernel has completed and its writes are visible.
template <typename... KArgs, typename... Args>
static inline cudaError_t launch_dependent(const RingHost& ring, void (*kernel)(KArgs...), dim3 grid, dim3 block,
                                           size_t smem, cudaStream_t stream, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = ring.dependent_launch ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

// ---- ntt.cu
cudaError_t ntt_forward(const RingHost& ring, const PolyBatch& B, u32 n_outer, int load, cudaStream_t stream);
cudaError_t ntt_inverse(const RingHost& ring, const PolyBatch& B, u32 n_outer, cudaStream_t stream);
// Forward transform of the centred lifts of P-residues with the ModDown epilogue fused into its last store.
cudaError_t ntt_forward_moddown(const RingHost& ring, const PolyBatch& B, u32 n_outer, const RotBatch& rb,
                                const ModDownEpilogue& epi, cudaStream_t stream);
// Inverse transforms of the output assembly (see OutputAssembly; B: n_m = 2r + as.n_t() slots of every output, tail_m = 2r,
// store_centred = 2), and the division that ends it: ct[p][comp][i] = (ct[p][comp][i] - sum of the centred P-residues T[p][.])
// * P^{-1}, T the n_t polynomials per output, the first n_u of them of key-switch results.
// rc, low non-null: the rescale from r primes follows in the same kernel; the result goes to low ([n_out][2][r-1][N])
cudaError_t ntt_inverse_assembly(const RingHost& ring, const PolyBatch& B, u32 n_outer, const OutputAssembly& as, cudaStream_t stream);
cudaError_t finish_division(const RingHost& ring, u64* ct, long long ct_stride, const u64* T, u32 n_u, u32 n_t, u32 n_out,
                            cudaStream_t stream, const RescaleConsts* rc = nullptr, u64* low = nullptr);
// out = (u0, u1) / P + (phi(c0), 0), plus ct where `add`, for n_ct ciphertexts [2][r][N] in the coefficient domain: u, [2][r+1][N] each,
// is the rotated key-switch result with its residue modulo P as a centred lift plus 2^59.  out must not overlap ct.
cudaError_t finish_rotation(const RingHost& ring, const u64* u, const u64* ct, u64* out, u32 n_ct, u32 gal_inv, bool add, cudaStream_t stream);
cudaError_t ntt_forward_split(const RingHost& ring, const PolyBatch& B, u32 n_outer, int load, void* final_dst,
                              const u32* scatter, u32 scatter_div, cudaStream_t stream);

// The inputs of a double-hoisted call and their digits (see PolyBatch::ingest; B names source, buffers and outputs).
cudaError_t ntt_forward_ingest(const RingHost& ring, const PolyBatch& B, u32 n_in, cudaStream_t stream);
// First pass alone of a forward transform of digits (LOAD_REDUCE).
cudaError_t ntt_forward_first(const RingHost& ring, const PolyBatch& B, u32 n_outer, cudaStream_t stream);
// Digits of n_sets sets (B: LOAD_REDUCE from a shared source, B.dst = room for the [n_sets * r][r + 1][N] words between the
// passes; n_sets = 0: they are there already) transformed and multiplied with the rotation keys (pre-permuted, tile-major):
//   u[rb.out[rot]][comp][m][n] = sum_j NTT_m(digit j of set rb.dig[rot])[n] * key'[rb.key[rot]][j][comp][m][n]
// stored at pinv[rb.key[rot]][n] where pinv is non-null.  xext non-null (double hoisting, with pinv): the result is finished
// as a rotated input in the extended basis, xext[rb.out[rot]][comp][m][pinv[..][n]] = u'[comp][m][n] + (comp == 0 ?
// xext[rb.c0[rot]][0][m][n] : 0), terms of [2][r+1][N] words (term rb.c0[rot] holds P times the un-rotated input).
// Rotations of the same set have to be consecutive.
cudaError_t ntt_forward_inner(const RingHost& ring, const PolyBatch& B, u32 n_sets, const RotBatch& rb, const void* keys, u64* u, u64* xext,
                              const u32* pinv, cudaStream_t stream);

// ---- kernels.cu : element-wise and streaming kernels of the linear layer
// out[t] = a[t] * b[t] pointwise, polynomial t modulo basis prime mod0 + t % n_m
cudaError_t launch_pointwise_mul(const RingHost& ring, const u64* a, const u64* b, u64* out, u32 n_polys, u32 n_m,
                                 u32 mod0, cudaStream_t stream);
u32 mac_split_bits(const RingHost& ring);   // limb width of cached 8-byte words modulo primes below 2^50
// layout of n_pj groups of n_terms diagonals held in n_primes primes (0 = the r ciphertext primes)
TileLayout mac_tile_layout(const RingHost& ring, u32 n_pj, u32 n_terms, u32 n_primes = 0);
size_t mac_tile_bytes(const TileLayout& t);                                 // bytes that layout occupies
size_t mac_accounted_bytes(const RingHost& ring, const TileLayout& t);      // bytes its words count for: 8 each unless compact_cache
// a: [n_pj][2][lay.n_primes][N]; every prime of the layout is processed.  baby null: x holds all terms,
// [n_terms][2][lay.n_primes][N].  baby non-null: x holds the un-rotated inputs, [n_in][2][lay.n_primes][N], and the
// rotated terms are computed inside.
cudaError_t launch_mac(const RingHost& ring, const u64* pt, const TileLayout& lay, const u64* x, u64* a, u32 n_pj,
                       u32 n_terms, cudaStream_t stream, const MacScatter& sc, const BabySteps* baby = nullptr);
cudaError_t launch_rescale(const RingHost& ring, const u64* in, u64* out, u32 n_ct, u32 level, const u64* inv,
                           const u64* invs, const u64* qlmod, cudaStream_t stream);

// 32-bit <-> 64-bit signed coefficients (the coefficient form of cached weights); narrowing sets *overflow_flag when a
// value does not fit
cudaError_t launch_widen_i32(const RingHost& ring, const int* src, i64* dst, size_t count, cudaStream_t stream);
cudaError_t launch_narrow_i64(const RingHost& ring, const i64* src, int* dst, size_t count, int* overflow_flag,
                              cudaStream_t stream);
cudaError_t launch_imad_probe(u64* sink, u32 blocks, u32 iters, cudaStream_t stream);   // 64 mad.wide per iteration and thread
cudaError_t launch_fma64_probe(u64* sink, u32 blocks, u32 iters, cudaStream_t stream);  // 64 fma.rn.f64 per iteration and thread

// ---- encode.cu : canonical-embedding encoder (fp64) for weight diagonals
struct EncodeTables {
    const u32* slot_of_pos;           // [n] slot index whose value sits at FFT input position a
    const double2* T;                 // [n/2] (cos, -sin)(2 pi t / n)
    const double2* Z;                 // [n]   (cos, -sin)(pi k / N)
    double scale_over_n;
};
struct DiagBatch {                    // diagonals d0 .. d0+count-1 in [j][p][q][k] order
    const float* W;
    u32 d_out, d_in, n_in, n_out, D, tau, b, g;
    u32 d0, count;
    u32 complex_pack;                 // two row blocks per plaintext: block 2p in the real parts, 2p+1 in the imaginary
};
cudaError_t launch_encode(const RingHost& ring, const EncodeTables& tab, const DiagBatch& db, double2* fft_scratch,
                          i64* coeff_out, int* overflow_flag, cudaStream_t stream);

}  // namespace bf
