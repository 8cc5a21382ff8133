// Element-wise kernels of the encrypted linear layer: the rescale (Sec. 2.1), width changes of cached coefficients.
#include "bf_host.h"

#include <cstring>

namespace bf {

// ------------------------------------------------------------------------------------------------
// Pointwise product of NTT-domain polynomials (parity helper for the transform).
__global__ void pointwise_mul_kernel(const RingDev R, const u64* __restrict__ a, const u64* __restrict__ b,
                                     u64* __restrict__ out, u32 n_m, u32 mod0) {
    const u32 poly = blockIdx.y;
    const u32 mod = mod0 + poly % n_m;
    const size_t idx = (size_t)poly * R.N + blockIdx.x * blockDim.x + threadIdx.x;
    u64 hi = 0, lo = 0;
    mac128(hi, lo, a[idx], b[idx]);
    out[idx] = reduce128(hi, lo, R.q[mod], R.mu[mod], R.c64[mod], R.c64s[mod]);
}

cudaError_t launch_pointwise_mul(const RingHost& ring, const u64* a, const u64* b, u64* out, u32 n_polys, u32 n_m,
                                 u32 mod0, cudaStream_t stream) {
    if (n_polys == 0) return cudaSuccess;
    dim3 grid(ring.dev.N / 256, n_polys);
    ProfScope prof(ring.prof, CAT_POINTWISE, stream);
    pointwise_mul_kernel<<<grid, 256, 0, stream>>>(ring.dev, a, b, out, n_m, mod0);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// Rescale (Sec. 2.1): drop the last prime q_L of a level-`level` ciphertext in coefficient form,
//   c'_i = (c_i - centred(c_L)) * q_L^{-1} mod q_i.
// Every address a thread touches is congruent to its coefficient index modulo N, and it reads all
// residues of that coefficient before writing, so one ciphertext can be rescaled in place even
// though the output is packed more tightly ([2][level-1][N]).

// `in` and `out` may alias, hence no __restrict__.  When they do and several ciphertexts are
// rescaled, the launch uses one thread per coefficient that walks the ciphertexts in order
// (n_seq > 1): the packed output of ciphertext t never reaches the input of ciphertext t+1.
__global__ void __launch_bounds__(256) rescale_kernel(const RingDev R, const RescaleConsts rc, const u64* in, u64* out,
                                                      u32 level, u32 n_seq) {
    grid_dependency_enter();
    const u32 N = R.N;
    const u32 n = blockIdx.x * blockDim.x + threadIdx.x;
    const u64 qL = R.q[level - 1];
  for (u32 ct = blockIdx.y; ct < blockIdx.y + n_seq; ++ct) {
    const u64* ip = in + (size_t)ct * 2 * level * N + n;
    u64* op = out + (size_t)ct * 2 * (level - 1) * N + n;
    // In place the packed output of residue (comp, i) lands where residue (comp, i) (component 0) or (comp, i - 1)
    // (component 1) was read, and the dropped residues are read before anything of their component is written: so
    // each residue is read, then its slot (or an earlier one) written, in order, with nothing held back.
#pragma unroll
    for (int comp = 0; comp < 2; ++comp) {
        const u64 t = ip[((size_t)comp * level + (level - 1)) * N];
        const bool high = t > (qL - 1) / 2;
        for (u32 i = 0; i + 1 < level; ++i) {
            const u64 q = R.q[i];
            u64 tq = barrett64(t, q, R.mu[i]);
            if (high) tq = sub_mod(tq, rc.qlmod[i], q);
            const u64 c = ip[((size_t)comp * level + i) * N];
            op[((size_t)comp * (level - 1) + i) * N] = mul_shoup(sub_mod(c, tq, q), rc.inv[i], rc.invs[i], q);
        }
    }
  }
}

// Out-of-place form: one thread per output word (coefficient, ciphertext, component, prime), so the launch is
// wide enough to hide its loads; the dropped prime's residue is read once per output prime (an L2 hit).
// grid: x = coefficients / 256, y = ciphertext, z = component * (level - 1) + prime.
__global__ void __launch_bounds__(256) rescale_wide_kernel(const RingDev R, const RescaleConsts rc, const u64* __restrict__ in,
                                                           u64* __restrict__ out, u32 level) {
    grid_dependency_enter();
    const u32 N = R.N;
    const u32 n = blockIdx.x * blockDim.x + threadIdx.x;
    const u32 ct = blockIdx.y, comp = blockIdx.z / (level - 1), i = blockIdx.z % (level - 1);
    const u64* ip = in + ((size_t)ct * 2 + comp) * level * N + n;
    const u64 qL = R.q[level - 1], q = R.q[i];
    const u64 t = ip[(size_t)(level - 1) * N];
    const u64 c = ip[(size_t)i * N];
    u64 tq = barrett64(t, q, R.mu[i]);
    if (t > (qL - 1) / 2) tq = sub_mod(tq, rc.qlmod[i], q);
    out[(((size_t)ct * 2 + comp) * (level - 1) + i) * N + n] = mul_shoup(sub_mod(c, tq, q), rc.inv[i], rc.invs[i], q);
}

cudaError_t launch_rescale(const RingHost& ring, const u64* in, u64* out, u32 n_ct, u32 level, const u64* inv,
                           const u64* invs, const u64* qlmod, cudaStream_t stream) {
    if (n_ct == 0) return cudaSuccess;
    RescaleConsts rc;
    memset(&rc, 0, sizeof(rc));
    for (u32 i = 0; i + 1 < level; ++i) { rc.inv[i] = inv[i]; rc.invs[i] = invs[i]; rc.qlmod[i] = qlmod[i]; }
    ProfScope prof(ring.prof, CAT_RESCALE, stream);
    if (in == out && n_ct > 1) {
        dim3 grid(ring.dev.N / 64, 1);
        launch_dependent(ring, rescale_kernel, grid, dim3(64), 0, stream, ring.dev, rc, in, out, level, n_ct);
    } else if (in == out || n_ct > 65535) {
        dim3 grid(ring.dev.N / 256, n_ct);
        launch_dependent(ring, rescale_kernel, grid, dim3(256), 0, stream, ring.dev, rc, in, out, level, 1u);
    } else {
        dim3 grid(ring.dev.N / 256, n_ct, 2 * (level - 1));
        launch_dependent(ring, rescale_wide_kernel, grid, dim3(256), 0, stream, ring.dev, rc, in, out, level);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------------------------
// Width changes of the rounded integer coefficients (the coefficient form of cached weights).
__global__ void __launch_bounds__(256) widen_i32_kernel(const int* __restrict__ src, i64* __restrict__ dst, size_t count) {
    grid_dependency_enter();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
        dst[i] = (i64)src[i];
}
__global__ void __launch_bounds__(256) narrow_i64_kernel(const i64* __restrict__ src, int* __restrict__ dst, size_t count,
                                                         int* __restrict__ overflow) {
    grid_dependency_enter();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
        const i64 v = src[i];
        if (v != (i64)(int)v) atomicExch(overflow, 1);
        dst[i] = (int)v;
    }
}
cudaError_t launch_widen_i32(const RingHost& ring, const int* src, i64* dst, size_t count, cudaStream_t stream) {
    if (!count) return cudaSuccess;
    ProfScope prof(ring.prof, CAT_POINTWISE, stream);
    const u32 blocks = (u32)((count + 1023) / 1024 < 148 * 16 ? (count + 1023) / 1024 : 148 * 16);
    return launch_dependent(ring, widen_i32_kernel, dim3(blocks), dim3(256), 0, stream, src, dst, count);
}
cudaError_t launch_narrow_i64(const RingHost& ring, const i64* src, int* dst, size_t count, int* overflow_flag,
                              cudaStream_t stream) {
    if (!count) return cudaSuccess;
    ProfScope prof(ring.prof, CAT_POINTWISE, stream);
    const u32 blocks = (u32)((count + 1023) / 1024 < 148 * 16 ? (count + 1023) / 1024 : 148 * 16);
    return launch_dependent(ring, narrow_i64_kernel, dim3(blocks), dim3(256), 0, stream, src, dst, count, overflow_flag);
}

// ------------------------------------------------------------------------------------------------
// Throughput probe for the 32x32+64-bit integer multiply-add the modular arithmetic is made of:
// every thread runs 8 independent mad.wide.u32 chains.  Gives the measured denominator for the
// integer-bound kernels (NTT, key switch).
__global__ void __launch_bounds__(256) imad_probe_kernel(u64* __restrict__ sink, u32 iters) {
    const u32 b = threadIdx.x * 2654435761u + blockIdx.x * 40503u + 12345u;
    u64 c[8];
    u32 d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { c[k] = b + k; d[k] = b * 3 + k; }
    for (u32 i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
#pragma unroll
            for (int k = 0; k < 8; ++k) asm volatile("mad.wide.u32 %0, %1, %2, %0;" : "+l"(c[k]) : "r"(b), "r"(d[(k + 1) & 7]));
        }
    }
    u64 v = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) v ^= c[k];
    if (v == 0x1234567ull) sink[0] = v;      // practically never true; keeps the chains alive
}

cudaError_t launch_imad_probe(u64* sink, u32 blocks, u32 iters, cudaStream_t stream) {
    imad_probe_kernel<<<blocks, 256, 0, stream>>>(sink, iters);
    return cudaGetLastError();
}

// The same probe for the fp64 fused multiply-add that the transforms of the ciphertext primes are made of:
// every thread runs 8 independent fma.rn.f64 chains.
__global__ void __launch_bounds__(256) fma64_probe_kernel(u64* __restrict__ sink, u32 iters) {
    const double b = 1.0 + (double)(threadIdx.x + blockIdx.x * 256u) * 1e-9;
    double c[8], d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { c[k] = b + k; d[k] = 1e-3 * (k + 1); }
    for (u32 i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
#pragma unroll
            for (int k = 0; k < 8; ++k) asm volatile("fma.rn.f64 %0, %1, %0, %2;" : "+d"(c[k]) : "d"(b), "d"(d[(k + 1) & 7]));
        }
    }
    double v = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) v += c[k];
    if (v == 0.1234567) sink[0] = (u64)__double_as_longlong(v);      // practically never true; keeps the chains alive
}

cudaError_t launch_fma64_probe(u64* sink, u32 blocks, u32 iters, cudaStream_t stream) {
    fma64_probe_kernel<<<blocks, 256, 0, stream>>>(sink, iters);
    return cudaGetLastError();
}

}  // namespace bf
