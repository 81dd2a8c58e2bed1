// Negacyclic number-theoretic transforms in shared memory (device functions), shared by the
// encryption, decryption and normalisation kernels.
//
// Forward: Cooley-Tukey butterflies with the powers of a primitive 2N-th root psi in bit-reversed
// order, output in bit-reversed order; inverse: Gentleman-Sande with the inverse powers (Longa
// and Naehrig, CANS 2016).  Butterflies keep their values lazily reduced (after Harvey, J. Symb. Comp.
// 2014) within the 16 q that 64 bits hold for q < 2^60: a product by a twiddle is below 4q, forward
// values stay below 16q with a conditional subtraction of 8q at every other level, inverse sums grow
// for two levels before they are reduced.  (Four conditional subtractions per three levels instead of
// twelve, and a high product of three partial ones: encryption of 1,000 templates 12.1 -> 11.6 ms.)
//
// What bounds them: integer multiplication (a Shoup product is two 64-bit low products and one
// high one), once the traffic per level is out of the way.  So a thread takes 8 elements through
// three levels in registers between two passes over shared memory (a radix-2 pass per level read
// and wrote shared memory and met a barrier 12 to 14 times instead of 4 or 5), and the twiddles
// sit next to their Shoup companions so that one 16-byte load fetches both.  Words are stored at
// ntt_pad(i) = i + i / 8: the last passes take 8 neighbouring words per thread, which unpadded
// would hit two of the sixteen 8-byte banks.  (An exclusive-or layout without any conflict measured
// 2 to 4% slower: its addresses cost more than the conflicts.)
#pragma once
#include "icm_device.cuh"

namespace icm {

__host__ __device__ __forceinline__ uint32_t ntt_pad(uint32_t i) { return i + (i >> 3); }
// shared-memory words of one polynomial of degree N
__host__ __device__ constexpr uint32_t ntt_words(uint32_t N) { return N + N / 8; }

// Twiddles of one modulus: [2][N] (w, floor(w 2^64 / q)), forward then inverse, bit-reversed order.
struct NttMod {
    const ulonglong2 *fwd, *inv;
    uint64_t q, ninv, ninvs;          // N^-1 mod q and its Shoup companion
    uint64_t rhi, rlo;                // floor(2^128 / q)
};

// a w mod q in [0, 4q) for any a < 2^64 and w < q with its Shoup companion: the high product without
// its lowest partial product is short by at most 2, and nq = 2^64 - q lets both low products accumulate.
__device__ __forceinline__ uint64_t mul_lazy(uint64_t a, ulonglong2 w, uint64_t nq) {
    const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)w.y, bh = (uint32_t)(w.y >> 32);
    const uint64_t h = (uint64_t)ah * bh + (((uint64_t)ah * bl) >> 32) + (((uint64_t)al * bh) >> 32);
    return a * w.x + h * nq;
}
__device__ __forceinline__ uint64_t sub_if(uint64_t x, uint64_t m) { return min(x, x - m); }   // x < m ? x : x - m
// forward butterfly: x < 16q (SUB) or 12q -> x + w y, x - w y, both below 12q (SUB) or 16q
template <bool SUB>
__device__ __forceinline__ void bf_fwd(uint64_t &x, uint64_t &y, ulonglong2 w, uint64_t q4, uint64_t nq) {
    const uint64_t u = SUB ? sub_if(x, 2 * q4) : x, v = mul_lazy(y, w, nq);
    x = u + v;
    y = u - v + q4;
}

// R levels (R = 1, 2, 3) starting at level m of the forward transform, on C polynomials of stride
// `stride` words: m blocks of N / m elements, a thread takes 2^R elements N / (m 2^R) apart.
template <int R>
__device__ __forceinline__ void ntt_fwd_pass(uint64_t *a, uint32_t C, uint32_t stride, uint32_t N, uint32_t m,
                                             const ulonglong2 *tw, uint64_t q) {
    constexpr uint32_t E = 1u << R;
    const uint32_t t = N / (m * E), lt = 31 - __clz(t), groups = N / E;
    const uint64_t q4 = 4 * q, nq = 0 - q;
    for (uint32_t x = threadIdx.x; x < groups; x += blockDim.x) {
        const uint32_t i = x >> lt, base = (i << (lt + R)) + (x & (t - 1));
        ulonglong2 w[E - 1];
#pragma unroll
        for (uint32_t r = 0; r < R; ++r)
#pragma unroll
            for (uint32_t b = 0; b < (1u << r); ++b) w[(1u << r) - 1 + b] = __ldg(tw + (m << r) + (i << r) + b);
        for (uint32_t c = 0; c < C; ++c) {
            uint64_t *p = a + c * stride;
            uint64_t v[E];
#pragma unroll
            for (uint32_t k = 0; k < E; ++k) v[k] = p[ntt_pad(base + k * t)];
#pragma unroll
            for (uint32_t r = 0; r < R; ++r) {
                const uint32_t h = E >> (r + 1);
#pragma unroll
                for (uint32_t k = 0; k < E; ++k)
                    if (!(k & h)) {
                        const ulonglong2 ww = w[(1u << r) - 1 + (k >> (R - r))];
                        if (r & 1) bf_fwd<false>(v[k], v[k + h], ww, q4, nq);
                        else bf_fwd<true>(v[k], v[k + h], ww, q4, nq);
                    }
            }
#pragma unroll
            for (uint32_t k = 0; k < E; ++k) p[ntt_pad(base + k * t)] = v[k];
        }
    }
    __syncthreads();
}

// R levels of the inverse transform ending at m blocks (m 2^R blocks before, each level halving).
template <int R>
__device__ __forceinline__ void ntt_inv_pass(uint64_t *a, uint32_t C, uint32_t stride, uint32_t N, uint32_t m,
                                             const ulonglong2 *tw, uint64_t q) {
    constexpr uint32_t E = 1u << R;
    const uint32_t t = N / (m * E), lt = 31 - __clz(t), groups = N / E;
    const uint64_t q4 = 4 * q, nq = 0 - q;
    for (uint32_t x = threadIdx.x; x < groups; x += blockDim.x) {
        const uint32_t i = x >> lt, base = (i << (lt + R)) + (x & (t - 1));
        ulonglong2 w[E - 1];
#pragma unroll
        for (uint32_t r = 0; r < R; ++r)
#pragma unroll
            for (uint32_t b = 0; b < (1u << r); ++b) w[(1u << r) - 1 + b] = __ldg(tw + (m << r) + (i << r) + b);
        for (uint32_t c = 0; c < C; ++c) {
            uint64_t *p = a + c * stride;
            uint64_t v[E];
#pragma unroll
            for (uint32_t k = 0; k < E; ++k) v[k] = p[ntt_pad(base + k * t)];
            // bnd[k]: v[k] is below 4 bnd[k] q (known when the loops are unrolled); sums may reach 16q
            uint32_t bnd[E];
#pragma unroll
            for (uint32_t k = 0; k < E; ++k) bnd[k] = 1;
#pragma unroll
            for (int r = R - 1; r >= 0; --r) {
                const uint32_t h = E >> (r + 1);
#pragma unroll
                for (uint32_t k = 0; k < E; ++k)
                    if (!(k & h)) {
                        if (bnd[k] + bnd[k + h] > 4) {
                            v[k] = sub_if(v[k], 2 * q4); bnd[k] = 2;
                            v[k + h] = sub_if(v[k + h], 2 * q4); bnd[k + h] = 2;
                        }
                        const uint64_t sum = v[k] + v[k + h], d = v[k] - v[k + h] + bnd[k + h] * q4;
                        v[k] = sum;
                        bnd[k] += bnd[k + h];
                        v[k + h] = mul_lazy(d, w[(1u << r) - 1 + (k >> (R - r))], nq);
                        bnd[k + h] = 1;
                    }
            }
#pragma unroll
            for (uint32_t k = 0; k < E; ++k) {
                if (bnd[k] > 2) v[k] = sub_if(v[k], 2 * q4);
                if (bnd[k] > 1) v[k] = sub_if(v[k], q4);
            }
#pragma unroll
            for (uint32_t k = 0; k < E; ++k) p[ntt_pad(base + k * t)] = v[k];
        }
    }
    __syncthreads();
}

// Forward transform of C polynomials (words at ntt_pad(i), values below 16q in and out).  The caller
// meets a barrier before; ends with one.
__device__ __forceinline__ void ntt_forward(uint64_t *a, uint32_t C, uint32_t stride, uint32_t N, const NttMod &T) {
    uint32_t m = 1;
    for (; m * 8 <= N; m *= 8) ntt_fwd_pass<3>(a, C, stride, N, m, T.fwd, T.q);
    if (m * 4 == N) ntt_fwd_pass<2>(a, C, stride, N, m, T.fwd, T.q);
    else if (m * 2 == N) ntt_fwd_pass<1>(a, C, stride, N, m, T.fwd, T.q);
}
// Inverse transform without the factor N^-1 (values below 4q in and out).
__device__ __forceinline__ void ntt_inverse(uint64_t *a, uint32_t C, uint32_t stride, uint32_t N, const NttMod &T) {
    uint32_t m = N;
    for (; m >= 8; m /= 8) ntt_inv_pass<3>(a, C, stride, N, m / 8, T.inv, T.q);
    if (m == 4) ntt_inv_pass<2>(a, C, stride, N, 1, T.inv, T.q);
    else if (m == 2) ntt_inv_pass<1>(a, C, stride, N, 1, T.inv, T.q);
}

// x < 16q -> [0, q)
__device__ __forceinline__ uint64_t ntt_canon(uint64_t x, uint64_t q) {
    return sub_if(sub_if(sub_if(sub_if(x, 8 * q), 4 * q), 2 * q), q);
}

// a b mod q in [0, 2q) for a < 16q, b < q, with R = floor(2^128 / q) = rhi 2^64 + rlo: the quotient
// estimate from the high words of x R / 2^128 is short by at most 4 (below 5q < 2^63 remains).
__device__ __forceinline__ uint64_t mul_r128_lazy(uint64_t a, uint64_t b, const NttMod &T) {
    const uint64_t lo = a * b, hi = __umul64hi(a, b);
    const uint64_t qe = hi * T.rhi + __umul64hi(hi, T.rlo) + __umul64hi(lo, T.rhi);
    uint64_t r = lo - qe * T.q;
    const uint64_t q2 = 2 * T.q;
    r = r >= q2 ? r - q2 : r;
    return r >= q2 ? r - q2 : r;
}

}  // namespace icm
