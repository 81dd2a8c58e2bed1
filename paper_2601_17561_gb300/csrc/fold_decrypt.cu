// Fold (Algorithm 2, linear key-free part) and decryption for checking.
//
// Fold: for eye e and group g of fold_k consecutive rotations, ct'_{e,g} = sum_{r in g} X^r ct_{e,r},
// applied to the a-part polynomial and to every b-block polynomial of the MSRLWE result.  The
// shift is the global rotation index r (Algorithm 2 rotates term rk + r' by rk + r'); X^r is the
// negacyclic monomial shift, (X^r p)[i] = p[i - r] for i >= r and -p[N + i - r] for i < r.  Slot i
// of the shifted result then carries database entry i - r, so that a group never stacks two
// scores of the same database entry (Section 4.3).  The kernel is HBM-bound: every input column
// is read once, one output column is written per group.
//
// Decryption (Section 2.2.2, Dec(a, b) = a * sk + b per b-block): D = C_b + s_{db,t} * C_a modulo
// every q_l, then a fixed-point CRT gives D / Q_db modulo 1, and the numerator is the nearest
// integer to D_centred / (Q' Delta).  After rescaling the same holds modulo Q with scale Delta.
//
// Rescaling by Q' (Section 2.2.2, Maintenance: RS divides by a modulus factor and rounds, here
// the factor Q' = q_Lq ... q_{L-1}, so the scores leave at the query modulus Q with scale Delta):
// per coefficient, yh_i = x_i (Q'/q_i)^-1 mod q_i for the limbs of Q', the correction
// v = floor((sum_i F_i + 2^63) / 2^64) from the 64-bit fixed-point fractions
// F_i = floor(yh_i floor(2^128 / q_i) / 2^64) (integer arithmetic only), the centred
// y = sum_i yh_i (Q'/q_i) - v Q' = x mod Q', and x'_j = (x_j - y mod q_j) Q'^-1 mod q_j for the
// limbs of Q.  HBM-bound: reads L words and writes L_q words per coefficient.
#include "icm_internal.h"

#include <algorithm>

namespace {

using icm::LayoutDev;

// Stored row position of coefficient `coef` of block `blk` (blk = -1: the a-part), or -1 if the
// coefficient is not stored (the gap between the real rows and the tail of a partial block).
__device__ __forceinline__ int64_t pos_of(const LayoutDev &L, int blk, uint32_t coef) {
    if (blk < 0) return coef;
    if ((uint32_t)blk < L.n_full) return (int64_t)L.N + (int64_t)blk * L.N + coef;
    const int64_t base = (int64_t)L.N + (int64_t)L.n_full * L.N;
    if (coef < L.rem) return base + coef;
    if (coef >= L.tail_lo) return base + L.rem + (coef - L.tail_lo);
    return -1;
}

// Block and coefficient of stored row x; tail rows of a partial block report tail = true.
__device__ __forceinline__ void coef_of(const LayoutDev &L, uint64_t x, int &blk, uint32_t &coef, bool &tail) {
    tail = false;
    if (x < L.N) { blk = -1; coef = (uint32_t)x; return; }
    const uint64_t b = x - L.N;
    const uint64_t full = (uint64_t)L.n_full * L.N;
    if (b < full) { blk = (int)(b / L.N); coef = (uint32_t)(b % L.N); return; }
    const uint32_t rel = (uint32_t)(b - full);
    blk = (int)L.n_full;
    if (rel < L.rem) { coef = rel; return; }
    coef = L.tail_lo + (rel - L.rem);
    tail = true;
}

struct FoldArgs {
    LayoutDev lay;
    uint32_t rho, k, groups, n_eyes, L;
    uint64_t q[ICM_MAX_LIMBS], r64[ICM_MAX_LIMBS];
    const uint64_t *in;    // [L][n_eyes*rho][M]
    uint64_t *out;         // [L][n_eyes*groups][M]
};

// grid: (ceil(M / 256), n_eyes * groups, L).  Each thread sums at most fold_k (<= 32) terms,
// adding q - v for the wrapped (negated) ones; fold_k * q < 2^64 keeps the sum exact.
__global__ void __launch_bounds__(256) k_fold(FoldArgs a) {
    const uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t oc = blockIdx.y, l = blockIdx.z;
    if (x >= a.lay.M) return;
    const uint32_t e = oc / a.groups, g = oc % a.groups;
    const uint64_t q = a.q[l];
    uint64_t *dst = a.out + ((size_t)l * a.n_eyes * a.groups + oc) * a.lay.M + x;
    int blk; uint32_t coef; bool tail;
    coef_of(a.lay, x, blk, coef, tail);
    if (tail) { *dst = 0; return; }
    const uint32_t r0 = g * a.k, r1 = min(r0 + a.k, a.rho);
    const uint64_t *col = a.in + ((size_t)l * a.n_eyes * a.rho + (size_t)e * a.rho) * a.lay.M;
    uint64_t acc = 0;
#pragma unroll 4
    for (uint32_t r = r0; r < r1; ++r) {
        const bool wrap = coef < r;
        const uint32_t src = wrap ? a.lay.N + coef - r : coef - r;
        const int64_t p = pos_of(a.lay, blk, src);
        const uint64_t v = (p >= 0) ? col[(size_t)r * a.lay.M + p] : 0;
        acc += wrap ? (v ? q - v : 0) : v;
    }
    *dst = reduce64(acc, q, a.r64[l]);
}

struct DecArgs {
    LayoutDev lay;
    uint32_t L, n_cols, shat_L;
    icm::NttMod nt[ICM_MAX_LIMBS];
    icm::CrtDecode crt;
    const ulonglong2 *shat;  // [blocks][shat_L][N]: transforms of s_{db,t}, times N^-1, with their companions
    const uint64_t *sc;    // [L][n_cols][M]
    int64_t *num;          // [n_cols][n_real]
    uint32_t *err_bits;    // optional: max |x - round(x)| over all outputs, as fp32 bits
    uint32_t h;
    const int32_t *sdb_pos; const int8_t *sdb_sgn;   // [blocks][h]: the supports, for the direct form
};

// F = sum_l y_l floor(2^128 / q_l) mod 2^128: adds y (rhi 2^64 + rlo)
__device__ __forceinline__ void crt_add(const icm::CrtDecode &crt, uint32_t l, uint64_t y, uint64_t &fhi, uint64_t &flo) {
    const uint64_t plo = y * crt.rlo[l];
    const uint64_t phi = __umul64hi(y, crt.rlo[l]) + y * crt.rhi[l];
    const uint64_t nlo = flo + plo;
    fhi = fhi + phi + (nlo < flo ? 1 : 0);
    flo = nlo;
}
// Numerator r of column j from F: F / 2^128 is D / Q_db modulo 1; as a signed 128-bit number it is the
// centred value.
__device__ __forceinline__ void decode(const DecArgs &a, uint32_t j, uint64_t r, uint64_t fhi, uint64_t flo) {
    const double frac = (double)(int64_t)fhi * 0x1p-64 + (double)flo * 0x1p-128;
    const double x = frac * a.crt.q_over_delta;
    const double n = rint(x);
    a.num[(size_t)j * a.lay.n_real + r] = (int64_t)n;
    if (a.err_bits) {
        // distance of the decoded value from the integer it rounds to (numerator units); the
        // bits of non-negative floats order like unsigned integers
        const uint32_t act = __activemask();
        const uint32_t e = __reduce_max_sync(act, __float_as_uint((float)fabs(x - n)));
        if ((threadIdx.x & 31) == (__ffs(act) - 1)) atomicMax(a.err_bits, e);
    }
}

// The direct form, grid (ceil(n_real / 256), n_cols): one thread per (column, real database row), h additions
// per limb from L2.  decrypt_direct says where that is the cheaper one.
__global__ void __launch_bounds__(256) k_decrypt_direct(const __grid_constant__ DecArgs a) {
    const uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t j = blockIdx.y, N = a.lay.N;
    if (r >= a.lay.n_real) return;
    const uint32_t t = (uint32_t)(r / N), i = (uint32_t)(r % N);
    const int64_t pos = pos_of(a.lay, (int)t, i);
    uint64_t fhi = 0, flo = 0;
    for (uint32_t l = 0; l < a.L; ++l) {
        const uint64_t q = a.nt[l].q;
        const uint64_t *col = a.sc + ((size_t)l * a.n_cols + j) * a.lay.M;
        uint64_t d = col[pos];
        for (uint32_t c = 0; c < a.h; ++c) {
            const uint32_t p = (uint32_t)a.sdb_pos[t * a.h + c];
            const int s = a.sdb_sgn[t * a.h + c];
            const uint64_t term = (i >= p) ? col[i - p] : col[N + i - p];
            const bool neg = (i >= p) ? (s < 0) : (s > 0);
            d = neg ? sub_mod(d, term, q) : add_mod(d, term, q);
        }
        crt_add(a.crt, l, mulmod_shoup(d, a.crt.inv[l], a.crt.invs[l], q), fhi, flo);
    }
    decode(a, j, r, fhi, flo);
}

__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint64_t ld_cluster(uint32_t addr, uint32_t rank) {
    uint32_t m;
    uint64_t v;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(m) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(m) : "memory");
    return v;
}

// One cluster of L blocks per column, one block per limb: the transform of the column's a-part stays
// in registers (WPT words per thread, WPT NT >= N; WPT = 0 where one b-block follows, which takes the
// transform where it lies), and per b-block t a pointwise product and one inverse transform give
// s_{db,t} * C_a (ntt.cuh); every block then holds its limb's y in shared memory, and the cluster
// combines the limbs of each coefficient through distributed shared memory, so no limb goes through
// global memory.  Integer products bound it (about 8 per coefficient and limb; the direct form added
// h = 512 terms per coefficient, from L2).  8 eyes x 3,000 codes, 8 limbs, N_db = 2^12: 4.30 ms with
// the direct form, 0.40 ms with one block of 512 threads per SM, 0.20 ms now.
template <int WPT, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) k_decrypt(const __grid_constant__ DecArgs a) {
    extern __shared__ uint64_t su[];
    const uint32_t l = blockIdx.x, j = blockIdx.y, N = a.lay.N;        // block rank in the cluster = limb
    const icm::NttMod &T = a.nt[l];
    const uint64_t q = T.q;
    const uint64_t *col = a.sc + ((size_t)l * a.n_cols + j) * a.lay.M;
    const uint32_t su_addr = (uint32_t)__cvta_generic_to_shared(su);
    for (uint32_t i = threadIdx.x; i < N; i += NT) su[icm::ntt_pad(i)] = col[i];
    __syncthreads();
    icm::ntt_forward(su, 1, 0, N, T);
    uint64_t ah[WPT ? WPT : 1];
#pragma unroll
    for (int w = 0; w < WPT; ++w) {
        const uint32_t i = threadIdx.x + w * NT;
        if (i < N) ah[w] = su[icm::ntt_pad(i)];
    }
    const uint32_t blocks = (uint32_t)((a.lay.n_real + N - 1) / N);
    for (uint32_t t = 0; t < blocks; ++t) {
        const ulonglong2 *sh = a.shat + ((size_t)t * a.shat_L + l) * N;
        if (WPT == 0)
            for (uint32_t i = threadIdx.x; i < N; i += NT) {
                uint64_t *w = su + icm::ntt_pad(i);
                *w = icm::mul_lazy(*w, __ldg(sh + i), 0 - q);
            }
#pragma unroll
        for (int w = 0; w < WPT; ++w) {
            const uint32_t i = threadIdx.x + w * NT;
            if (i < N) su[icm::ntt_pad(i)] = icm::mul_lazy(ah[w], __ldg(sh + i), 0 - q);
        }
        __syncthreads();
        icm::ntt_inverse(su, 1, 0, N, T);
        const uint64_t r0 = (uint64_t)t * N;
        const uint32_t rows = (uint32_t)min((uint64_t)N, a.lay.n_real - r0);
        for (uint32_t i = threadIdx.x; i < rows; i += NT) {
            // (s_{db,t} * C_a)[i], below 4q
            const uint64_t sa = icm::sub_if(icm::sub_if(su[icm::ntt_pad(i)], 2 * q), q);
            const uint64_t d = add_mod(col[pos_of(a.lay, (int)t, i)], sa, q);
            su[icm::ntt_pad(i)] = mulmod_shoup(d, a.crt.inv[l], a.crt.invs[l], q);
        }
        __syncwarp();
        cluster_barrier();
        for (uint32_t i = l * NT + threadIdx.x; i < rows; i += a.L * NT) {
            uint64_t fhi = 0, flo = 0;
            for (uint32_t k = 0; k < a.L; ++k) crt_add(a.crt, k, ld_cluster(su_addr + icm::ntt_pad(i) * 8, k), fhi, flo);
            decode(a, j, r0 + i, fhi, flo);
        }
        __syncwarp();
        cluster_barrier();                              // the limbs are read before the next block's product
    }
}

struct RsArgs {
    icm::RescaleConsts k;
    const uint64_t *in;    // [L][n]
    uint64_t *out;         // [Lq][n]
    uint64_t n;
};

// Rescale one coefficient c of [L][n] into [Lq][n].
__device__ __forceinline__ void rescale_one(const icm::RescaleConsts &k, const uint64_t *in, uint64_t *out, uint64_t n,
                                            uint64_t c) {
    const uint32_t L = k.L, Lq = k.Lq;
    uint64_t yh[ICM_MAX_LIMBS];
    uint64_t slo = 0, shi = 0;                                     // sum of the F_i, 128-bit
#pragma unroll
    for (uint32_t i = 0; i < ICM_MAX_LIMBS; ++i) {
        if (i < Lq || i >= L) continue;
        const uint64_t q = k.q[i];
        yh[i] = mulmod_shoup(in[(size_t)i * n + c], k.yinv[i], k.yinvs[i], q);
        // F_i = yh rhi + floor(yh rlo / 2^64): exact, and < 2^64 because yh < q_i
        const uint64_t f = yh[i] * k.rhi[i] + __umul64hi(yh[i], k.rlo[i]);
        slo += f;
        shi += slo < f ? 1 : 0;
    }
    const uint64_t v = shi + ((slo >> 63) & 1);                    // floor((S + 2^63) / 2^64)
    // x'_j = (x_j - y) Q'^-1 = x_j Q'^-1 + sum_i yh_i w_ji + v mod q_j: one 128-bit sum of products below
    // 2^123 and one reduction (a Shoup product with its reduction for each term took three 64-bit
    // products where the sum takes one)
    for (uint32_t j = 0; j < Lq; ++j) {
        const uint64_t q = k.q[j], x = in[(size_t)j * n + c];
        uint64_t lo = x * k.qpinv[j], hi = __umul64hi(x, k.qpinv[j]);
        lo += v;
        hi += lo < v ? 1 : 0;
#pragma unroll
        for (uint32_t i = 0; i < ICM_MAX_LIMBS; ++i)
            if (i >= Lq && i < L) {
                const uint64_t p = yh[i] * k.w[j][i];
                lo += p;
                hi += __umul64hi(yh[i], k.w[j][i]) + (lo < p ? 1 : 0);
            }
        // the quotient estimate is short by at most 4, so the remainder is below 5 q < 2^63
        const uint64_t qe = hi * k.rhi[j] + __umul64hi(hi, k.rlo[j]) + __umul64hi(lo, k.rhi[j]);
        uint64_t r = lo - qe * q;
        r = r >= 2 * q ? r - 2 * q : r;
        r = r >= 2 * q ? r - 2 * q : r;
        out[(size_t)j * n + c] = r >= q ? r - q : r;
    }
}

// Two coefficients per thread, one after the other (36 registers hold one's words); consecutive threads read
// consecutive words of a limb.  Bound by the waits on those loads (8 of the 18 cycles between two
// instructions of a warp, 67% of the warps resident), with the FMA-heavy pipe 49% and DRAM 27% busy; so the
// fewer products above gave 0.303 -> 0.277 ms for the rescaling and fold of 32 eyes x 3,000 codes on 8
// limbs, and nothing at 1.3e8 coefficients (5.0 to 5.2 ms, 0.30 of the copy bandwidth).
__global__ void __launch_bounds__(256) k_rescale(const __grid_constant__ RsArgs a) {
    const uint64_t c0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x);
    const uint64_t half = (a.n + 1) / 2;
    if (c0 >= half) return;
    rescale_one(a.k, a.in, a.out, a.n, c0);
    if (c0 + half < a.n) rescale_one(a.k, a.in, a.out, a.n, c0 + half);
}

}  // namespace

namespace icm {

cudaError_t launch_rescale(const icm_ctx *c, const uint64_t *d_in, uint64_t n, uint64_t *d_out, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    RsArgs a{c->rs, d_in, d_out, n};
    const uint64_t threads = (n + 1) / 2;
    k_rescale<<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(a);
    return cudaGetLastError();
}


cudaError_t launch_fold(const icm_ctx *c, const LayoutDev &lay, const uint64_t *d_in, uint32_t n_eyes, uint32_t limbs,
                        uint64_t *d_out, cudaStream_t st) {
    FoldArgs a{};
    a.lay = lay; a.rho = c->p.rho; a.k = c->p.fold_k;
    a.groups = (c->p.rho + c->p.fold_k - 1) / c->p.fold_k;
    a.n_eyes = n_eyes; a.L = limbs;                 // the first `limbs` primes (Q's come first)
    for (uint32_t l = 0; l < a.L; ++l) { a.q[l] = c->q[l]; a.r64[l] = c->lt.r64[l]; }
    a.in = d_in; a.out = d_out;
    if (n_eyes == 0 || lay.M == 0) return cudaSuccess;
    dim3 grid((unsigned)((lay.M + 255) / 256), n_eyes * a.groups, a.L);
    k_fold<<<grid, 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t decrypt_set_attributes() {
    return allow_smem(k_decrypt<0, 256, 4>, k_decrypt<0, 512, 2>, k_decrypt<0, 1024, 1>, k_decrypt<16, 256, 3>,
                      k_decrypt<32, 256, 2>, k_decrypt<16, 1024, 1>);
}

// Whether h additions per row and limb take less time than the transforms.  Both sides in us, fitted to
// measurements at L = 4 (2 to 248 columns, 10 to 3,000 rows, N = 2^5 to 2^14, h = 16 to 512): the additions run
// at 1.4 ps each, but no faster than a row's chain of them; the transforms by columns and limbs, but no faster
// than a block of a cluster.  248 columns, us, additions / transforms: N = 2^14, h = 64, 1,000 rows 142 / 443;
// 2^13, 100 rows 69 / 202; 2^12 65 / 100, 3,000 rows 299 / 116; 2^7, 3,000 rows, h = 16 93 / 396; h = 512, 3,000
// rows 2^12 2,157 / 115, 100 rows 2^14 660 / 423.
static bool decrypt_direct(uint32_t h, uint32_t N, uint32_t L, uint64_t rows, uint32_t n_cols) {
    const double n = N, w = (double)n_cols * L, blocks = (double)((rows + N - 1) / N);
    const double direct = (double)h * L * std::max(1.4e-6 * (double)rows * n_cols, 0.1 + 5e-6 * n);
    const double transforms = blocks <= 1 ? n * std::max(2.2e-5 * w, 2.9e-3)
                                          : (blocks + 1) * std::max(w * (0.0135 + 7e-6 * n), 3.6 + 7e-4 * n);
    return direct < transforms;
}

cudaError_t launch_decrypt(const icm_ctx *c, const LayoutDev &lay, const uint64_t *d_scores, uint32_t n_cols,
                           bool rescaled, int64_t *d_num, cudaStream_t st, uint32_t *d_err_bits) {
    DecArgs a{};
    a.lay = lay; a.L = rescaled ? c->p.n_limbs_q : c->p.n_limbs; a.n_cols = n_cols;
    a.shat_L = c->p.n_limbs;
    for (uint32_t l = 0; l < a.L; ++l) a.nt[l] = c->nt.db[l];
    a.crt = rescaled ? c->crt_q : c->crt;
    a.shat = c->nt.shat_db;
    a.sc = d_scores; a.num = d_num; a.err_bits = d_err_bits;
    if (n_cols == 0 || lay.n_real == 0) return cudaSuccess;
    if (!a.shat) return cudaErrorInvalidValue;                           // rings above 2^14
    if (decrypt_direct(c->p.hamming_weight, lay.N, a.L, lay.n_real, n_cols)) {
        a.h = c->p.hamming_weight; a.sdb_pos = c->d_sdb_pos; a.sdb_sgn = c->d_sdb_sgn;
        k_decrypt_direct<<<dim3((unsigned)((lay.n_real + 255) / 256), n_cols), 256, 0, st>>>(a);
        return cudaGetLastError();
    }
    const size_t smem = (size_t)ntt_words(lay.N) * 8;
    auto run = [&](auto kern, int nt) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        cfg.gridDim = dim3(a.L, n_cols); cfg.blockDim = dim3(nt);
        cfg.dynamicSmemBytes = smem; cfg.stream = st;
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = a.L; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, a);
    };
    // Blocks per SM hide the waits at the cluster's barriers.  One b-block: nothing is kept in registers,
    // and 64 registers a thread allow 1,024 threads per SM, in blocks as small as shared memory lets that
    // many be resident (248 columns, four limbs: N = 2^12 131 / 143 / 168 us with blocks of 256 / 512 /
    // 1,024, 2^13 282 / 268 / 317, 2^14 869 / 642 / 573).  Several b-blocks: the transformed a-part takes
    // N / NT words of registers (2^12 236 us with 256 threads, 311 with 512; 2^13 523 and 594; 2^14 857
    // with 1,024 threads, 955 with 512).
    if (lay.n_real <= lay.N)
        return lay.N <= 4096 ? run(k_decrypt<0, 256, 4>, 256)
                             : lay.N <= 8192 ? run(k_decrypt<0, 512, 2>, 512) : run(k_decrypt<0, 1024, 1>, 1024);
    return lay.N <= 4096 ? run(k_decrypt<16, 256, 3>, 256)
                         : lay.N <= 8192 ? run(k_decrypt<32, 256, 2>, 256) : run(k_decrypt<16, 1024, 1>, 1024);
}

}  // namespace icm
