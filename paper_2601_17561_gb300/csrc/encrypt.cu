// Encryption kernels of libicm (setup path, not timed in the matching step).
//
// Database chunk, MSRLWE-RGSW form (Section 6.2.1: a pair of encryptions of M_db and of
// M_db * S_q under the database secrets, modulus Q_db = Q * Q'):
//   a-part row i, column k:   A[i][k] uniform modulo Q_db (an independent residue per limb)
//   b-row r = t * N_db + i:   B[r][k] = -(s_{db,t} * A[:, k])[i] + Q' * W[r][k] + E[r][k]
//   W[r][k] = c'_r[k] for k < d2 (the masked bit-vector of template r, Section 2.1.3) and
//   W[r][d2 + j] = (M_db S_q)[r][j] for j < N_q (S_q: vertical stack of the negacyclic matrices
//   of the query secrets).  The gadget factor Q' makes Q' * Q = 0 modulo Q_db, which removes
//   the query's wrap-around multiple of Q from the decrypted product.
// Stored rows are written in the balanced-digit form of icm_device.cuh (to_digit_form).
// Query eyes, MSRLWE form modulo Q (Section 2.3):
//   b_{t,j} = -(s_{q,t} * a_j) + Delta * c'_j[t N_q .. (t+1) N_q) + e_{t,j},  a_j uniform mod Q,
//   where column j = eye * rho + r holds rotation r of the eye (Section 2.1.2).
#include "icm_internal.h"

#include <algorithm>
#include <string>

namespace {

using icm::LayoutDev;

// Map a b-region index (0-based, after the a-part rows) to its logical row (t, i).
__device__ __forceinline__ void b_row_of(const LayoutDev &L, uint64_t bidx, uint32_t &t, uint32_t &i) {
    const uint64_t full = (uint64_t)L.n_full * L.N;
    if (bidx < full) {
        t = (uint32_t)(bidx / L.N);
        i = (uint32_t)(bidx % L.N);
    } else {
        const uint32_t rel = (uint32_t)(bidx - full);
        t = L.n_full;
        i = rel < L.rem ? rel : L.tail_lo + (rel - L.rem);
    }
}

__device__ __forceinline__ int template_bit(const uint8_t *tpl, uint32_t b) { return (tpl[b >> 3] >> (b & 7)) & 1; }

struct DbMsgArgs {
    LayoutDev lay;
    uint32_t K, d2, Nq, nqblk, h, code_bits, Lq;
    const uint8_t *codes, *masks;      // [n_real][code_bits/8]
    const int32_t *wmsg;               // message rows [n_real][d2] (slot encoding), or null: c' of codes
    const int32_t *sq_pos; const int8_t *sq_sgn;   // [nqblk][h]
    uint64_t qp[ICM_MAX_LIMBS], qps[ICM_MAX_LIMBS], q[ICM_MAX_LIMBS];
    uint64_t *db;                      // [L][M][K]
};

// Pass 1: the message residues Q' * W[r][k] of every stored b-row, for the limbs of Q (they are zero
// modulo the limbs of Q', which pass 2 does not read).  The message
// row is the masked bit-vector c' of template r (coefficient encoding, BITS) or, for a slot-encoded
// chunk, the given row of rounded slot-encoding coefficients.
//
// (M_db S_q)[r][j] = sum over the query secrets' non-zeros (position p, sign s) of s e[j + p], e = c'
// followed by -c' (the negacyclic wrap): h d2 / N_q additions per entry.  With c' in {-1, 0, 1} four
// entries are added at once as bytes 1 + s c' of a word: the row is kept as 1 + c', 1 - c', 1 + c' (a
// negative sign starts N_q later), unaligned words come from two aligned ones by a funnel shift, and the
// bytes are widened every 127 terms.  Shared-memory reads bound it (two words per four additions):
// 1,030 rows, N_q = 2^13: 0.6 ms, 3.8 ms with one addition at a time.
template <bool BITS>
__global__ void __launch_bounds__(512) k_db_messages(const __grid_constant__ DbMsgArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    // BITS: [nqblk][3 N_q + 4] bytes, else [d2] words; then the supports (BITS: start offsets)
    const uint32_t stride = 3 * a.Nq + 4;
    int32_t *cp = reinterpret_cast<int32_t *>(smem);
    int32_t *spos = reinterpret_cast<int32_t *>(smem + (BITS ? (size_t)a.nqblk * stride : (size_t)((a.d2 + 3) & ~3u) * 4));
    int8_t *ssgn = reinterpret_cast<int8_t *>(spos + a.nqblk * a.h);

    const uint64_t bidx = blockIdx.x;
    const uint64_t pos = a.lay.N + bidx;
    uint32_t t, i;
    b_row_of(a.lay, bidx, t, i);
    const uint64_t r = (uint64_t)t * a.lay.N + i;
    const bool real = r < a.lay.n_real;
    const uint32_t tb = a.code_bits / 8;
    auto put = [&](uint32_t k, int32_t W) {
        for (uint32_t l = 0; l < a.Lq; ++l) {
            uint64_t v = 0;
            if (W != 0) {
                const uint64_t m = mulmod_shoup((uint64_t)(W < 0 ? -W : W), a.qp[l], a.qps[l], a.q[l]);
                v = (W < 0 && m) ? a.q[l] - m : m;
            }
            a.db[((size_t)l * a.lay.M + pos) * a.K + k] = v;
        }
    };
    for (uint32_t k = threadIdx.x; k < a.d2; k += blockDim.x) {
        int v = 0;
        if (real && !BITS && a.wmsg) {
            v = a.wmsg[r * a.d2 + k];
        } else if (real && k < a.code_bits) {
            const int c = template_bit(a.codes + r * tb, k), m = template_bit(a.masks + r * tb, k);
            v = m - 2 * (c & m);
        }
        if (!BITS) {
            cp[k] = v;
        } else {
            unsigned char *e = smem + (size_t)(k / a.Nq) * stride + k % a.Nq;
            e[0] = (unsigned char)(1 + v);
            e[a.Nq] = (unsigned char)(1 - v);
            e[2 * a.Nq] = (unsigned char)(1 + v);
        }
        put(k, v);
    }
    for (uint32_t x = threadIdx.x; x < a.nqblk * a.h; x += blockDim.x) {
        const int8_t g = a.sq_sgn[x];
        spos[x] = a.sq_pos[x] + (BITS && g < 0 ? (int32_t)a.Nq : 0);
        if (!BITS) ssgn[x] = g;
    }
    if (BITS)
        for (uint32_t x = threadIdx.x; x < a.nqblk * 4; x += blockDim.x) smem[(size_t)(x >> 2) * stride + 3 * a.Nq + (x & 3)] = 0;
    __syncthreads();
    if (!real) {
        for (uint32_t k = a.d2 + threadIdx.x; k < a.K; k += blockDim.x) put(k, 0);
        return;
    }
    if (BITS) {
        const uint32_t nw = a.Nq / 4, terms = a.nqblk * a.h;
        constexpr int V = 4;                                             // words (of four entries) per thread
        for (uint32_t w0 = threadIdx.x; w0 < nw; w0 += blockDim.x * V) {
            uint32_t lo[V] = {}, hi[V] = {};                             // 16-bit sums of the even and odd entries
            for (uint32_t tt = 0; tt < a.nqblk; ++tt) {
                const uint32_t *e = reinterpret_cast<const uint32_t *>(smem + (size_t)tt * stride);
                for (uint32_t c0 = 0; c0 < a.h; c0 += 127) {
                    const uint32_t c1 = min(c0 + 127, a.h);
                    uint32_t acc[V] = {};
                    for (uint32_t c = c0; c < c1; ++c) {
                        const uint32_t o = (uint32_t)spos[tt * a.h + c], sh = 8 * (o & 3);
                        const uint32_t *p = e + w0 + (o >> 2);
#pragma unroll
                        for (int x = 0; x < V; ++x)
                            if (w0 + x * blockDim.x < nw)
                                acc[x] += __funnelshift_r(p[x * blockDim.x], p[x * blockDim.x + 1], sh);
                    }
#pragma unroll
                    for (int x = 0; x < V; ++x) { lo[x] += acc[x] & 0x00FF00FFu; hi[x] += (acc[x] >> 8) & 0x00FF00FFu; }
                }
            }
#pragma unroll
            for (int x = 0; x < V; ++x) {
                const uint32_t j = 4 * (w0 + x * blockDim.x);
                if (j >= a.Nq) continue;
                put(a.d2 + j, (int32_t)(lo[x] & 0xFFFF) - (int32_t)terms);
                put(a.d2 + j + 1, (int32_t)(hi[x] & 0xFFFF) - (int32_t)terms);
                put(a.d2 + j + 2, (int32_t)(lo[x] >> 16) - (int32_t)terms);
                put(a.d2 + j + 3, (int32_t)(hi[x] >> 16) - (int32_t)terms);
            }
        }
    } else for (uint32_t j = threadIdx.x; j < a.Nq; j += blockDim.x) {
        // only k' = (j + p) mod Nq with s_{q,t}[p] != 0 contribute, with sign -1 when j + p wraps past Nq
        int32_t W = 0;
        for (uint32_t tt = 0; tt < a.nqblk; ++tt) {
            const int32_t *crow = cp + tt * a.Nq;
            for (uint32_t c = 0; c < a.h; ++c) {
                const uint32_t p = (uint32_t)spos[tt * a.h + c];
                const int s = ssgn[tt * a.h + c];
                const uint32_t jp = j + p;
                W += (jp < a.Nq) ? s * crow[jp] : -s * crow[jp - a.Nq];
            }
        }
        put(a.d2 + j, W);
    }
}

struct DbEncArgs {
    LayoutDev lay;
    uint32_t K, eta, n_blocks, Lq, logc;             // 2^logc columns per block
    uint64_t seed, chunk;
    icm::NttMod nt[ICM_MAX_LIMBS];
    const ulonglong2 *shat;                          // [blocks][L][N]: transforms of s_{db,t}, times N^-1
    uint32_t h;
    const int32_t *sdb_pos; const int8_t *sdb_sgn;   // [blocks][h]: the supports, for the direct form
    LimbTable lt;
    uint64_t *db;
};

// Threads of the kernels that multiply by a secret: 128 registers each, of which a thread keeps
// up to 32 words of a transformed polynomial.
constexpr int NT_MUL = 512;

// Pass 2, one block per (2^logc columns k, limb l): draw the a-part columns into shared memory and
// write them, then finish every b-row: B = msg - (s_{db,t} * a)[i] + e (mod q_l).
//
// The products by the secrets are negacyclic transforms (ntt.cuh): one forward transform of a, which
// stays in registers, and per block t a pointwise product and one inverse transform.  Integer
// arithmetic bounds both this and the direct form (h = 512 modular additions per coefficient),
// but a transform costs about 7 Shoup products per coefficient.  Columns are taken four at a time
// where 2^14 words hold them, so that a row's words fill a 32-byte sector and the columns share
// their twiddles.  1,000 templates at N_db = 2^12, four primes (4.0 GB): 69.5 ms with the
// additions, 10.95 ms now (10.3 of them here: 6.6 the transforms, 1.6 the pointwise products (2.3
// without the secrets' companions), 1 the noise and the rows' update, 0.8 drawing and storing the
// a-part).  Twice the threads (64 registers, the polynomial kept in shared memory or not at all) or
// two blocks of half the columns give the same time, one column per block takes 13.2 ms:
// multiplications bound it, not latency.
template <int WPT>
__global__ void __launch_bounds__(NT_MUL, 1) k_db_apart_b(const __grid_constant__ DbEncArgs a) {
    extern __shared__ uint64_t su[];                                     // [2^logc][stride]
    const uint32_t C = 1u << a.logc, l = blockIdx.y, N = a.lay.N, k0 = blockIdx.x << a.logc;
    const uint32_t stride = icm::ntt_words(N) + 4, CN = N << a.logc;
    const uint64_t q = a.lt.q[l];
    const icm::NttMod &T = a.nt[l];
    const uint64_t ka = stream_key(a.seed, ICM_KIND_A_DB, a.chunk, l);
    const uint64_t ke = stream_key(a.seed, ICM_KIND_E_DB, a.chunk, 0);
    uint64_t *dbl = a.db + (size_t)l * a.lay.M * a.K;
    // word x: column x mod C of coefficient x / C
    for (uint32_t x = threadIdx.x; x < CN; x += NT_MUL) {
        const uint32_t c = x & (C - 1), i = x >> a.logc, k = k0 + c;
        uint64_t v = 0;
        if (k < a.K) {
            v = uniform_mod(sm64(ka, (uint64_t)i * a.K + k), q);
            dbl[(size_t)i * a.K + k] = to_digit_form(v, q);
        }
        su[c * stride + icm::ntt_pad(i)] = v;
    }
    if (a.n_blocks == 0) return;
    __syncthreads();
    icm::ntt_forward(su, C, stride, N, T);
    uint64_t ah[WPT];
#pragma unroll
    for (int j = 0; j < WPT; ++j) {
        const uint32_t x = threadIdx.x + j * NT_MUL;
        if (x < CN) ah[j] = su[(x & (C - 1)) * stride + icm::ntt_pad(x >> a.logc)];
    }
    for (uint32_t t = 0; t < a.n_blocks; ++t) {
        // a thread overwrites only the words that it read itself
        const ulonglong2 *sh = a.shat + ((size_t)t * a.lt.n + l) * N;
#pragma unroll
        for (int j = 0; j < WPT; ++j) {
            const uint32_t x = threadIdx.x + j * NT_MUL;
            if (x < CN)
                su[(x & (C - 1)) * stride + icm::ntt_pad(x >> a.logc)] = icm::mul_lazy(ah[j], __ldg(sh + (x >> a.logc)), 0 - q);
        }
        __syncthreads();
        icm::ntt_inverse(su, C, stride, N, T);
        const bool part = t >= a.lay.n_full;                             // the partial last block
        for (uint32_t x = threadIdx.x; x < CN; x += NT_MUL) {
            const uint32_t c = x & (C - 1), i = x >> a.logc, k = k0 + c;
            if (k >= a.K || (part && i >= a.lay.rem && i < a.lay.tail_lo)) continue;
            const uint64_t row = (uint64_t)N + (uint64_t)t * N + (part && i >= a.lay.rem ? a.lay.rem + (i - a.lay.tail_lo) : i);
            const uint64_t r = (uint64_t)t * N + i;
            // (s_{db,t} * a)[i], below 4q
            const uint64_t sa = icm::sub_if(icm::sub_if(su[c * stride + icm::ntt_pad(i)], 2 * q), q);
            uint64_t *dst = dbl + (size_t)row * a.K + k;
            const int e = cbd_sample(sm64(ke, r * a.K + k), a.eta);
            // messages are multiples of Q', zero modulo the limbs of Q'
            uint64_t v = sub_mod(l < a.Lq ? *dst : 0, sa, q);
            v = e >= 0 ? add_mod(v, (uint64_t)e, q) : sub_mod(v, (uint64_t)(-e), q);
            *dst = to_digit_form(v, q);
        }
    }
}

// Pass 2 in the direct form, one block per (column k, limb l): h additions per stored b-row.  A chunk of few
// templates stores few rows of its ring (and small rings leave most of a transform's threads idle):
// db_direct says where that is the cheaper one.
__global__ void __launch_bounds__(1024) k_db_apart_b_direct(const __grid_constant__ DbEncArgs a) {
    extern __shared__ uint64_t su[];
    uint64_t *acol = su;                                                 // [N]
    int32_t *spos = reinterpret_cast<int32_t *>(acol + a.lay.N);         // [n_blocks * h]
    int8_t *ssgn = reinterpret_cast<int8_t *>(spos + a.n_blocks * a.h);
    const uint32_t k = blockIdx.x, l = blockIdx.y, N = a.lay.N;
    const uint64_t q = a.lt.q[l];
    const uint64_t ka = stream_key(a.seed, ICM_KIND_A_DB, a.chunk, l);
    const uint64_t ke = stream_key(a.seed, ICM_KIND_E_DB, a.chunk, 0);
    uint64_t *dbl = a.db + (size_t)l * a.lay.M * a.K;
    for (uint32_t i = threadIdx.x; i < N; i += blockDim.x) {
        const uint64_t v = uniform_mod(sm64(ka, (uint64_t)i * a.K + k), q);
        acol[i] = v;
        dbl[(size_t)i * a.K + k] = to_digit_form(v, q);
    }
    for (uint32_t x = threadIdx.x; x < a.n_blocks * a.h; x += blockDim.x) { spos[x] = a.sdb_pos[x]; ssgn[x] = a.sdb_sgn[x]; }
    __syncthreads();
    const uint64_t nb = a.lay.M - N;
    for (uint64_t bidx = threadIdx.x; bidx < nb; bidx += blockDim.x) {
        uint32_t t, i;
        b_row_of(a.lay, bidx, t, i);
        uint64_t sa = 0;                                                 // (s_{db,t} * a)[i] mod q
        for (uint32_t c = 0; c < a.h; ++c) {
            // X^p X^(i-p): wraps with a sign flip when i < p
            const uint32_t p = (uint32_t)spos[t * a.h + c];
            const int s = ssgn[t * a.h + c];
            const uint64_t term = (i >= p) ? acol[i - p] : acol[N + i - p];
            const bool neg = (i >= p) ? (s < 0) : (s > 0);
            sa = neg ? sub_mod(sa, term, q) : add_mod(sa, term, q);
        }
        uint64_t *dst = dbl + (size_t)(N + bidx) * a.K + k;
        const int e = cbd_sample(sm64(ke, ((uint64_t)t * N + i) * a.K + k), a.eta);
        uint64_t v = sub_mod(l < a.Lq ? *dst : 0, sa, q);
        v = e >= 0 ? add_mod(v, (uint64_t)e, q) : sub_mod(v, (uint64_t)(-e), q);
        *dst = to_digit_form(v, q);
    }
}

struct QEncArgs {
    uint32_t K, d2, Nq, eta, rho, code_bits, Lq, nqblk, logc;            // 2^logc columns per block
    uint64_t seed;
    const uint8_t *codes, *masks;        // [n_eyes][code_bits/8]
    const uint64_t *eye_ids;
    icm::NttMod nt[2];
    const ulonglong2 *shat;              // [nqblk][Lq][Nq]: transforms of s_{q,t}, times Nq^-1
    uint32_t h;
    const int32_t *sq_pos; const int8_t *sq_sgn;     // [nqblk][h]: the supports, for the direct form
    uint64_t q[ICM_MAX_LIMBS], dl[ICM_MAX_LIMBS];   // primes and Delta mod q_l
    uint32_t n_cols;
    uint64_t *ct;                        // [Lq][n_cols][K]
};

// Message coefficient k of rotation r of a masked code: x_s[row, col, b] = x[row, (col + s) mod 200, b] on
// 16 x 200 x 4.
__device__ __forceinline__ int rotated_bit(const QEncArgs &a, const uint8_t *code, const uint8_t *mask, uint32_t r, uint32_t k) {
    if (k >= a.code_bits) return 0;
    const int shift = (int)r - (int)(a.rho - 1) / 2;
    const uint32_t row = k / 800, cc = (k / 4) % 200, b = k % 4;
    const uint32_t src = (row * 200 + (uint32_t)(((int)cc + shift + 200) % 200)) * 4 + b;
    const int cb = template_bit(code, src), mb = template_bit(mask, src);
    return mb - 2 * (cb & mb);
}
// b = -(s a) + Delta m + e of one coefficient, given sa = (s a) mod q
__device__ __forceinline__ uint64_t query_b(const QEncArgs &a, uint32_t l, uint64_t sa, int m, uint64_t ke, uint64_t at) {
    const uint64_t q = a.q[l];
    uint64_t v = sa ? q - sa : 0;
    if (m > 0) v = add_mod(v, a.dl[l], q);
    else if (m < 0) v = sub_mod(v, a.dl[l], q);
    const int err = cbd_sample(sm64(ke, at), a.eta);
    return err >= 0 ? add_mod(v, (uint64_t)err, q) : sub_mod(v, (uint64_t)(-err), q);
}

// One block per (2^logc query columns, limb l < Lq): the same transforms as k_db_apart_b.  32 eyes
// (992 columns, N_q = 2^13, two primes): 23.2 ms with h = 512 additions per coefficient, 1.24 ms with
// the column and eye of each word divided out, 1.01 ms with pointwise products by 128-bit reduction,
// 0.96 ms now.
template <int WPT>
__global__ void __launch_bounds__(NT_MUL, 1) k_query_encrypt(const __grid_constant__ QEncArgs a) {
    extern __shared__ uint64_t su[];                               // [2^logc][stride]
    const uint32_t C = 1u << a.logc, l = blockIdx.y, N = a.Nq, j0 = blockIdx.x << a.logc;
    const uint32_t stride = icm::ntt_words(N) + 4, CN = N << a.logc, lgN = 31 - __clz(N);
    const uint64_t q = a.q[l];
    const icm::NttMod &T = a.nt[l];
    for (uint32_t c = 0; c < C; ++c) {
        const uint32_t j = j0 + c, r = j % a.rho;
        const uint64_t ka = j < a.n_cols ? stream_key(a.seed, ICM_KIND_A_Q, a.eye_ids[j / a.rho], l) : 0;
        for (uint32_t i = threadIdx.x; i < N; i += NT_MUL) {
            uint64_t v = 0;
            if (j < a.n_cols) {
                v = uniform_mod(sm64(ka, (uint64_t)r * N + i), q);
                a.ct[((size_t)l * a.n_cols + j) * a.K + a.d2 + i] = v;
            }
            su[c * stride + icm::ntt_pad(i)] = v;
        }
    }
    __syncthreads();
    icm::ntt_forward(su, C, stride, N, T);
    // word x: coefficient x mod N of column x / N
    uint64_t ah[WPT];
#pragma unroll
    for (int w = 0; w < WPT; ++w) {
        const uint32_t x = threadIdx.x + w * NT_MUL;
        if (x < CN) ah[w] = su[(x >> lgN) * stride + icm::ntt_pad(x & (N - 1))];
    }
    const uint32_t tb = a.code_bits / 8;
    for (uint32_t t = 0; t < a.nqblk; ++t) {
        const ulonglong2 *sh = a.shat + ((size_t)t * a.Lq + l) * N;
#pragma unroll
        for (int w = 0; w < WPT; ++w) {
            const uint32_t x = threadIdx.x + w * NT_MUL;
            if (x < CN)
                su[(x >> lgN) * stride + icm::ntt_pad(x & (N - 1))] = icm::mul_lazy(ah[w], __ldg(sh + (x & (N - 1))), 0 - q);
        }
        __syncthreads();
        icm::ntt_inverse(su, C, stride, N, T);
        for (uint32_t c = 0; c < C; ++c) {
            const uint32_t j = j0 + c, e = j / a.rho, r = j % a.rho;
            if (j >= a.n_cols) break;
            const uint8_t *code = a.codes + (size_t)e * tb, *mask = a.masks + (size_t)e * tb;
            const uint64_t ke = stream_key(a.seed, ICM_KIND_E_Q, a.eye_ids[e], 0);
            uint64_t *ct = a.ct + ((size_t)l * a.n_cols + j) * a.K + (size_t)t * N;
            for (uint32_t i = threadIdx.x; i < N; i += NT_MUL) {
                const uint32_t k = t * N + i;
                const uint64_t sa = icm::sub_if(icm::sub_if(su[c * stride + icm::ntt_pad(i)], 2 * q), q);
                ct[i] = query_b(a, l, sa, rotated_bit(a, code, mask, r, k), ke, (uint64_t)r * a.d2 + k);
            }
        }
        // Word c N + i is written by thread (c N + i) mod NT_MUL above and read by thread i mod NT_MUL here:
        // the same one unless a column is shorter than the block.
        if (N < NT_MUL) __syncthreads();
    }
}

// The direct form, one block per (query column j, limb l < Lq): h additions per coefficient (query_direct).
__global__ void __launch_bounds__(1024) k_query_encrypt_direct(const __grid_constant__ QEncArgs a) {
    extern __shared__ uint64_t su[];                               // the column's a [Nq]
    const uint32_t j = blockIdx.x, l = blockIdx.y, e = j / a.rho, r = j % a.rho, N = a.Nq, tb = a.code_bits / 8;
    const uint64_t q = a.q[l];
    const uint64_t ka = stream_key(a.seed, ICM_KIND_A_Q, a.eye_ids[e], l), ke = stream_key(a.seed, ICM_KIND_E_Q, a.eye_ids[e], 0);
    const uint8_t *code = a.codes + (size_t)e * tb, *mask = a.masks + (size_t)e * tb;
    uint64_t *ct = a.ct + ((size_t)l * a.n_cols + j) * a.K;
    for (uint32_t i = threadIdx.x; i < N; i += blockDim.x) {
        const uint64_t v = uniform_mod(sm64(ka, (uint64_t)r * N + i), q);
        su[i] = v;
        ct[a.d2 + i] = v;
    }
    __syncthreads();
    for (uint32_t k = threadIdx.x; k < a.d2; k += blockDim.x) {
        const uint32_t t = k / N, i = k % N;
        uint64_t sa = 0;
        for (uint32_t c = 0; c < a.h; ++c) {
            const uint32_t p = (uint32_t)a.sq_pos[t * a.h + c];
            const int s = a.sq_sgn[t * a.h + c];
            const uint64_t term = (i >= p) ? su[i - p] : su[N + i - p];
            const bool neg = (i >= p) ? (s < 0) : (s > 0);
            sa = neg ? sub_mod(sa, term, q) : add_mod(sa, term, q);
        }
        ct[k] = query_b(a, l, sa, rotated_bit(a, code, mask, r, k), ke, (uint64_t)r * a.d2 + k);
    }
}

// Transform tables of one modulus (icm_internal.h): entry k of [0, N) is psi^bitrev(k), then psi^-1.
struct TabArgs {
    uint32_t N, logN;
    uint64_t psi, ipsi;
    icm::NttMod T;
    ulonglong2 *out;                     // [2][N]
};
__device__ __forceinline__ uint64_t mul_exact(uint64_t a, uint64_t b, const icm::NttMod &T) {
    const uint64_t r = icm::mul_r128_lazy(a, b, T);
    return r >= T.q ? r - T.q : r;
}
// (w, floor(w 2^64 / q)) for w < q: the estimate from floor(2^128 / q) is short by at most one
__device__ __forceinline__ ulonglong2 with_companion(uint64_t w, const icm::NttMod &T) {
    uint64_t ws = w * T.rhi + __umul64hi(w, T.rlo);
    if ((uint64_t)0 - ws * T.q >= T.q) ++ws;
    return make_ulonglong2(w, ws);
}
__global__ void k_ntt_table(const __grid_constant__ TabArgs a) {
    const uint32_t x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= 2 * a.N) return;
    uint32_t e = __brev(x & (a.N - 1)) >> (32 - a.logN);
    uint64_t b = x >= a.N ? a.ipsi : a.psi, w = 1;
    for (; e; e >>= 1, b = mul_exact(b, b, a.T))
        if (e & 1) w = mul_exact(w, b, a.T);
    a.out[x] = with_companion(w, a.T);
}

// Transforms of the sparse secrets, times N^-1: one block per (secret t, limb l).
struct SecArgs {
    uint32_t N, h, L;
    icm::NttMod nt[ICM_MAX_LIMBS];
    const int32_t *pos; const int8_t *sgn;           // [t][h]
    ulonglong2 *out;                                 // [t][L][N] (value, Shoup companion)
};
__global__ void __launch_bounds__(NT_MUL, 1) k_ntt_secret(const __grid_constant__ SecArgs a) {
    extern __shared__ uint64_t su[];
    const uint32_t t = blockIdx.x, l = blockIdx.y;
    const icm::NttMod &T = a.nt[l];
    for (uint32_t i = threadIdx.x; i < icm::ntt_words(a.N); i += NT_MUL) su[i] = 0;
    __syncthreads();
    for (uint32_t c = threadIdx.x; c < a.h; c += NT_MUL)
        su[icm::ntt_pad((uint32_t)a.pos[t * a.h + c])] = a.sgn[t * a.h + c] < 0 ? T.q - 1 : 1;
    __syncthreads();
    icm::ntt_forward(su, 1, 0, a.N, T);
    for (uint32_t i = threadIdx.x; i < a.N; i += NT_MUL)
        a.out[((size_t)t * a.L + l) * a.N + i] = with_companion(mulmod_shoup(su[icm::ntt_pad(i)], T.ninv, T.ninvs, T.q), T);
}

}  // namespace

namespace icm {

cudaError_t encrypt_set_attributes() {
    return allow_smem(k_db_messages<false>, k_db_messages<true>, k_db_apart_b_direct, k_db_apart_b<8>, k_db_apart_b<16>, k_db_apart_b<32>,
                      k_query_encrypt_direct, k_query_encrypt<8>, k_query_encrypt<16>, k_query_encrypt<32>, k_ntt_secret);
}

cudaError_t launch_db_messages(const icm_ctx *c, const LayoutDev &lay, const uint8_t *d_codes,
                               const uint8_t *d_masks, uint64_t *d_db, cudaStream_t st, const int32_t *d_wmsg) {
    DbMsgArgs a{};
    a.lay = lay;
    a.K = c->K; a.d2 = c->p.d2; a.Nq = c->N_q; a.nqblk = c->n_qblk; a.h = c->p.hamming_weight;
    a.code_bits = c->p.code_bits; a.Lq = c->p.n_limbs_q;
    a.codes = d_codes; a.masks = d_masks; a.wmsg = d_wmsg;
    a.sq_pos = c->d_sq_pos; a.sq_sgn = c->d_sq_sgn;
    for (uint32_t l = 0; l < a.Lq; ++l) { a.qp[l] = c->qp_mod[l]; a.qps[l] = c->qp_mods[l]; a.q[l] = c->q[l]; }
    a.db = d_db;
    const uint64_t nb = lay.M - lay.N;
    if (nb == 0) return cudaSuccess;
    // 16-bit sums of bytes below 3 hold 32,767 terms.  A query ring below 2^10 has at most 128 words of four
    // entries for 512 threads; one addition at a time then leaves fewer idle (3,000 templates, h = 512, two limbs
    // of N_db = 2^12: N_q = 2^9 24.4 ms with words of four, 15.5 without; 2^10 10.9 and 15.1).
    const bool bits = !d_wmsg && a.Nq >= 1024 && (uint64_t)a.nqblk * a.h < 32768;
    const size_t smem = (bits ? (size_t)a.nqblk * (3 * a.Nq + 4) : (size_t)((a.d2 + 3) & ~3u) * 4) + (size_t)a.nqblk * a.h * 5;
    auto run = [&](auto kern) {
        kern<<<(unsigned)nb, 512, smem, st>>>(a);
        return cudaGetLastError();
    };
    return bits ? run(k_db_messages<true>) : run(k_db_messages<false>);
}

// Columns per block of the secret-product kernels: as many as 2^14 words hold, at most `want`.
static uint32_t mul_logc(uint32_t N, uint32_t want) {
    uint32_t lc = 0;
    while ((2u << lc) <= want && ((uint64_t)N << (lc + 1)) <= 16384) ++lc;
    return lc;
}
static size_t mul_smem(uint32_t N, uint32_t logc) { return ((size_t)(ntt_words(N) + 4) << logc) * 8; }

template <typename K, typename A>
static cudaError_t launch_mul(K kern, const A &a, dim3 grid, size_t smem, cudaStream_t st) {
    kern<<<grid, NT_MUL, smem, st>>>(a);
    return cudaGetLastError();
}

// Whether h additions per stored b-row cost less than a forward transform and an inverse one per block, per
// column and limb.  Measured in additions (1.24 ps each), a transform takes 7 per coefficient, and 4,500 in rings
// below 2^9, which leave its threads idle.  L = 4, ms, additions / transforms:
//   h = 512, 100 templates: N_db = 2^12 11.6 / 8.4, 2^13 16.0 / 22.3, 2^14 21.6 / 52.6
//   h = 512, 1,000: 2^13 70.7 / 23.6;  h = 64, 3,000: 2^7 18.7 / 18.7, 2^8 18.5 / 10.8, 2^12 23.4 / 10.6
//   h = 64, 100: 2^12 3.8 / 8.3, 2^11 2.5 / 4.0, 2^10 2.3 / 2.3;  h = 16, 3,000: 2^5 8.5 / 39.8, 2^7 7.3 / 14.6
static bool db_direct(uint32_t h, uint32_t N, uint32_t n_blocks, uint64_t rows) {
    return rows * h < (uint64_t)(n_blocks + 1) * std::max(7 * N, 4500u) &&
           (size_t)N * 8 + (size_t)n_blocks * h * 5 <= 200 * 1024;
}

cudaError_t launch_db_apart_and_b(const icm_ctx *c, const LayoutDev &lay, uint64_t chunk_id, uint64_t *d_db,
                                  cudaStream_t st) {
    if (!c->nt.shat_db) return cudaErrorInvalidValue;                    // rings above 2^14
    DbEncArgs a{};
    a.lay = lay; a.K = c->K; a.eta = c->p.noise_eta; a.Lq = c->p.n_limbs_q;
    a.n_blocks = (uint32_t)((lay.M - lay.N) ? (lay.n_full + (lay.rem ? 1 : 0)) : 0);
    a.seed = c->p.seed; a.chunk = chunk_id;
    a.logc = mul_logc(lay.N, 4);
    for (uint32_t l = 0; l < c->p.n_limbs; ++l) a.nt[l] = c->nt.db[l];
    a.shat = c->nt.shat_db;
    a.lt = c->lt; a.db = d_db;
    if (db_direct(c->p.hamming_weight, lay.N, a.n_blocks, lay.M - lay.N)) {
        a.h = c->p.hamming_weight; a.sdb_pos = c->d_sdb_pos; a.sdb_sgn = c->d_sdb_sgn;
        const size_t smem = (size_t)lay.N * 8 + (size_t)a.n_blocks * a.h * 5;
        k_db_apart_b_direct<<<dim3(c->K, c->p.n_limbs), 1024, smem, st>>>(a);
        return cudaGetLastError();
    }
    const size_t smem = mul_smem(lay.N, a.logc);
    dim3 grid((c->K + (1u << a.logc) - 1) >> a.logc, c->p.n_limbs);
    const uint32_t wpt = (uint32_t)(((uint64_t)lay.N << a.logc) + NT_MUL - 1) / NT_MUL;
    return wpt > 16 ? launch_mul(k_db_apart_b<32>, a, grid, smem, st)
                    : wpt > 8 ? launch_mul(k_db_apart_b<16>, a, grid, smem, st) : launch_mul(k_db_apart_b<8>, a, grid, smem, st);
}

// Whether h additions per coefficient cost less than the transforms of a column (one forward, one inverse per
// secret), per limb.  12 eyes, two primes, d2 = 2^14, us, additions / transforms: h = 16 N_q = 2^5 478 / 4,800, 2^7
// 472 / 1,700, 2^9 472 / 695, 2^10 471 / 528, 2^13 482 / 568; h = 64 2^7 1,246 / 1,674, 2^8 1,248 / 1,008, 2^10
// 1,242 / 528; h = 512 8,420 / 470 to 690.
static bool query_direct(uint32_t h, uint32_t d2, uint32_t N) {
    return (uint64_t)h * d2 < (uint64_t)(d2 / N + 1) * std::max(16 * N, 11500u);
}

cudaError_t launch_query_encrypt(const icm_ctx *c, const uint8_t *d_codes, const uint8_t *d_masks,
                                 const uint64_t *d_eye_ids, uint32_t n_eyes, uint64_t *d_ct, cudaStream_t st) {
    QEncArgs a{};
    a.K = c->K; a.d2 = c->p.d2; a.Nq = c->N_q; a.eta = c->p.noise_eta;
    a.rho = c->p.rho; a.code_bits = c->p.code_bits; a.Lq = c->p.n_limbs_q; a.nqblk = c->n_qblk;
    a.seed = c->p.seed; a.codes = d_codes; a.masks = d_masks; a.eye_ids = d_eye_ids;
    for (uint32_t l = 0; l < a.Lq; ++l) { a.q[l] = c->q[l]; a.dl[l] = c->delta_mod[l]; a.nt[l] = c->nt.q[l]; }
    a.shat = c->nt.shat_q;
    a.n_cols = n_eyes * c->p.rho;
    a.ct = d_ct;
    if (a.n_cols == 0) return cudaSuccess;
    if (!a.shat) return cudaErrorInvalidValue;                           // rings above 2^14
    if (query_direct(c->p.hamming_weight, a.d2, a.Nq)) {
        a.h = c->p.hamming_weight; a.sq_pos = c->d_sq_pos; a.sq_sgn = c->d_sq_sgn;
        k_query_encrypt_direct<<<dim3(a.n_cols, a.Lq), 1024, (size_t)a.Nq * 8, st>>>(a);
        return cudaGetLastError();
    }
    // two columns share their twiddles where there are enough of them to fill the SMs
    a.logc = mul_logc(a.Nq, a.n_cols * a.Lq >= 2 * 152 ? 2 : 1);
    const size_t smem = mul_smem(a.Nq, a.logc);
    dim3 grid((a.n_cols + (1u << a.logc) - 1) >> a.logc, a.Lq);
    const uint32_t wpt = ((a.Nq << a.logc) + NT_MUL - 1) / NT_MUL;
    return wpt > 16 ? launch_mul(k_query_encrypt<32>, a, grid, smem, st)
                    : wpt > 8 ? launch_mul(k_query_encrypt<16>, a, grid, smem, st)
                              : launch_mul(k_query_encrypt<8>, a, grid, smem, st);
}

// Builds the transform tables and the secrets' transforms into the empty set S (icm_keygen, from the supports
// on the device; after an error the caller releases S).  Rings above 2^14 have no secret-product
// kernels and get no tables.
cudaError_t build_ntt(const icm_ctx *c, const int32_t *sdb_pos, const int8_t *sdb_sgn, uint32_t n_sdb, const int32_t *sq_pos,
                      const int8_t *sq_sgn, NttSet &S, std::string &why) {
    const uint32_t rings[2] = {c->N_db, c->N_q}, limbs[2] = {c->p.n_limbs, c->p.n_limbs_q};
    const uint32_t secrets[2] = {n_sdb, c->n_qblk};
    for (int w = 0; w < 2; ++w) {
        const uint32_t N = rings[w], L = limbs[w];
        if (N > 16384) continue;
        uint32_t logN = 0;
        while ((1u << logN) < N) ++logN;
        ulonglong2 **tab = w ? &S.tab_q : &S.tab_db;
        ulonglong2 **shat = w ? &S.shat_q : &S.shat_db;
        NttMod *nt = w ? S.q : S.db;
        cudaError_t e = cudaMalloc(tab, (size_t)L * 2 * N * sizeof(ulonglong2));
        if (e != cudaSuccess) return e;
        for (uint32_t l = 0; l < L; ++l) {
            const uint64_t q = c->q[l];
            if ((q - 1) % (2ull * N)) { why = "primes must be 1 mod 2 N"; return cudaErrorInvalidValue; }
            // psi: a primitive 2N-th root of unity, g^((q-1)/2N) for a quadratic non-residue g
            uint64_t psi = 0;
            for (uint64_t g = 2; g < 1000 && !psi; ++g)
                if (pow_mod(g, (q - 1) / 2, q) == q - 1) psi = pow_mod(g, (q - 1) / (2ull * N), q);
            if (!psi || pow_mod(psi, N, q) != q - 1) { why = "no primitive 2N-th root"; return cudaErrorInvalidValue; }
            NttMod &m = nt[l];
            m.q = q;
            m.ninv = pow_mod(N, q - 2, q); m.ninvs = shoup_of(m.ninv, q);
            m.rhi = c->crt.rhi[l]; m.rlo = c->crt.rlo[l];
            m.fwd = *tab + (size_t)l * 2 * N; m.inv = m.fwd + N;
            TabArgs a{N, logN, psi, pow_mod(psi, q - 2, q), m, *tab + (size_t)l * 2 * N};
            k_ntt_table<<<(2 * N + 255) / 256, 256>>>(a);
        }
        e = cudaMalloc(shat, (size_t)secrets[w] * L * N * sizeof(ulonglong2));
        if (e != cudaSuccess) return e;
        SecArgs a{};
        a.N = N; a.h = c->p.hamming_weight; a.L = L;
        for (uint32_t l = 0; l < L; ++l) a.nt[l] = nt[l];
        a.pos = w ? sq_pos : sdb_pos; a.sgn = w ? sq_sgn : sdb_sgn;
        a.out = *shat;
        e = launch_mul(k_ntt_secret, a, dim3(secrets[w], L), (size_t)ntt_words(N) * 8, nullptr);
        if (e != cudaSuccess) return e;
    }
    return cudaStreamSynchronize(nullptr);
}

void NttSet::release() {
    cudaFree(tab_db); cudaFree(tab_q); cudaFree(shat_db); cudaFree(shat_q);
    *this = NttSet{};
}

}  // namespace icm
