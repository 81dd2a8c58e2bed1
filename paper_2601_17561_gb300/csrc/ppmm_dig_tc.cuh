// The fp16 form for few columns on the tcgen05 tensor cores (included by ppmm_crt_tc.cu, whose
// barrier, TMA, MMA and TMEM helpers it uses).
//
// With few columns the CRT kernel is bound by the conversion of every database word to r = 18
// residues (9 instructions per two words and modulus), whatever the width of the product.  Here the
// database enters as it is stored: word a = sum_t 256^t d_t with signed bytes d_t, which are exact
// fp16 integers after 5 instructions per four of them, and the weights go to the query side,
//     C = sum_k a[k] b[k] = sum_k sum_t d_t[k] (256^t b[k] mod q)  (mod q),
// where 256^t b[k] mod q is split into 8 signed bytes in turn: C = sum_u 256^u S_u with
// S_u = sum_{k,t} d_t[k] e_{t,u}[k].  That is one fp16 product of depth 8 K with 8 columns per query
// column, 64 products per modular multiply-add instead of 18, but no residues: 256 MMA columns take
// 32 query columns through 8 words of K in 512 cycles per 256 rows (a pair of blocks), at the full
// rate of M 256 N 256.  So it pays up to 64 columns (two passes over a row tile), where the CRT
// kernel's time has not begun to depend on the width.
//   Measured (GB300, 8 limbs, N_db = 2^12, full pass): 1 eye x 3,000 codes 3.8 ms, CRT 13.1 ms.
//
// Exactness: |d_t|, |e| <= 128, so 960 products and a residue of the previous sums stay below 2^24
// in the fp32 accumulators.  Two accumulators of 256 columns take intervals of 960 products in turn;
// while one is filled, the epilogue passes the carries of the other one up the digits, S_u -> S_u -
// 256 c_u, S_{u+1} += c_u, which leaves |S_u| <= 128, and collects the carry out of the top digit in
// registers.  So the MMAs never wait for a reduction.  Query operand: dig_planes_bytes.
#pragma once

constexpr int DG_ROWS = 128;                      // database rows of a block (M 256 over the pair)
constexpr int DG_TILE = 2 * DG_ROWS;              // database rows of a pair
constexpr int DG_WORDS = 8;                       // storage words of K in a stage (64 of the MMA's K)
constexpr int DG_BLK = 2048;                      // one word: 128 rows or columns x 8 digits x 2 bytes
constexpr int DG_OP = DG_WORDS * DG_BLK;          // 16 KB: one operand of a block and stage
constexpr int DG_RAW = DG_ROWS * 16 * 8;          // 16 KB: raw slab of 16 words, two stages
constexpr int DG_S = 4, DG_RS = 4;                // operand stages, raw slots
constexpr uint32_t DG_FLUSH = 15;                 // stages between hand-overs of an accumulator (960 products)
constexpr int DG_OFF_A = DG_RS * DG_RAW, DG_OFF_B = DG_OFF_A + DG_S * DG_OP, DG_BARS = DG_OFF_B + DG_S * DG_OP;
constexpr int DG_SMEM = DG_BARS + 1024 + 1024;
constexpr int DG_NCV = 8, DG_W_EPI = DG_NCV, DG_W_RAW = DG_W_EPI + 8, DG_W_QRY = DG_W_RAW + 1, DG_W_MMA = DG_W_QRY + 1;
constexpr int DG_THREADS = (DG_W_MMA + 1) * 32;
static_assert(DG_SMEM <= 227 * 1024, "shared memory budget");

struct DigArgs {
    CUtensorMap tmA[ICM_MAX_CHUNKS];  // per chunk: [L][M_c][K] u64, box 16 x 128, 128-byte swizzle
    CUtensorMap tmB;                  // digit planes as rows of 2 KB: [L][groups][2][Kp]
    icm::ChunkTab tab;
    uint32_t t0[ICM_MAX_CHUNKS + 1];  // prefix sums of 256-row tiles
    uint64_t N, K, Kp;                // query columns of this product
    uint64_t col0, n_out;             // their first column in the outputs, columns of the outputs
    uint32_t n_limbs, groups;         // column groups of 32
    uint64_t n_tiles;                 // L x row tiles x groups
    uint64_t wait_ns;
    uint32_t inject_stall;
    uint64_t q[ICM_MAX_LIMBS], r64[ICM_MAX_LIMBS], p32[ICM_MAX_LIMBS], p32s[ICM_MAX_LIMBS];   // 2^32 mod q
};

struct __align__(8) DigBars {
    uint64_t rawfull[DG_RS], rawempty[DG_RS], full[DG_S], empty[DG_S], accfull[2], accfree[2], done;
    uint32_t tmem;
    int abort_flag;
};

struct DigTile { uint32_t l, c, g; uint64_t m0, M; };
// tile -> (limb, row tile, column group), the group fastest
__device__ __forceinline__ DigTile dig_tile(const DigArgs &p, uint64_t tile) {
    DigTile t;
    t.g = (uint32_t)(tile % p.groups);
    tile /= p.groups;
    const uint32_t rt = (uint32_t)(tile % p.t0[p.tab.n]);
    t.l = (uint32_t)(tile / p.t0[p.tab.n]);
    uint32_t c = 0;
    while (c + 1 < p.tab.n && rt >= p.t0[c + 1]) ++c;
    t.c = c;
    t.M = p.tab.M[c];
    t.m0 = (uint64_t)(rt - p.t0[c]) * DG_TILE;
    return t;
}

constexpr uint32_t DG_IDESC = (1u << 4) | ((uint32_t)(256 >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
__device__ __forceinline__ void dig_umma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 :: "r"(d_tmem), "l"(a), "l"(b), "r"(DG_IDESC), "r"(accumulate) : "memory");
}

// Four signed bytes as fp16: the bytes offset by 128 under the high byte 0x64 are the f16 1024 + 128 + d.
__device__ __forceinline__ uint2 digits4(uint32_t x) {
    const uint32_t y = x ^ 0x80808080u;
    uint2 o;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o.x) : "r"(__byte_perm(y, 0x64u, 0x4140)), "r"(0xE480E480u));
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o.y) : "r"(__byte_perm(y, 0x64u, 0x4342)), "r"(0xE480E480u));
    return o;
}
// Passes the carries of eight digit sums up; returns the carry out of the last.
__device__ __forceinline__ float carry8(uint32_t *v) {
    float c = 0.0f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const float x = __uint_as_float(v[u]) + c;
        c = __fsub_rn(fmaf(x, 0.00390625f, RINT), RINT);
        v[u] = __float_as_uint(fmaf(-256.0f, c, x));
    }
    return c;
}

__global__ void __launch_bounds__(DG_THREADS, 1) k_dig_tc(const __grid_constant__ DigArgs p) {
    static_assert(sizeof(DigBars) <= 1024, "barrier block");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char *sW = smem, *sA = smem + DG_OFF_A, *sB = smem + DG_OFF_B;
    DigBars *bars = reinterpret_cast<DigBars *>(smem + DG_BARS);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const WaitCtx wc{&bars->abort_flag, nullptr, p.wait_ns};
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const uint32_t b_rawfull = smem_u32(bars->rawfull), b_rawempty = smem_u32(bars->rawempty);
    const uint32_t b_full = smem_u32(bars->full), b_empty = smem_u32(bars->empty);
    const uint32_t b_accfull = smem_u32(bars->accfull), b_accfree = smem_u32(bars->accfree);

    if (tid == 0) {
        for (int s = 0; s < DG_RS; ++s) { mbar_init(&bars->rawfull[s], 1); mbar_init(&bars->rawempty[s], 4); }
        for (int s = 0; s < DG_S; ++s) {
            mbar_init(&bars->full[s], 2 * 2 + 1);       // the converter warps of both blocks + the leader's announcement
            mbar_init(&bars->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) { mbar_init(&bars->accfull[b], 1); mbar_init(&bars->accfree[b], 2 * 8); }
        mbar_init(&bars->done, 1);
        bars->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&bars->tmem)), "r"(TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = bars->tmem;

    const uint32_t nk = (uint32_t)((p.K + 15) / 16), nst = 2 * nk;      // raw slabs and stages of a tile
    const uint32_t n_iv = (nst + DG_FLUSH - 1) / DG_FLUSH;              // accumulator intervals of a tile
    const uint32_t t_first = blockIdx.x >> 1, t_step = gridDim.x >> 1;

    if (warp < DG_NCV) {
        // converters: group grp (2 warps of 64 rows) takes the stages u mod 4 = grp, half a raw slab each.
        // A lane loads 16 bytes (words 2c, 2c + 1 of the stage) of row (lane mod 8) + 8 i and stores the 8
        // digits of each as a 16-byte row of a core matrix; all accesses are free of bank conflicts.
        const uint32_t grp = (uint32_t)warp & 3, sub = (uint32_t)warp >> 2;
        const uint32_t c = (uint32_t)lane >> 3, rr = lane & 7, h = grp & 1;
        const uint32_t roff = (sub * 64 + rr) * 128 + (((4 * h + c) ^ rr) << 4);
        const uint32_t aoff = 2 * c * DG_BLK + sub * 1024 + rr * 16;
        const uint32_t full0 = map_rank(b_full, 0);
        uint64_t u = grp, u_end = 0;
        uint32_t rs = grp >> 1, rpar = 0, spar = 0;
        bool alive = true;
        for (uint64_t tile = t_first; alive && tile < p.n_tiles; tile += t_step) {
            u_end += nst;
            for (; u < u_end; u += 4) {
                if (!mbar_wait(b_rawfull + rs * 8, rpar, wc)) { alive = false; break; }
                // half of the words are converted before the stage is free, the others are loaded: what
                // follows the wait is in the ring's turnaround
                const unsigned char *src = sW + rs * DG_RAW + roff;
                unsigned char *dst = sA + grp * DG_OP + aoff;
                uint4 z[8], y[4];
#pragma unroll
                for (int i = 0; i < 8; ++i) z[i] = *reinterpret_cast<const uint4 *>(src + i * 1024);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint2 w0 = digits4(z[i].x), w1 = digits4(z[i].y), w2 = digits4(z[i].z), w3 = digits4(z[i].w);
                    z[i] = make_uint4(w0.x, w0.y, w1.x, w1.y);
                    y[i] = make_uint4(w2.x, w2.y, w3.x, w3.y);
                }
                if (!mbar_wait(b_empty + grp * 8, spar ^ 1, wc)) { alive = false; break; }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    *reinterpret_cast<uint4 *>(dst + i * 128) = z[i];
                    *reinterpret_cast<uint4 *>(dst + DG_BLK + i * 128) = y[i];
                }
#pragma unroll
                for (int i = 4; i < 8; ++i) {
                    const uint2 w0 = digits4(z[i].x), w1 = digits4(z[i].y), w2 = digits4(z[i].z), w3 = digits4(z[i].w);
                    *reinterpret_cast<uint4 *>(dst + i * 128) = make_uint4(w0.x, w0.y, w1.x, w1.y);
                    *reinterpret_cast<uint4 *>(dst + DG_BLK + i * 128) = make_uint4(w2.x, w2.y, w3.x, w3.y);
                }
                // the stores hold every raw word, so the reads have returned when the slot goes back
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(b_rawempty + rs * 8);
                    mbar_arrive_cluster(full0 + grp * 8);
                }
                rs += 2;
                if (rs >= (uint32_t)DG_RS) { rs -= DG_RS; rpar ^= 1; }
                spar ^= 1;
            }
        }
    } else if (warp < DG_W_RAW) {
        // epilogue: two warps per TMEM lane quarter, 16 query columns (128 accumulator columns) each
        const uint32_t qtr = (uint32_t)warp & 3, half = (uint32_t)(warp - DG_W_EPI) >> 2;
        const uint32_t free0 = map_rank(b_accfree, 0);
        const uint32_t tb = tmem + ((qtr * 32) << 16) + half * 128;
        uint32_t ev = 0;
        bool alive = true;
        for (uint64_t tile = t_first; alive && tile < p.n_tiles; tile += t_step) {
            const DigTile tc = dig_tile(p, tile);
            float top[16];
#pragma unroll
            for (int n = 0; n < 16; ++n) top[n] = 0.0f;
            for (uint32_t iv = 0; iv < n_iv; ++iv) {
                const uint32_t b = iv & 1;
                if (!mbar_wait(b_accfull + b * 8, (ev >> b) & 1, wc)) { alive = false; break; }
                ev ^= 1u << b;
                tc_fence_after();
                if (iv + 1 < n_iv) {
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        uint32_t v[32];
                        tmem_ld<32>(tb + b * 256 + x * 32, v);
#pragma unroll
                        for (int n = 0; n < 4; ++n) top[4 * x + n] += carry8(v + 8 * n);
                        tmem_st<32>(tb + b * 256 + x * 32, v);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                    // the last but one interval's sums are read again with the last's
                    if (iv + 2 < n_iv) {
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(free0 + b * 8);
                    }
                } else {
                    const uint64_t q = p.q[tc.l], r64 = p.r64[tc.l];
                    const uint64_t row = tc.m0 + rank * DG_ROWS + qtr * 32 + lane;
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        uint32_t v[32];
                        tmem_ld<32>(tb + b * 256 + x * 32, v);
                        if (n_iv > 1) {
                            uint32_t w[32];
                            tmem_ld<32>(tb + (b ^ 1) * 256 + x * 32, w);
#pragma unroll
                            for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) + __uint_as_float(w[i]));
                        }
#pragma unroll
                        for (int n = 0; n < 4; ++n) {
                            // sum_u 256^u S_u = lo + 2^32 hi with |lo| < 2^40 and |hi| < 2^54
                            const float tp = top[4 * x + n] + carry8(v + 8 * n);
                            int64_t lo = 0, hi = (int64_t)__float2int_rn(tp);
#pragma unroll
                            for (int u = 3; u >= 0; --u) {
                                lo = lo * 256 + __float2int_rn(__uint_as_float(v[8 * n + u]));
                                hi = hi * 256 + __float2int_rn(__uint_as_float(v[8 * n + 4 + u]));
                            }
                            const uint64_t col = (uint64_t)tc.g * 32 + half * 16 + 4 * x + n;
                            if (row < tc.M && col < p.N)
                                p.tab.C[tc.c][((size_t)tc.l * p.n_out + p.col0 + col) * tc.M + row] =
                                    add_mod(reduce_s64(lo, q, r64), mulmod_shoup(reduce_s64(hi, q, r64), p.p32[tc.l], p.p32s[tc.l], q), q);
                        }
                        __syncwarp();
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) {
                        mbar_arrive_cluster(free0 + b * 8);
                        if (n_iv > 1) mbar_arrive_cluster(free0 + (b ^ 1) * 8);
                    }
                }
            }
        }
    } else if (warp == DG_W_RAW) {
        const bool el = elect_one();
        uint64_t n = 0;
        uint32_t rs = 0, rpar = 0;
        bool alive = true;
        for (uint64_t tile = t_first; alive && tile < p.n_tiles; tile += t_step) {
            const DigTile tc = dig_tile(p, tile);
            const int row = (int)(tc.m0 + rank * DG_ROWS);
            for (uint32_t kt = 0; kt < nk; ++kt, ++n) {
                if (!mbar_wait(b_rawempty + rs * 8, rpar ^ 1, wc)) { alive = false; break; }
                if (el) {
                    mbar_expect_tx(b_rawfull + rs * 8, DG_RAW);
                    tma_load_3d(smem_u32(sW) + rs * DG_RAW, &p.tmA[tc.c], (int)(kt * 16), row, (int)tc.l, b_rawfull + rs * 8);
                }
                __syncwarp();
                if (++rs == (uint32_t)DG_RS) { rs = 0; rpar ^= 1; }
            }
        }
        const uint64_t deadline = gtime() + p.wait_ns;
        for (uint64_t i = n > (uint64_t)DG_RS ? n - DG_RS : 0; i < n; ++i)
            mbar_wait_until(&bars->rawfull[i % DG_RS], (uint32_t)((i / DG_RS) & 1), deadline);
    } else if (warp == DG_W_QRY) {
        const bool el = elect_one();
        const uint32_t full0 = map_rank(b_full, 0);
        uint64_t n = 0;
        uint32_t s = 0, spar = 0;
        bool alive = true;
        for (uint64_t tile = t_first; alive && tile < p.n_tiles && !p.inject_stall; tile += t_step) {
            const DigTile tc = dig_tile(p, tile);
            const uint32_t row0 = (uint32_t)((((uint64_t)tc.l * p.groups + tc.g) * 2 + rank) * p.Kp);
            for (uint32_t st = 0; st < nst; ++st, ++n) {
                if (!mbar_wait(b_empty + s * 8, spar ^ 1, wc)) { alive = false; break; }
                if (el) {
                    if (rank == 0) mbar_expect_tx(b_full + s * 8, 2 * DG_OP);
                    tma_load_2d_pair(smem_u32(sB) + s * DG_OP, &p.tmB, 0, (int)(row0 + st * DG_WORDS), full0 + s * 8);
                }
                __syncwarp();
                if (++s == (uint32_t)DG_S) { s = 0; spar ^= 1; }
            }
        }
        const uint64_t deadline = gtime() + p.wait_ns;
        for (uint64_t i = n > (uint64_t)DG_S ? n - DG_S : 0; i < n; ++i)
            mbar_wait_until(&bars->empty[i % DG_S], (uint32_t)((i / DG_S) & 1), deadline);
    } else if (rank == 0) {
        const bool el = elect_one();
        const uint64_t adesc0 = sdesc(smem_u32(sA), DG_BLK, 128), bdesc0 = sdesc(smem_u32(sB), DG_BLK, 128);
        uint32_t s = 0, par = 0, used = 0, fpar = 0;                     // accumulators used before, parities of accfree
        bool alive = true, ready = false;                                // ready: the next stage has been seen full
        for (uint64_t tile = t_first; alive && tile < p.n_tiles; tile += t_step) {
            uint32_t left = 0, iv = 0, b = 1;                            // stages left of interval iv - 1, its accumulator
            for (uint32_t st = 0; st < nst; ++st) {
                const bool start = left == 0;
                if (start) {
                    b = iv & 1;
                    if ((used >> b) & 1) {
                        if (!mbar_wait(b_accfree + b * 8, (fpar >> b) & 1, wc)) { alive = false; break; }
                        fpar ^= 1u << b;
                    }
                    used |= 1u << b;
                    left = DG_FLUSH;
                    ++iv;
                }
                if (!ready && !mbar_wait<true>(b_full + s * 8, par, wc)) { alive = false; break; }
                tc_fence_after();
                --left;
                const uint64_t ad = adesc0 + (uint64_t)(s * (DG_OP >> 4)), bd = bdesc0 + (uint64_t)(s * (DG_OP >> 4));
                const uint32_t d = tmem + b * 256;
                constexpr int LAST = DG_WORDS / 2 - 1;
                if (el) {
#pragma unroll
                    for (int k = 0; k < LAST; ++k)
                        dig_umma(d, ad + (uint64_t)(k * ((2 * DG_BLK) >> 4)), bd + (uint64_t)(k * ((2 * DG_BLK) >> 4)),
                                 start && iv <= 2 && k == 0 ? 0u : 1u);
                }
                __syncwarp();
                // the next stage's barrier is probed while the tensor core is busy (see k_crt_tc)
                const uint32_t sn = s + 1 == (uint32_t)DG_S ? 0 : s + 1, pn = s + 1 == (uint32_t)DG_S ? par ^ 1u : par;
                ready = mbar_test<true>(b_full + sn * 8, pn);
                if (el) {
                    dig_umma(d, ad + (uint64_t)(LAST * ((2 * DG_BLK) >> 4)), bd + (uint64_t)(LAST * ((2 * DG_BLK) >> 4)), 1u);
                    umma_commit(b_empty + s * 8);
                    if (left == 0 || st + 1 == nst) umma_commit(b_accfull + b * 8);
                }
                ready = __all_sync(0xffffffffu, ready);
                s = sn; par = pn;
            }
        }
        if (el) umma_commit(smem_u32(&bars->done));
        __syncwarp();
        mbar_wait_until(&bars->done, 0, gtime() + p.wait_ns);
    }
    tc_fence_before();
    __syncthreads();
    if (rank == 1 && tid == 0) mbar_wait_until(&bars->done, 0, gtime() + p.wait_ns);
    __syncwarp();
    cluster_sync();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Digit planes of the query operand: [L][groups of 32 columns][2][Kp] blocks of 2 KB, block (half, k) holding
// for 16 columns x 8 digits u the 8 values t of digit u of 256^t b[k] mod q (a core-matrix row of 16
// bytes); zero beyond N and K.  Eight lanes take a word: lane t forms 256^t b mod q and its bytes, the
// lanes transpose the 8 x 8 bytes among themselves (three exchanges), and lane u stores row u, so a
// warp's stores fill 512 contiguous bytes.  Bound by those stores (128 bytes per operand word): 1 eye, 8
// limbs, 805 MB in 162 us (494 us with a word per lane, whose stores were 128 bytes apart).
struct DigPlanesArgs {
    const uint64_t *op;               // first column of [L][n_op][K] canonical residues
    unsigned char *planes;
    uint64_t n_op, N, K, Kp;
    uint32_t groups;
    uint64_t q[ICM_MAX_LIMBS], w[ICM_MAX_LIMBS][8], ws[ICM_MAX_LIMBS][8];    // 256^t mod q, Shoup companions
};
__global__ void __launch_bounds__(256) k_dig_planes(const __grid_constant__ DigPlanesArgs a) {
    const uint32_t l = blockIdx.y, lane = threadIdx.x & 31, t = lane & 7, sub = lane >> 3;
    const uint64_t q = a.q[l], w = a.w[l][t], ws = a.ws[l][t];
    // a warp: 4 columns of a half group x 8 consecutive k
    const uint64_t n_oct = a.Kp / 8, total = n_oct * a.groups * 8;
    for (uint64_t x = (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5); x < total; x += (uint64_t)gridDim.x * 8) {
        const uint64_t y = x >> 3, k0 = (y % n_oct) * 8;
        const uint32_t g = (uint32_t)(y / n_oct), nl = (uint32_t)(x & 7) * 4 + sub;   // column of the group
        const uint64_t n = (uint64_t)g * 32 + nl;
        const uint64_t *src = a.op + ((size_t)l * a.n_op + n) * a.K;
        unsigned char *dst = a.planes + ((((size_t)l * a.groups + g) * 2 + (nl >> 4)) * a.Kp + k0) * DG_BLK + (nl & 15) * 128 + t * 16;
        for (uint32_t i = 0; i < 8; ++i) {
            const uint64_t v = (n < a.N && k0 + i < a.K) ? __ldg(src + k0 + i) : 0;
            const uint64_t z = to_digit_form(mulmod_shoup(v, w, ws, q), q) ^ ICM_DIGIT_BIAS;
            uint32_t lo = (uint32_t)z, hi = (uint32_t)(z >> 32);         // bytes u of lane t -> bytes t of lane u
            {   // 4-byte halves between lanes t and t ^ 4
                const uint32_t r = __shfl_xor_sync(0xffffffffu, t & 4 ? lo : hi, 4);
                if (t & 4) lo = r; else hi = r;
            }
            {   // 2-byte pairs between lanes t and t ^ 2
                const uint32_t r = __shfl_xor_sync(0xffffffffu, __byte_perm(lo, hi, t & 2 ? 0x5410 : 0x7632), 2);
                if (t & 2) { lo = __byte_perm(r, lo, 0x7610); hi = __byte_perm(r, hi, 0x7632); }
                else { lo = __byte_perm(lo, r, 0x5410); hi = __byte_perm(hi, r, 0x7610); }
            }
            {   // bytes between lanes t and t ^ 1
                const uint32_t r = __shfl_xor_sync(0xffffffffu, __byte_perm(lo, hi, t & 1 ? 0x6420 : 0x7531), 1);
                if (t & 1) { lo = __byte_perm(r, lo, 0x7150); hi = __byte_perm(r, hi, 0x7352); }
                else { lo = __byte_perm(lo, r, 0x5240); hi = __byte_perm(hi, r, 0x7260); }
            }
            uint4 o;
            asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o.x) : "r"(__byte_perm(lo, 0x64u, 0x4140)), "r"(0xE480E480u));
            asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o.y) : "r"(__byte_perm(lo, 0x64u, 0x4342)), "r"(0xE480E480u));
            asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o.z) : "r"(__byte_perm(hi, 0x64u, 0x4140)), "r"(0xE480E480u));
            asm("add.rn.f16x2 %0, %1, %2;" : "=r"(o.w) : "r"(__byte_perm(hi, 0x64u, 0x4342)), "r"(0xE480E480u));
            *reinterpret_cast<uint4 *>(dst + (size_t)i * DG_BLK) = o;
        }
    }
}
