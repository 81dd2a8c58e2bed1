// Phase 1 of the fp16 small-modulus CRT product on the tcgen05 tensor cores (Blackwell 5th-gen
// MMA with accumulators in tensor memory).  Same arithmetic as k_crt_p1<fp16> (ppmm_crt.cu):
// for one (limb, database chunk, 128-row tile, modulus m_i, column round of up to 1,024) it computes
// c_i = (sum_k a[k] b[k]) mod m_i over residues held exactly in fp16 (at most 128 in magnitude on the database
// side, where the rounding of s / m may miss by less than 1 / m, and 127 on the query side), accumulating
// in fp32 TMEM and reducing each accumulator modulo m_i (to a remainder below m_i <= 255 in magnitude) every
// 1,024 columns of K, so that it stays an exact integer: 1024 * 128 * 127 + 254 < 2^24.  c_i goes to the byte scratch
// that phase 2 (k_crt_combine) recombines.
//
// Tile of one block pair (a cluster of two on cta_group::2).  The queries are the M side and the
// database rows the N side of the MMA (M 256 over the pair, N 128, K 16): a column group of 256
// query columns x 128 database rows is one accumulator of 128 TMEM columns in each block (block
// rank r holds its own 128 of the 256 query columns, in its TMEM lanes), and four of them fill the
// 512 TMEM columns.  So a pair covers 128 database rows x 1,024 query columns, and each block
// fetches and converts only 64 of the 128 rows: half the conversions, half the raw bytes and half
// the database passes of a block that works alone on 128 x 512, with the same bytes of query
// planes per MMA.  With fewer columns the accumulators are shared out to several moduli of the
// same row tile (G column groups x NM moduli <= 4), which read one raw slab.
//   Copies: a bulk copy issued inside a lane-dependent branch takes a thread 51 cycles, an elected one 17, and
//   one copy of 4 to 16 KB ~383 cycles, so an operand stage is 32 deep (one copy of up to 32 KB per
//   modulus) and producers and issuer run on warp-uniform values with one elected lane.  Conversions:
//   9 half-rate instructions per two residues (res_pair).
//   The MMA runs at 71 cycles for M 256 N 128 K 16 (64 is the peak; N 256 reaches 128 of 128, but
//   needs twice the conversions): 570 cycles per 32-deep stage.
//   Measured (GB300): 32 eyes against N_db + 16,384 rows, 8 limbs: 218 -> 161 to 166 ms per pass; 734 cycles
//   per stage at the 1.75 GHz that the power limit leaves.  What is left is the ring: 4 stages of
//   36 KB, of which an accumulator under reduction holds up to two.
//
// Pipeline, the stages decoupled by rings of shared-memory slots with "full" / "empty" mbarriers:
//  * raw producer (1 warp per block): one TMA load per 16-deep slab of the 64 x
//    16 balanced-digit storage words of the block's rows (128-byte swizzle: the 16-byte chunk c of
//    row r sits at chunk c ^ (r mod 8)) into a ring of RS raw slots;
//  * converters (8 warps in NCG = 4 groups): the group of slab g (g mod NCG) converts it, each warp
//    32 rows: 8 consecutive storage words of a row become 8 fp16 residues in registers, then, once
//    the operand stage is free, 16-byte stores into the MMA's K-major core-matrix layout (no
//    swizzle);
//  * query producer (1 warp per block): per stage and modulus one TMA load of the block's pre-tiled plane
//    block, signalled on the leader's barrier;
//  * MMA issuer (leader block only): per stage one wait, two tcgen05.mma (cta_group::2) per accumulator
//    and one commit to both blocks.  The leader's "full" barrier of a stage counts the converter
//    warps of both blocks and the bytes of both blocks' planes;
//  * epilogue (8 warps per block, two per TMEM lane quarter): reduces an accumulator in place
//    (tcgen05.ld / st) at its reduction points or writes the final residues, 64 database rows of
//    one query column per thread.  The accumulators' reduction points are
//    staggered by a quarter of the interval; the issuer goes on with the others while one is
//    reduced and catches up when it is back.
// Option SYNC (cooperative launch): the pairs start fetching the operands of their w-th tile only
// once every pair has issued all fetches of its (w-1)-th tile.  Keeping the waves together keeps
// the database slabs (shared by the moduli of a row tile) and the query planes (shared by the row
// tiles of a modulus) in L2 between their readers.  The moduli are taken in groups of mgrp (the
// modulus varies fastest inside a group, then the row tile, then the group): a wave of 76 pairs
// then reads mgrp moduli's planes and 76 / mgrp row tiles, which balances the two.
//
// Every wait is bounded by %globaltimer (a launch argument, default 2 s); on expiry the block
// records ICM_DEV_TIMEOUT in the device status word, stops issuing work in both blocks, waits
// (bounded) for its own MMAs and copies in flight, and frees its TMEM.  A test-only launch flag
// makes the query producers skip their copies, so that the MMA issuers' waits run out.
#include "icm_internal.h"
#include "ppmm_i8.h"

#include <algorithm>
#include <cuda.h>
#include <cuda_fp16.h>
#include <mutex>

namespace {

constexpr int BM = 128;                           // database rows of a pair's tile (N of the MMA)
constexpr int ROWS = BM / 2;                      // rows fetched and converted by one block
constexpr int QT = 128;                           // query columns of one block in an accumulator
constexpr int KS = 16;                            // K of a raw slab (an MMA step)
constexpr int R_BLK = ROWS * KS * 2;              // 2 KB: residues of one slab and modulus
constexpr int Q_TILE = QT * KS * 2;               // 4 KB: planes of one column group, modulus, slab
constexpr int RAW_SLOT = ROWS * KS * 8;           // 8 KB
constexpr uint32_t TMEM_COLS = 512;               // four accumulators of 128 columns
constexpr int FLUSH_K = 1024;                     // columns of K between reductions
constexpr int NCG = 4, WPG = 2, NCV = NCG * WPG;  // converter groups, warps per group
constexpr int ROWS_W = ROWS / WPG, ITEMS = ROWS_W / 16;   // rows of a converter warp, in items of 16
constexpr int NEP = 8;                            // epilogue warps: two per TMEM lane quarter
constexpr int EP_COLS = BM / 2;                   // accumulator columns (database rows) of one epilogue warp
static_assert(EP_COLS == 64, "store_residues");
constexpr uint64_t LAUNCH_COLS = 1024;            // columns of one launch: the scratch width

// Configuration of a launch: G column groups of 256 x NM moduli per tile, S operand stages of KH slabs,
// RS raw slots.  Shared memory: raw slots first (1024-byte aligned for the 128-byte swizzle), then the
// plane and residue stages, then the mbarriers.
template <int G_, int NM_, int S_, int RS_>
struct Cfg {
    static constexpr int G = G_, NM = NM_, S = S_, RS = RS_, NACC = G * NM;
    static constexpr int KH = 2;                      // slabs of a stage
    static constexpr int Q_MOD = KH * G * Q_TILE;     // planes of one modulus in a stage: [KH][G]
    static constexpr int Q_STAGE = NM * Q_MOD, R_STAGE = NM * KH * R_BLK;
    static constexpr int OFF_Q = RS * RAW_SLOT, OFF_R = OFF_Q + S * Q_STAGE, BARS = OFF_R + S * R_STAGE;
    static constexpr int SMEM = BARS + 1024 + 1024;   // barriers + slack to align the base to 1024
    static constexpr int W_EPI = NCV, W_RAW = NCV + NEP, W_QRY = W_RAW + 1, W_MMA = W_QRY + 1;
    static constexpr int NTHREADS = (W_MMA + 1) * 32;
    static constexpr uint32_t KST = KS * KH;          // K of a stage
    static constexpr uint32_t FLUSH = FLUSH_K / KST;  // stages between an accumulator's reductions
    static constexpr uint32_t STAGGER = FLUSH / 4;    // offset of the accumulators' reductions
    static constexpr uint32_t DEFER = S / 2;          // stages that an accumulator may lag while it is reduced
    static_assert(DEFER < STAGGER, "one accumulator lags at a time");
    static_assert(NACC * BM <= (int)TMEM_COLS, "accumulators");
    static_assert(SMEM <= 227 * 1024, "shared memory budget");
    static_assert(RS % NCG == 0 && (KH * S) % NCG == 0, "a slot always belongs to one converter group");
};

struct TcMod {
    int32_t wlo, whi;                 // centred 256^t mod m, t = 0..3 and 4..7
    uint32_t f0, hneg2;               // residue conversion: float bits F_0, f16x2 of its final offset
    float m, inv_m, k1;               // k1 = 1.5 2^23 - F_0 / m
};

struct TcArgs {
    CUtensorMap tmA[ICM_MAX_CHUNKS];  // per chunk: [L][M_c][K] u64, box 16 x 64, 128-byte swizzle
    CUtensorMap tmQ;                  // the launch's limbs of fp16 planes as rows of 2 KB (crt_f16_off)
    uint64_t q_row0, q_plane_rows;    // rows before the launch's column round in a plane; rows of a plane
    icm::ChunkTab tab;
    uint8_t *R;                       // [L][r][nch][sum M_c]
    uint64_t N, K, n0, nch;           // query columns; this launch's first column and its width
    uint32_t n_mod, n_limbs;
    uint32_t n_mt, mgrp;              // modulus tiles (of NM moduli), modulus tiles per group
    uint32_t slabs;                   // slabs of the planes (Kp / 16)
    uint64_t n_tiles;                 // L x row tiles x modulus tiles
    uint32_t *sync;                   // [0]: fetch arrivals (wave bound), [1]: a block gave up; zeroed per launch
    uint64_t wait_ns;                 // bound of every wait
    uint32_t canonical;               // database words are canonical residues modulo q, not in the storage form
    uint64_t q[ICM_MAX_LIMBS];
    uint32_t inject_stall;            // test only: the query producers never copy
    uint32_t zero;                    // 0
    TcMod md[ICM_MAX_MODULI];
};

// Device status word: ICM_DEV_TIMEOUT once any block gave up a bounded wait (read and cleared by
// icm_device_status).
__device__ uint32_t g_status;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t gtime() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(bar)), "r"(count) : "memory");
}
// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" :: "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}"
                 :: "r"(bar), "r"(bytes) : "memory");
}
// A probe that finds its phase incomplete suspends the thread until the phase completes, or for
// about this long.
constexpr uint32_t SUSPEND_NS = 100000;
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(SUSPEND_NS) : "memory");
    return ok != 0;
}
// Relaxed probe for the MMA issuer's operand waits: after a wait with the default acquire
// semantics, the next tcgen05.mma of the waiting thread is held until that thread's previous MMA
// has completed (one MMA per MMA latency instead of back to back; measured on GB300: 490 instead
// of 256 cycles for two M128 N256 K16 MMAs).  The operands need no acquire here: the converters
// publish their residues with fence.proxy.async before a release arrive, the query planes land
// through TMA completion, and the MMA is an async-proxy read ordered after the wait by
// tcgen05.fence::after_thread_sync.
__device__ __forceinline__ bool mbar_try_rlx(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.relaxed.cta.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity), "r"(SUSPEND_NS) : "memory");
    return ok != 0;
}
// Whether the phase of the given parity has completed, without waiting.
template <bool RLX = false>
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if (RLX)
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.relaxed.cta.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Shared memory address of this block's `addr` in block `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrive on a barrier of another block of the cluster (mapped address).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t mapped) {
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" :: "r"(mapped) : "memory");
}
// What a bounded wait needs besides its barrier.
struct WaitCtx {
    volatile int *abort_flag;         // this block's, in shared memory
    uint32_t *sync;                   // the launch's give-up word follows its wave counter; may be null
    uint64_t wait_ns;
};
// A wait ran out: both blocks of the pair stop issuing work.
__device__ __noinline__ void give_up(const WaitCtx &w) {
    *w.abort_flag = 1;
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], 1;"
                 :: "r"(map_rank(smem_u32(const_cast<int *>(w.abort_flag)), rank ^ 1u)) : "memory");
    atomicExch(&g_status, (uint32_t)ICM_DEV_TIMEOUT);
    if (w.sync) atomicExch(&w.sync[1], 1u);
}
template <bool RLX>
__device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, const WaitCtx &w) {
    const uint64_t t0 = gtime();
    for (;;) {
        if (RLX ? mbar_try_rlx(bar, parity) : mbar_try(bar, parity)) return true;
        if (*w.abort_flag) return false;
        if (gtime() - t0 > w.wait_ns) {
            give_up(w);
            return false;
        }
    }
}
// Bounded wait of a whole warp; false on timeout or when another thread of the pair has given up.
// RLX: relaxed probe (the MMA issuer's operand waits), else acquire.  Only the first probe is
// inline: the roles' loops share the instruction caches, and a loop that carries its slow paths
// ran at 16 cycles per instruction.
template <bool RLX = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const WaitCtx &w) {
    bool ok = RLX ? mbar_try_rlx(bar, parity) : mbar_try(bar, parity);
    if (!ok) ok = mbar_wait_slow<RLX>(bar, parity, w);
    return __all_sync(0xffffffffu, ok);
}
// Bounded wait that ignores the abort flag (drains this block's own copies and MMAs before it
// frees TMEM and exits); gives up at the %globaltimer deadline shared by a whole drain.
__device__ __forceinline__ void mbar_wait_until(uint64_t *bar, uint32_t parity, uint64_t deadline) {
    while (!mbar_try(smem_u32(bar), parity))
        if (gtime() > deadline) {
            atomicExch(&g_status, (uint32_t)ICM_DEV_TIMEOUT);
            return;
        }
}

// TMA tile load into this block's shared memory, completing on an mbarrier.
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int c0, int c1, int c2, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 :: "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
                 : "memory");
}
// The same for rows of the plane map, completing on a barrier of either block of the pair (mapped
// address `bar`).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int c0, int c1, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar) : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared memory matrix descriptor: start address >> 4 [0,14), leading byte offset >> 4 [16,30),
// stride byte offset >> 4 [32,46), version 1 [46,48), base offset 0, swizzle mode [61,64)
// (0: none).  K-major without swizzle: 8-row x 16-byte core matrices, the leading offset steps
// from k 0-7 to k 8-15, the stride offset from one group of 8 rows to the next.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// Instruction descriptor, kind::f16: D = f32 [4,6), A = B = f16 [7,10) [10,13), both K-major,
// N >> 3 [17,23), M >> 4 [24,29): M 256 query columns (128 per block), N 128 database rows (64 per
// block).
constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(BM >> 3) << 17) | ((uint32_t)((2 * QT) >> 4) << 24);

__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 :: "r"(d_tmem), "l"(a), "l"(b), "r"(IDESC), "r"(accumulate) : "memory");
}
// Commit this thread's MMAs to the barrier at the same offset in both blocks.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 :: "r"(bar), "h"((uint16_t)3) : "memory");
}

// W columns of 32-bit TMEM words per thread (lane quarter of the warp).  A load comes with its wait in
// one statement: the compiler may otherwise copy a destination register before the load has landed.
template <int W>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[W]);
template <int W>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[W]);
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}
template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                   "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                   "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr) : "memory");
}
template <>
__device__ __forceinline__ void tmem_st<32>(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
                 :: "r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
                   "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
                   "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
                   "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
                 : "memory");
}

__device__ __forceinline__ uint64_t pack2(uint32_t lo, uint32_t hi) { return (uint64_t)hi << 32 | lo; }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t dup2(float x) { return pack2(__float_as_uint(x), __float_as_uint(x)); }
constexpr float RINT = 12582912.0f;               // 1.5 2^23: adding it rounds to an integer

// Per-thread constants of the residue conversion modulo m.
struct ResMod {
    int wlo, whi, f0;
    uint32_t hneg2;
    uint64_t inv, k1, nm;
    __device__ __forceinline__ ResMod() {}
    __device__ __forceinline__ explicit ResMod(const TcMod &t)
        : wlo(t.wlo), whi(t.whi), f0((int)t.f0), hneg2(t.hneg2), inv(dup2(t.inv_m)), k1(dup2(t.k1)), nm(dup2(-t.m)) {}
};
// Residues modulo m of two balanced-digit storage words, as f16x2 bits.  The digits' sum
// s = sum_t d_t (256^t mod m), |s| < 2^17, is accumulated by dp4a onto the bits of the float
// F_0 = 2^23 + X with X = 0x30000 + L, so the bits are those of F_0 + s.  m divides F_0, so
// (F_0 + s) / m + (1.5 2^23 - F_0 / m) rounds s / m to an integer k (the sum's error, 2^16 2^-24 at
// most, moves the rounding by less than 1 / m), and F_0 + s - m k = F_0 + r is exact with
// |r| <= (m + 1) / 2 <= 128.  L is chosen with 0x6480 <= L < 0x6780, so the low half of the bits,
// L + r, is the f16 1024 + (L + r - 0x6400), and one f16x2 add leaves r exactly.  Two words take
// 4 dp4a, 3 packed fp32 operations, a permute and the add (9; the integer form with a
// multiply-high takes 11, all at half the fp32 rate).
__device__ __forceinline__ uint32_t res_pair(uint64_t z0, uint64_t z1, const ResMod &c) {
    const int v0 = __dp4a((int)(uint32_t)(z0 >> 32), c.whi, __dp4a((int)(uint32_t)z0, c.wlo, c.f0));
    const int v1 = __dp4a((int)(uint32_t)(z1 >> 32), c.whi, __dp4a((int)(uint32_t)z1, c.wlo, c.f0));
    const uint64_t f = pack2((uint32_t)v0, (uint32_t)v1);
    const uint64_t r = fma2(add2(fma2(f, c.inv, c.k1), dup2(-RINT)), c.nm, f);
    uint32_t out;
    asm("add.rn.f16x2 %0, %1, %2;" : "=r"(out) : "r"(__byte_perm((uint32_t)r, (uint32_t)(r >> 32), 0x5410)), "r"(c.hneg2));
    return out;
}

// Writes the first n (0..64) of a thread's 64 bytes to an address of any alignment: whole rows as 4-byte
// words with bytes at the edges.  (64 single bytes, each a 32-line store of the warp, took the epilogue
// 16,000 cycles per accumulator: 8 eyes against three chunks of odd sizes 20.8 -> 18.5 ms.)
__device__ __forceinline__ void store_residues(uint8_t *d, const uint32_t (&w)[16], uint32_t n) {
    if (n == 64) {
        const uint32_t head = (4u - (uint32_t)(reinterpret_cast<uintptr_t>(d) & 3)) & 3u;   // bytes before the first whole word
        uint32_t *q = reinterpret_cast<uint32_t *>(d + head);
#pragma unroll
        for (int i = 0; i < 15; ++i) q[i] = __funnelshift_r(w[i], w[i + 1], 8 * head);
        if (head == 0) {
            q[15] = w[15];
        } else {
            for (uint32_t i = 0; i < head; ++i) d[i] = (uint8_t)(w[0] >> (8 * i));
            for (uint32_t i = head; i < 4; ++i) d[60 + i] = (uint8_t)(w[15] >> (8 * i));
        }
    } else {
#pragma unroll
        for (int i = 0; i < 64; ++i)
            if ((uint32_t)i < n) d[i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
    }
}

template <class C>
struct __align__(8) Bars {
    // raw slots; operand stages (planes and residues; "full" is used in the leader only); per
    // accumulator: handed to the epilogue, handed back (leader only); MMAs drained
    uint64_t rawfull[C::RS], rawempty[C::RS], full[C::S], empty[C::S], accfull[C::NACC], accfree[C::NACC], done;
    uint32_t tmem;
    int abort_flag;
};

struct TileCoord {
    uint32_t l, c, mi0, nm;           // limb, chunk, first modulus, moduli of the tile
    uint64_t m0, M;
};
// tile -> (limb, modulus group, row tile, modulus tile of the group), the last fastest
template <int NM>
__device__ __forceinline__ TileCoord tile_coord(const TcArgs &p, uint64_t tile) {
    TileCoord t;
    const uint32_t mt_total = p.tab.mt0[p.tab.n];
    const uint64_t per_limb = (uint64_t)mt_total * p.n_mt;
    t.l = (uint32_t)(tile / per_limb);
    uint64_t tt = tile % per_limb;
    const uint32_t grp = (uint32_t)(tt / ((uint64_t)mt_total * p.mgrp));
    tt -= (uint64_t)grp * mt_total * p.mgrp;
    const uint32_t size = min(p.mgrp, p.n_mt - grp * p.mgrp);
    const uint32_t mtg = (uint32_t)(tt / size);
    t.mi0 = (grp * p.mgrp + (uint32_t)(tt % size)) * NM;
    t.nm = min((uint32_t)NM, p.n_mod - t.mi0);
    uint32_t c = 0;
    while (c + 1 < p.tab.n && mtg >= p.tab.mt0[c + 1]) ++c;
    t.c = c;
    t.M = p.tab.M[c];
    t.m0 = (uint64_t)(mtg - p.tab.mt0[c]) * BM;
    return t;
}
// Reduction points within a tile of nst stages: after stages STAGGER, 2 STAGGER, ... below nst, in turn
// of accumulators 3, 2, 1, 0 (each every FLUSH stages), and the final write of all after the last.
__device__ __forceinline__ uint32_t reduced_acc(uint32_t e) { return (4u - (e & 3u)) & 3u; }

// Wave bound (SYNC): wait until every block has issued all fetches of its (w-1)-th tile.  Each
// block's fetching threads (raw and query producers) add one to sync[0] per tile.
__device__ __noinline__ bool wave_wait(const uint32_t need, const WaitCtx &w) {
    const uint64_t t0 = gtime();
    bool ok = true;
    for (;;) {
        if (*(volatile uint32_t *)&w.sync[0] >= need) break;
        if (*w.abort_flag || *(volatile uint32_t *)&w.sync[1]) { ok = false; break; }
        if (gtime() - t0 > w.wait_ns) {
            give_up(w);
            ok = false;
            break;
        }
        __nanosleep(200);
    }
    return __all_sync(0xffffffffu, ok);
}

template <class C, bool SYNC>
__global__ void __launch_bounds__(C::NTHREADS, 1) k_crt_tc(const __grid_constant__ TcArgs p) {
    constexpr int G = C::G, NM = C::NM, KH = C::KH, S = C::S, RS = C::RS, NACC = C::NACC;
    using BR = Bars<C>;
    static_assert(sizeof(BR) <= 1024, "barrier block");
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    // the swizzle patterns are functions of shared-memory address bits: align the base to 1024 (the
    // same offset in both blocks of the pair)
    unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    unsigned char *sW = smem;                          // [RS][RAW_SLOT]
    unsigned char *sQ = smem + C::OFF_Q;               // [S][NM][KH][G][Q_TILE]
    unsigned char *sR = smem + C::OFF_R;               // [S][NM][KH][R_BLK]
    BR *bars = reinterpret_cast<BR *>(smem + C::BARS);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);        // uniform over the warp
    const WaitCtx wc{&bars->abort_flag, p.sync, p.wait_ns};
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    // barrier addresses (arrays of 8 bytes per slot)
    const uint32_t b_rawfull = smem_u32(bars->rawfull), b_rawempty = smem_u32(bars->rawempty);
    const uint32_t b_full = smem_u32(bars->full), b_empty = smem_u32(bars->empty);
    const uint32_t b_accfull = smem_u32(bars->accfull), b_accfree = smem_u32(bars->accfree);

    if (tid == 0) {
        for (int s = 0; s < RS; ++s) { mbar_init(&bars->rawfull[s], 1); mbar_init(&bars->rawempty[s], WPG); }
        for (int s = 0; s < S; ++s) {
            // full: the converter warps of the stage's slabs in both blocks + the leader's query producer
            mbar_init(&bars->full[s], 2 * KH * WPG + 1);
            mbar_init(&bars->empty[s], 1);              // the MMA issuer's commit
        }
        for (int a = 0; a < NACC; ++a) { mbar_init(&bars->accfull[a], 1); mbar_init(&bars->accfree[a], 2 * NEP); }
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
    cluster_sync();                                    // barriers of both blocks are initialised
    tc_fence_after();
    const uint32_t tmem = bars->tmem;

    const uint32_t nst = (uint32_t)((p.K + C::KST - 1) / C::KST);  // operand stages of a tile
    const uint32_t nk = nst * KH;                                  // slabs of a tile
    const uint64_t Mall = p.tab.row0[p.tab.n];
    const uint32_t t_first = blockIdx.x >> 1, t_step = gridDim.x >> 1;   // persistent tile sequence of the pair
    constexpr uint32_t FETCHERS = 2;

    if (warp < NCV) {
        // ------------------------------------------------------------------ converter warps
        // group grp converts the slabs g with g mod NCG = grp, so NCG slabs are converted at once;
        // each warp converts ROWS_W rows of its group's slabs.  item it: rows sub ROWS_W + 16 it +
        // 8 (lane >> 4) + (lane & 7); 16-byte chunks [4 cj, 4 cj + 4) of the swizzled 128-byte raw row
        // (k 8 cj .. 8 cj + 7) -> 16 bytes of residues; every quarter-warp covers 8 consecutive rows
        // with the same chunks (8 distinct bank groups)
        const uint32_t grp = (uint32_t)warp % NCG, sub = (uint32_t)warp / NCG;
        const uint32_t lrow0 = sub * ROWS_W + ((uint32_t)(lane >> 4) << 3) + (lane & 7);
        const uint32_t cj = (lane >> 3) & 1;
        const uint32_t rsw = lane & 7;                                   // = row mod 8
        const uint32_t a_off0 = cj * (ROWS * 16) + (lrow0 >> 3) * 128 + (lrow0 & 7) * 16;
        const uint32_t full0 = map_rank(b_full, 0);                      // the leader's "full" barriers
        // the group's next slab: index, raw slot and the parity of its phase, half of a stage, stage
        // slot and the parity of its phase; a slot and a half always belong to the same group
        uint64_t g = grp, g_end = 0;
        uint32_t rs = grp, rpar = 0, h = grp % KH, s = (grp / KH) % S, spar = 0;
        bool alive = true;
        for (uint64_t tile = t_first; alive && tile < p.n_tiles; tile += t_step) {
            const TileCoord tc = tile_coord<NM>(p, tile);
            g_end += nk;                                                 // the groups' turns continue across tiles
            ResMod mds[NM];                                              // constants of the tile's moduli
#pragma unroll
            for (int mu = 0; mu < NM; ++mu) mds[mu] = ResMod(p.md[min(tc.mi0 + mu, p.n_mod - 1)]);
            for (; g < g_end; g += NCG) {
                if (!mbar_wait(b_rawfull + rs * 8, rpar, wc)) { alive = false; break; }
                const unsigned char *r_s = sW + rs * RAW_SLOT + lrow0 * 128;
                ulonglong2 z[ITEMS][4];
#pragma unroll
                for (int it = 0; it < ITEMS; ++it)
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        z[it][c] = *reinterpret_cast<const ulonglong2 *>(r_s + it * 16 * 128 + (((cj * 4 + c) ^ rsw) << 4));
                if (p.canonical) {                                       // canonical residues: to the storage form
                    const uint64_t q = p.q[tc.l];
#pragma unroll
                    for (int it = 0; it < ITEMS; ++it)
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            z[it][c] = make_ulonglong2(to_digit_form(z[it][c].x, q), to_digit_form(z[it][c].y, q));
                }
#pragma unroll
                for (int mu = 0; mu < NM; ++mu) {
                    if (NM > 1 && mu >= (int)tc.nm) break;
                    const ResMod &md = mds[mu];
                    uint32_t w[ITEMS][4];
#pragma unroll
                    for (int it = 0; it < ITEMS; ++it)
#pragma unroll
                        for (int c = 0; c < 4; ++c) w[it][c] = res_pair(z[it][c].x, z[it][c].y, md);
                    if (mu == 0) {
                        // The raw slot goes back to the TMA (another proxy) only when every read of it has
                        // returned: the barrier's address is made to depend on all the values (p.zero is
                        // 0).  Program order is not enough: without it the arrival overtook the last reads.
                        uint32_t dep = 0;
#pragma unroll
                        for (int it = 0; it < ITEMS; ++it) dep |= w[it][0] | w[it][1] | w[it][2] | w[it][3];
                        dep &= p.zero;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(b_rawempty + rs * 8 + dep);
                        // the stage is free once every accumulator's MMAs that read it have completed
                        // (its first phase: the parity of the phase before passes at once)
                        if (!mbar_wait(b_empty + s * 8, spar ^ 1, wc)) { alive = false; break; }
                    }
#pragma unroll
                    for (int it = 0; it < ITEMS; ++it)
                        *reinterpret_cast<uint4 *>(sR + s * C::R_STAGE + (mu * KH + h) * R_BLK + a_off0 + it * 2 * 128) =
                            make_uint4(w[it][0], w[it][1], w[it][2], w[it][3]);
                }
                if (!alive) break;
                // residues written through the generic proxy are read by the tensor cores
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(full0 + s * 8);
                rs += NCG;
                if (rs >= (uint32_t)RS) { rs -= RS; rpar ^= 1; }
                s += NCG / KH;
                if (s >= (uint32_t)S) { s -= S; spar ^= 1; }
            }
        }
    } else if (warp < C::W_RAW) {
        // ------------------------------------------------------------------ epilogue warps
        const uint32_t qtr = (uint32_t)warp & 3;                          // TMEM lane quarter
        const uint32_t half = (uint32_t)(warp - C::W_EPI) >> 2;           // column half of the accumulator
        const uint32_t trow = qtr * 32 + lane;                            // query column of this thread in its group
        const uint32_t free0 = map_rank(b_accfree, 0);                    // the leader's hand-back barriers
        uint32_t ev = 0;                                                  // parities of accfull, one bit per accumulator
        bool alive = true;
        for (uint64_t tile = t_first; alive && tile < p.n_tiles; tile += t_step) {
            const TileCoord tc = tile_coord<NM>(p, tile);
            const uint32_t nacc = tc.nm * G;
            // the issuer's reduction points in stage order, then the final write of every accumulator
            const uint32_t n_red = (nst - 1) / C::STAGGER, n_ev = n_red + nacc;
            for (uint32_t e = 1; e <= n_ev; ++e) {
                const bool final = e > n_red;
                const uint32_t a = final ? e - n_red - 1 : reduced_acc(e);
                if (a >= nacc) continue;
                if (!mbar_wait(b_accfull + a * 8, (ev >> a) & 1, wc)) { alive = false; break; }
                ev ^= 1u << a;
                tc_fence_after();
                const uint32_t mi = tc.mi0 + a / G;
                const float fm = p.md[mi].m;
                const uint64_t inv2 = dup2(p.md[mi].inv_m), nm2 = dup2(-fm);
                const uint32_t tbase = tmem + ((qtr * 32) << 16) + a * BM + half * EP_COLS;
                // column of the launch and first row of this thread's part
                const uint64_t col = (uint64_t)rank * (QT * G) + (a % G) * QT + trow;
                const uint64_t row0 = tc.m0 + half * EP_COLS;
                const bool col_ok = col < p.nch && p.n0 + col < p.N;
                uint8_t *dst = p.R + ((size_t)tc.l * p.n_mod + mi) * p.nch * Mall + (col_ok ? col : 0) * Mall +
                               p.tab.row0[tc.c] + row0;
                // x - m round(x / m): the fma adds 1.5 2^23 to the exact x / m estimate and rounds
                // once, which rounds it to an integer (|x / m| < 2^22); the result is an exact
                // integer in (-m, m)
                auto reduce = [&](auto &v) {
#pragma unroll
                    for (int i = 0; i < (int)(sizeof(v) / 4); i += 2) {
                        const uint64_t x = pack2(v[i], v[i + 1]);
                        const uint64_t r = fma2(add2(fma2(x, inv2, dup2(RINT)), dup2(-RINT)), nm2, x);
                        v[i] = (uint32_t)r;
                        v[i + 1] = (uint32_t)(r >> 32);
                    }
                };
                if (!final) {
#pragma unroll
                    for (uint32_t c = 0; c < EP_COLS; c += 32) {
                        uint32_t v[32];
                        tmem_ld<32>(tbase + c, v);
                        reduce(v);
                        tmem_st<32>(tbase + c, v);
                    }
                    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                } else {
                    // residues in [0, m) of 16 database rows as bytes (the float's low mantissa bits, r + 2^23)
                    auto chunk = [&](uint32_t c, uint32_t *w) {
                        uint32_t va[16];
                        tmem_ld<16>(tbase + c * 16, va);
                        reduce(va);
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const float r = __uint_as_float(va[i]);
                            va[i] = __float_as_uint((r < 0.0f ? r + fm : r) + 8388608.0f);
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            w[i] = __byte_perm(__byte_perm(va[4 * i], va[4 * i + 1], 0x0040),
                                               __byte_perm(va[4 * i + 2], va[4 * i + 3], 0x0040), 0x5410);
                    };
                    const uint32_t rows = col_ok && row0 < tc.M ? (uint32_t)min((uint64_t)EP_COLS, tc.M - row0) : 0u;
                    if (((reinterpret_cast<uintptr_t>(p.R) | Mall | p.tab.row0[tc.c]) & 15) == 0) {
                        // every column's rows start on 16 bytes
#pragma unroll 1
                        for (uint32_t c = 0; c < EP_COLS / 16; ++c) {
                            uint32_t w[4];
                            chunk(c, w);
                            if (rows >= (c + 1) * 16) {
                                *reinterpret_cast<uint4 *>(dst + c * 16) = make_uint4(w[0], w[1], w[2], w[3]);
                            } else {
#pragma unroll
                                for (uint32_t i = 0; i < 16; ++i)
                                    if (c * 16 + i < rows) dst[c * 16 + i] = (uint8_t)(w[i >> 2] >> (8 * (i & 3)));
                            }
                            __syncwarp();
                        }
                    } else {
                        uint32_t w[EP_COLS / 4];
#pragma unroll
                        for (uint32_t c = 0; c < EP_COLS / 16; ++c) chunk(c, w + 4 * c);
                        store_residues(dst, w, rows);
                        __syncwarp();
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(free0 + a * 8);
            }
        }
    } else if (warp < C::W_QRY) {
        // ------------------------------------------------------------------ raw database producer
        // The producers' and the issuer's loops run in whole warps on uniform values, with one elected
        // lane for the copies and MMAs: a copy issued inside a lane-dependent branch costs 51 cycles,
        // an elected one 17.
        const bool el = elect_one();
        uint64_t g = 0;                                                   // slabs issued
        uint32_t rs = 0, rpar = 0, w = 0;                                 // slot, parity of its phase
        for (uint64_t tile = t_first; tile < p.n_tiles; tile += t_step, ++w) {
            const TileCoord tc = tile_coord<NM>(p, tile);
            if (SYNC && w && !wave_wait(FETCHERS * gridDim.x * w, wc)) break;
            const int row = (int)(tc.m0 + rank * ROWS);
            const CUtensorMap *map = &p.tmA[tc.c];
            bool alive = true;
            for (uint32_t kt = 0; kt < nk; ++kt, ++g) {
                if (!mbar_wait(b_rawempty + rs * 8, rpar ^ 1, wc)) { alive = false; break; }
                if (el) {
                    mbar_expect_tx(b_rawfull + rs * 8, RAW_SLOT);
                    tma_load_3d(smem_u32(sW) + rs * RAW_SLOT, map, (int)(kt * KS), row, (int)tc.l, b_rawfull + rs * 8);
                }
                __syncwarp();
                if (++rs == (uint32_t)RS) { rs = 0; rpar ^= 1; }
            }
            if (!alive) break;
            if (SYNC && el) atomicAdd(&p.sync[0], 1u);
            __syncwarp();
        }
        // every load issued by this warp has landed before the block exits
        const uint64_t deadline = gtime() + p.wait_ns;
        for (uint64_t i = g > (uint64_t)RS ? g - RS : 0; i < g; ++i)
            mbar_wait_until(&bars->rawfull[i % RS], (uint32_t)((i / RS) & 1), deadline);
    } else if (warp < C::W_MMA) {
        // ------------------------------------------------------------------ query plane producer
        const bool el = elect_one();
        const uint32_t full0 = map_rank(b_full, 0);
        uint64_t n = 0, n0 = 0;                                          // next stage, first stage of the tile
        uint32_t s = 0, spar = 0, w = 0;
        for (uint64_t tile = t_first; tile < p.n_tiles && !p.inject_stall; tile += t_step, ++w, n0 += nst) {
            const TileCoord tc = tile_coord<NM>(p, tile);
            if (SYNC && w && !wave_wait(FETCHERS * gridDim.x * w, wc)) break;
            // a slab of this block is 2 G rows of 2 KB; the blocks' halves of a round are p.slabs apart
            // (a tile short of moduli repeats its last one, so that the bytes of a stage are always the same)
            const uint32_t row0 = (uint32_t)(((uint64_t)tc.l * p.n_mod + tc.mi0) * p.q_plane_rows + p.q_row0 +
                                             (uint64_t)rank * p.slabs * (2 * G));
            const uint32_t plane_rows = (uint32_t)p.q_plane_rows;
            bool alive = true;
            for (; n < n0 + nst; ++n) {
                // the stage is free once every accumulator's MMAs that read it have completed
                if (!mbar_wait(b_empty + s * 8, spar ^ 1, wc)) { alive = false; break; }
                if (el) {
                    // the leader announces the bytes of both blocks and all moduli
                    if (rank == 0) mbar_expect_tx(b_full + s * 8, 2 * C::Q_STAGE);
#pragma unroll
                    for (int mu = 0; mu < NM; ++mu)
                        tma_load_2d_pair(smem_u32(sQ) + s * C::Q_STAGE + mu * C::Q_MOD, &p.tmQ, 0,
                                         (int)(row0 + min((uint32_t)mu, tc.nm - 1) * plane_rows + (uint32_t)(n - n0) * (2 * G * KH)),
                                         full0 + s * 8);
                }
                __syncwarp();
                if (++s == (uint32_t)S) { s = 0; spar ^= 1; }
            }
            if (!alive) break;
            if (SYNC && el) atomicAdd(&p.sync[0], 1u);
            __syncwarp();
        }
        // every copy issued by this warp has been consumed before the block exits (after a give-up
        // the MMAs may not come: one deadline bounds the whole drain)
        const uint64_t deadline = gtime() + p.wait_ns;
        for (uint64_t i = n > (uint64_t)S ? n - S : 0; i < n; ++i)
            mbar_wait_until(&bars->empty[i % S], (uint32_t)((i / S) & 1), deadline);
    } else if (rank == 0) {
        // ------------------------------------------------------------------ MMA issuer (leader)
        // Descriptors of stage 0; stage s adds s Q_STAGE / 16 and s R_STAGE / 16 to the
        // start-address fields, the next slab of a stage G Q_TILE / 16 and R_BLK / 16.
        const bool el = elect_one();
        const uint64_t qdesc0 = sdesc(smem_u32(sQ), QT * 16, 128);
        const uint64_t rdesc0 = sdesc(smem_u32(sR), ROWS * 16, 128);
        auto issue = [&](uint32_t a, uint32_t s, bool first) {
            const uint64_t qd = qdesc0 + (uint64_t)(s * (C::Q_STAGE >> 4) + ((a / G * C::Q_MOD + a % G * Q_TILE) >> 4));
            const uint64_t rd = rdesc0 + (uint64_t)(s * (C::R_STAGE >> 4) + ((a / G * KH * R_BLK) >> 4));
#pragma unroll
            for (int h = 0; h < KH; ++h)
                umma(tmem + a * BM, qd + (uint64_t)(h * ((G * Q_TILE) >> 4)), rd + (uint64_t)(h * (R_BLK >> 4)),
                     first && h == 0 ? 0u : 1u);
        };
        uint32_t s = 0, par = 0;                                         // stage slot, parity of its phase
        uint32_t pend = 0, fpar = 0;                                     // accumulators at the epilogue; parities of accfree
        bool alive = true;
        for (uint64_t tile = t_first; alive && tile < p.n_tiles; tile += t_step) {
            const uint32_t nacc = NM == 1 ? NACC : tile_coord<NM>(p, tile).nm * G;
            // the tile's first stage: each accumulator once its last tile's residues are written
            if (!mbar_wait<true>(b_full + s * 8, par, wc)) break;
#pragma unroll
            for (uint32_t a = 0; a < (uint32_t)NACC; ++a) {
                if (a < nacc && alive) {
                    if ((pend >> a) & 1) {
                        alive = mbar_wait(b_accfree + a * 8, (fpar >> a) & 1, wc);
                        fpar ^= 1u << a;
                        pend &= ~(1u << a);
                    }
                    tc_fence_after();
                    if (el && alive) issue(a, s, true);
                    __syncwarp();
                }
            }
            if (!alive) break;
            // While accumulator `lag` is being reduced, the others go on; its MMAs of the `n_lag` stages
            // since then follow when it is back, and only then are those stages released.  The loop
            // holds little besides the MMAs and a commit: it has 71 cycles per MMA.
            uint32_t lag = NACC, n_lag = 0;
            for (uint32_t st = 1;; ++st) {
                if (lag == (uint32_t)NACC) {
                    if (el) umma_commit(b_empty + s * 8);
                    __syncwarp();
                } else {
                    if (++n_lag >= C::DEFER || st == nst ||
                        __all_sync(0xffffffffu, mbar_test(b_accfree + lag * 8, (fpar >> lag) & 1))) {
                        if (!mbar_wait(b_accfree + lag * 8, (fpar >> lag) & 1, wc)) { alive = false; break; }
                        fpar ^= 1u << lag;
                        tc_fence_after();
#pragma unroll 1
                        for (uint32_t back = n_lag; back-- > 0;) {
                            const uint32_t ks = s >= back ? s - back : s + S - back;
                            if (el) {
                                issue(lag, ks, false);
                                umma_commit(b_empty + ks * 8);
                            }
                            __syncwarp();
                        }
                        lag = NACC;
                    }
                }
                // st stages are issued (all but the lagging accumulator's)
                if (st == nst) break;
                if (st % C::STAGGER == 0) {
                    const uint32_t a = reduced_acc(st / C::STAGGER);
                    if (a < nacc) {
                        if (el) umma_commit(b_accfull + a * 8);
                        __syncwarp();
                        lag = a;
                        n_lag = 0;
                    }
                }
                if (++s == S) { s = 0; par ^= 1u; }
                if (!mbar_wait<true>(b_full + s * 8, par, wc)) { alive = false; break; }
                tc_fence_after();
                if (el) {
#pragma unroll
                    for (uint32_t a = 0; a < (uint32_t)NACC; ++a)
                        if ((NM == 1 || a < nacc) && a != lag) issue(a, s, false);
                }
                __syncwarp();
            }
            if (!alive) break;
            // the tile's sums go to the epilogue
            for (uint32_t a = 0; a < nacc; ++a) {
                if (el) umma_commit(b_accfull + a * 8);
                __syncwarp();
                pend |= 1u << a;
            }
            if (++s == S) { s = 0; par ^= 1u; }
        }
        // every MMA issued by this warp has completed before TMEM is freed
        if (el) umma_commit(smem_u32(&bars->done));
        __syncwarp();
        mbar_wait_until(&bars->done, 0, gtime() + p.wait_ns);
    }
    tc_fence_before();
    __syncthreads();
    // the commits' arrivals in the other block have landed before either block exits
    if (rank == 1 && tid == 0) mbar_wait_until(&bars->done, 0, gtime() + p.wait_ns);
    __syncwarp();
    cluster_sync();                                    // the pair's MMAs and remote arrivals are done
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(TMEM_COLS) : "memory");
}

#include "ppmm_dig_tc.cuh"

// ---------------------------------------------------------------- host side

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link against libcuda).
EncodeTiled encode_fn() {
    static std::once_flag once;
    static EncodeTiled fn = nullptr;
    std::call_once(once, [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiled>(f);
    });
    return fn;
}

// Configurations by column groups of the launch (256 columns each): the accumulators a launch does
// not need for columns take further moduli of the same row tile.
using Cfg4 = Cfg<4, 1, 4, 8>;
using Cfg3 = Cfg<3, 1, 4, 12>;
using Cfg2 = Cfg<2, 2, 4, 8>;
using Cfg1 = Cfg<1, 3, 4, 8>;

template <class C, bool SYNC>
cudaError_t launch_cfg(const TcArgs &a, int sms, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3(2 * (unsigned)std::min<uint64_t>(a.n_tiles, (uint64_t)(sms / 2)));
    cfg.blockDim = dim3(C::NTHREADS);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    // every block must be resident at once for the wave bound: a cooperative launch fails instead
    // of stalling
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = SYNC ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k_crt_tc<C, SYNC>, a);
}

template <class C>
cudaError_t set_attr() {
    cudaError_t e = cudaFuncSetAttribute(k_crt_tc<C, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_crt_tc<C, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    return e;
}

template <class C>
cudaError_t run_cfg(TcArgs &a, bool sync, uint32_t mgrp, int sms, cudaStream_t st) {
    a.n_mt = (a.n_mod + C::NM - 1) / C::NM;
    a.mgrp = std::max(1u, std::min(a.n_mt, mgrp));
    a.n_tiles = (uint64_t)a.n_limbs * a.tab.mt0[a.tab.n] * a.n_mt;
    if (a.n_tiles == 0) return cudaSuccess;
    return sync ? launch_cfg<C, true>(a, sms, st) : launch_cfg<C, false>(a, sms, st);
}

}  // namespace

namespace icm {

cudaError_t crt_tc_set_attributes() {
    cudaError_t e = set_attr<Cfg4>();
    if (e == cudaSuccess) e = set_attr<Cfg3>();
    if (e == cudaSuccess) e = set_attr<Cfg2>();
    if (e == cudaSuccess) e = set_attr<Cfg1>();
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_dig_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SMEM);
    return e;
}

// Deepest product of the digit form: the carries out of the top digit are summed in fp32.  An interval of 960
// products adds at most 4,082 to the sum (top digits of weights below 2^59 in magnitude are at most 8:
// (960 128 8 + 61,690) / 256), so the 2,185 intervals of 2^18 words stay below 2^24 (8.92e6); 493,200 words would too.
constexpr uint64_t DIG_MAX_K = 1ull << 18;

// The digit form takes the columns that would leave the last group of 256 nearly empty, where its planes
// fit the residue planes' place in the operand (so that buffer sizes do not depend on the choice): up to
// n_mod / 8 groups of 32 columns, 2 for 60-bit primes.  One pass of a row tile per group costs 2,048 cycles
// per 16 words and 256 rows whatever the rest.  Measured for 8,192 rows and 8 limbs (ms): digits 3.6 per
// group; residues 13.2, 19.9, 33.4, 40.3 for one to four groups of 256.  So one group of 32 always
// goes to the digits, two where the last group of 256 would be the first or third of its launch.
// Past residue columns they take a further launch, one pass of K (0.85 ms at K = 20,480) whatever the rows, which
// a database of few row tiles does not repay.  9 eyes against N_db + 630 rows (ms; all columns as residues on
// mma.sync in brackets): N_db = 2^11 on two limbs 2.00 (1.82), on three 2.30 (2.93); 2^12 on two 2.58 (3.24);
// 2^10 on two, as residues here, 1.14 (1.49).  A database has at least N_db rows.
uint32_t dig_cols(uint32_t n_mod, uint32_t n_limbs, uint32_t n_db, uint64_t N, uint64_t K) {
    const uint32_t rem = (uint32_t)(N % 256), g = (rem + 31) / 32;
    const bool pays = g == 1 || (g == 2 && (N / 256) % 2 == 0);
    const bool rows = N < 256 || (uint64_t)n_limbs * n_db >= 6144;
    return pays && rows && g * 8 <= n_mod && crt_tc_supported(K) && K <= DIG_MAX_K ? rem : 0;
}

cudaError_t launch_dig_planes(const I8Consts &k, const uint64_t *op, uint64_t n_op, void *planes, uint64_t N, uint64_t K,
                              uint64_t Kp, cudaStream_t st) {
    if (reinterpret_cast<uintptr_t>(planes) % 16) return cudaErrorInvalidValue;
    DigPlanesArgs a{};
    a.op = op; a.planes = reinterpret_cast<unsigned char *>(planes);
    a.n_op = n_op; a.N = N; a.K = K; a.Kp = Kp; a.groups = (uint32_t)((N + 31) / 32);
    for (uint32_t l = 0; l < k.n_limbs; ++l) {
        a.q[l] = k.q[l];
        for (int t = 0; t < 8; ++t) { a.w[l][t] = k.pw8[l][t]; a.ws[l][t] = k.pw8s[l][t]; }
    }
    const uint64_t warps = Kp / 8 * a.groups * 8;
    k_dig_planes<<<dim3((unsigned)std::min<uint64_t>((warps + 7) / 8, 152u * 16u), k.n_limbs), 256, 0, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_ppmm_dig(const I8Consts &k, const ChunkTab &tab, const void *Bp, uint64_t col0, uint64_t N, uint64_t K,
                            uint64_t Kp, cudaStream_t st) {
    if (tab.row0[tab.n] == 0 || N == 0) return cudaSuccess;
    if (!crt_tc_aligned(tab) || reinterpret_cast<uintptr_t>(Bp) % 16) return cudaErrorInvalidValue;
    EncodeTiled enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    static_assert(sizeof(DigArgs) <= 32000, "kernel parameter space");
    DigArgs a{};
    const cuuint32_t estr[3] = {1, 1, 1};
    for (uint32_t c = 0; c < tab.n; ++c) {
        const cuuint64_t M = tab.M[c] ? tab.M[c] : 1;
        const cuuint64_t dims[3] = {K, M, k.n_limbs}, strides[2] = {K * 8, M * K * 8};
        const cuuint32_t box[3] = {16, DG_ROWS, 1};
        if (enc(&a.tmA[c], CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<uint64_t *>(tab.A[c]), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        a.t0[c + 1] = a.t0[c] + (uint32_t)((tab.M[c] + DG_TILE - 1) / DG_TILE);
    }
    a.groups = (uint32_t)((N + 31) / 32);
    const cuuint64_t dims[2] = {256, (cuuint64_t)k.n_limbs * a.groups * 2 * Kp}, strides[1] = {2048};
    const cuuint32_t box[2] = {256, DG_WORDS};
    if (enc(&a.tmB, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void *>(Bp), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    a.tab = tab;
    a.N = N; a.K = K; a.Kp = Kp; a.n_limbs = k.n_limbs; a.col0 = col0; a.n_out = tab.n_out ? tab.n_out : N;
    a.n_tiles = (uint64_t)k.n_limbs * a.t0[tab.n] * a.groups;
    a.wait_ns = k.tc_wait_ns ? k.tc_wait_ns : 2000000000ull;
    a.inject_stall = k.tc_inject_stall;
    for (uint32_t l = 0; l < k.n_limbs; ++l) {
        a.q[l] = k.q[l]; a.r64[l] = k.r64[l]; a.p32[l] = k.pw8[l][4]; a.p32s[l] = k.pw8s[l][4];
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3(2 * (unsigned)std::min<uint64_t>(a.n_tiles, (uint64_t)(sms / 2)));
    cfg.blockDim = dim3(DG_THREADS);
    cfg.dynamicSmemBytes = DG_SMEM;
    cfg.stream = st;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_dig_tc, a);
}

// The tcgen05 path needs an even K and 16-byte aligned chunks (tensor-map base addresses and row
// strides are multiples of 16 bytes); the caller uses the mma.sync kernel otherwise.
bool crt_tc_supported(uint64_t K) { return K > 0 && K % 2 == 0; }
bool crt_tc_aligned(const ChunkTab &tab) {
    for (uint32_t c = 0; c < tab.n; ++c)
        if (reinterpret_cast<uintptr_t>(tab.A[c]) % 16) return false;
    return true;
}

uint32_t device_status(bool clear) {
    uint32_t v = 0;
    if (cudaMemcpyFromSymbol(&v, g_status, sizeof(v)) != cudaSuccess) return 0xFFFFFFFFu;
    if (clear && v) {
        const uint32_t z = 0;
        cudaMemcpyToSymbol(g_status, &z, sizeof(z));
    }
    return v;
}

cudaError_t launch_ppmm_crt_tc(const I8Consts &k, const ChunkTab &tab, const void *Bp, uint64_t N, uint64_t K,
                               uint64_t Kp, void *scratch, int variant, cudaStream_t st) {
    const uint64_t Mall = tab.row0[tab.n];
    if (Mall == 0 || N == 0) return cudaSuccess;
    if (!crt_tc_supported(K) || Kp % KS || !crt_tc_variant(variant)) return cudaErrorInvalidValue;
    EncodeTiled enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);

    static_assert(sizeof(TcArgs) <= 32000, "kernel parameter space");
    TcArgs a{};
    // database chunks: [L][M_c][K] u64, box 16 words x 64 rows x 1 limb
    for (uint32_t c = 0; c < tab.n; ++c) {
        const cuuint64_t M = tab.M[c] ? tab.M[c] : 1;
        const cuuint64_t dims[3] = {K, M, k.n_limbs};
        const cuuint64_t strides[2] = {K * 8, M * K * 8};
        const cuuint32_t box[3] = {KS, ROWS, 1}, estr[3] = {1, 1, 1};
        if (enc(&a.tmA[c], CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, const_cast<uint64_t *>(tab.A[c]), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    // 16-byte aligned for the TMA loads
    if (reinterpret_cast<uintptr_t>(Bp) % 16) return cudaErrorInvalidValue;
    a.q_plane_rows = crt_f16_ncols(N) * Kp * 2 / 2048;
    a.slabs = (uint32_t)(Kp / KS);
    a.tab = tab;
    a.R = reinterpret_cast<uint8_t *>(scratch);
    // wave counter and give-up word after the residue scratch (crt_scratch_bytes reserves them)
    a.sync = reinterpret_cast<uint32_t *>(reinterpret_cast<char *>(scratch) +
                                          crt_scratch_main_bytes(k.n_limbs, k.n_mod, N, Mall));
    a.N = N; a.K = K;
    a.n_mod = k.n_mod;
    a.n_limbs = k.n_limbs;
    a.wait_ns = k.tc_wait_ns ? k.tc_wait_ns : 2000000000ull;
    a.inject_stall = k.tc_inject_stall;
    a.canonical = tab.a_digits ? 0u : 1u;
    for (uint32_t l = 0; l < k.n_limbs; ++l) a.q[l] = k.q[l];
    for (uint32_t i = 0; i < k.n_mod; ++i) {
        const uint32_t m = (uint32_t)k.mod[i];
        uint32_t L = 0x6480;                                             // m <= 255 divides F_0 for some L < 0x6780
        while ((0x830000u + L) % m) ++L;
        const uint32_t hb = 0xE400u | (L - 0x6400u);                     // f16 bits of -(1024 + L - 0x6400)
        a.md[i] = TcMod{k.wlo[i], k.whi[i], 0x4B030000u + L, hb | (hb << 16), (float)m, k.inv_m[i],
                        12582912.0f - (float)((0x830000u + L) / m)};
    }
    // one launch and one combine per 1,024 columns
    for (uint64_t n0 = 0; n0 < N; n0 += LAUNCH_COLS) {
        const uint64_t nch = std::min<uint64_t>(LAUNCH_COLS, N - n0);
        const cuuint32_t G = (cuuint32_t)((nch + 255) / 256);
        // query planes: tiled fp16 blocks (crt_f16_off) as rows of 2 KB, one box per stage and modulus
        const cuuint64_t dims[2] = {256, (cuuint64_t)k.n_limbs * k.n_mod * a.q_plane_rows}, strides[1] = {2048};
        const cuuint32_t box[2] = {256, 2 * G * Cfg4::KH}, estr[2] = {1, 1};
        if (enc(&a.tmQ, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<void *>(Bp), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        a.n0 = n0; a.nch = nch;
        a.q_row0 = n0 * Kp * 2 / 2048;
        cudaError_t e = cudaMemsetAsync(a.sync, 0, 2 * sizeof(uint32_t), st);
        if (e != cudaSuccess) return e;
        const bool sync = variant != 1;
        const uint32_t mgrp = variant == 3 ? ICM_MAX_MODULI : 6;
        if (G == 4) e = run_cfg<Cfg4>(a, sync, mgrp, sms, st);
        else if (G == 3) e = run_cfg<Cfg3>(a, sync, mgrp, sms, st);
        else if (G == 2) e = run_cfg<Cfg2>(a, sync, mgrp, sms, st);
        else e = run_cfg<Cfg1>(a, sync, mgrp, sms, st);
        if (e != cudaSuccess) return e;
        e = launch_crt_combine(k, tab, scratch, N, n0, nch, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace icm
