// Score passes on the 5th-generation tensor cores (tcgen05 + TMEM + TMA), sm_103a.
//
// Both passes contract the receiver query Q_s = [(r, h) rows x d] of one KV group
// s = (l, g) with that group's keys K_s = [positions x d] (App. C.1: a_{l,h,r,t} is the
// softmax over t of scale * <q, k>).  Operands are K-major bf16 tiles in the 128-byte
// swizzled layout, staged by TMA; one thread issues tcgen05.mma (fp32 accumulation in TMEM);
// the epilogue warps read TMEM with tcgen05.ld.  A paged sender cache (pages of at least 8 rows) is
// read by pass 1 page by page, and the tiles it has staged go on, by TMA stores out of the ring,
// into a contiguous copy that pass 2 reads: pass 2's tiles of every fourth position would need a
// load for every four rows (at least 144 us for the loads alone of qwen8b in 16-position pages,
// with four issuing warps).  Shorter pages are copied by k_depage first.
//
//   k_stats_tc  pass 1, D = Q_s K_tile^T: TMEM lane = row (r, h), column = position.
//               Each epilogue thread owns one row and one quarter of a tile's positions and keeps
//               the sum of exp2 over a chunk of positions.  The query tokens' own keys, where a
//               call has them, are further tiles of the last chunk under a causal mask.
//   k_accum_tc  pass 2, D = K_tile Q_s^T (+ one more K-step of ones x the rows' offset terms,
//               so TMEM holds z - (offset - centre) / scale, centre a whole number): TMEM lane = position, column = row (r, h).
//               A block of positions is four tiles: tile j holds every fourth position from j on,
//               so a thread owns four neighbouring positions, one of each tile.  exp2 of its
//               logits (a / G), the head mean b and the sums over tokens stay in registers; Pool
//               over positions needs the neighbouring lanes' prefix and suffix maxima only.  A
//               block's four lane quarters cover 128 positions each, 120 of them outputs (480 a
//               block).
//   k_narrow_tc pass 2 of short senders and of few blocks: a position a lane, 104 outputs a block.
//
// Rows: a group's m * G query rows, padded to 128, are processed in row chunks of up to 512
// (pass 1) or 256 rows (pass 2) whose Q fits in shared memory; a row chunk is the outermost part
// of a work unit, and the grid is a multiple of the row-chunk count, so that the CTAs of
// different row chunks walk the same K tiles at the same time and all but the first read them
// from L2.
//
// Warp roles (640 threads, one CTA per SM, persistent over a contiguous range of work
// units): warp 0 producer, warps 1 and 2 MMA issuers (warp 1 owns TMEM), warp 3 pass 1's stores of
// staged pages and pass 2's sums, warps 4-19 epilogue (warp w reads TMEM lanes 32*(w%4)..+31; the
// four warps of a lane quarter share a buffer's columns).  K tiles flow through a ring of smem
// stages; TMEM holds a ring of four 128-column accumulator buffers, each drained by all sixteen
// epilogue warps: the MMA runs up to four buffers ahead.  Two issuers, because one thread that
// waits, fences and commits for every tile issues a 128 x 128 x 16 step in 76.5 cycles and two in
// 64.1, the tensor core's own rate.
// Every mbarrier wait is bounded (1 s); on a timeout the kernel records kErrTimeout, drains
// its copies and MMAs, frees TMEM and returns.
#include <algorithm>
#include <atomic>
#include <cfloat>
#include <cstdint>
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>
#include <memory>
#include <mutex>
#include <type_traits>
#include <vector>

#include "cb_internal.cuh"
#include "cb_sm100.cuh"

namespace cbk {
namespace tc {   // (not anonymous: the parts of this file, below, share these types)

constexpr int kWarpsTc = 20;                // 0 TMA, 1 and 2 MMA, 3 page stores (pass 1) or sums (pass 2), 4..19 epilogue
constexpr int kThreadsTc = kWarpsTc * 32;
constexpr int kEpiWarps = 16;
constexpr int kEpi0 = 4;                    // first epilogue warp (TMEM lane quarter = warp % 4)
constexpr int kMaxStages = 8;
constexpr int kTileRows = 128;          // K rows per tile
constexpr int kMinPageShift = 3;        // shortest pages pass 1 reads itself: 8 rows, one swizzle atom
constexpr int kChunk1 = kStatsChunkTc;  // pass-1 positions per chunk, or twice as many (stats_chunk)
constexpr int kRowHalf = 128;           // query rows of one accumulator buffer
constexpr int kHalves1 = 4, kHalves2 = 2;        // most 128-row halves of a row chunk (pass 1, pass 2)
constexpr int kMargin = 4;              // pass-2 positions before/after a lane quarter's outputs
constexpr float kRaise = 8.f;           // pass 1, second run: a logit this far (log2 domain) above a row's offset raises it
constexpr int64_t kLongChunkUnits = 1024;  // pass-1 units from which chunks are twice as long
constexpr int kOutW = 128 - 2 * kMargin;         // 120 output positions per pass-2 lane quarter
constexpr int kOut2 = 4 * kOutW;                 // 480 output positions per pass-2 block
constexpr int kMarginN = 3, kOutNW = 32 - 2 * kMarginN, kOutN = 4 * kOutNW;   // the same of k_narrow_tc: 3, 26, 104
constexpr int64_t kNarrowUnits = 33;             // pass-2 units up to which blocks are of one tile (narrow_blocks)
constexpr uint32_t kTmemCols = 512;
constexpr uint64_t kWaitNs = 1000000000ull;      // 1 s per wait
constexpr uint32_t kPollNs = 1000000u;           // longest suspension of one poll (woken at completion)
constexpr int kMaxTcSenders = 32;         // their tensor maps fill most of the 32,764 bytes of kernel parameters

// Rows up to which a sender's last half's columns go to the warps in eights (pass 2; for G = 1 and d = 128,
// all halves'), and the most halves of such a sender: one half of ten gains less than the code
// for it costs the others (12 layers, T = 6001, 1200 rows: 231 against 225 us).
constexpr int kFewRows = 64, kFewHalves = 4;

struct TcMaps {
    CUtensorMap k[3];     // pass 1: k[0] = 4D {d, T, Hkv, nL}, box {64, 128, 1, 1}; k[1] the same over the
                          // query tokens' own keys {d, m, Hkv, nL} (senders that have them).  Of a paged
                          // sender k[0] = 5D {d, rows of a page, pages, Hkv, nL}, box {64, min(rows, 128), 1, 1, 1},
                          // and k[2] = the copy, 4D like a strided sender's.
                          // pass 2: k[0] = 5D {d, T / 4, 4, Hkv, nL} (position 4 i + j at (i, j)), box
                          // {64, 32, 1, 1, 1}; k[1] = 4D as in pass 1 with every fourth of 128 positions in its box (the
                          // 5D tensor lacks the last T mod 4 positions), or of a narrow sender 32 positions;
                          // k[2] = E, the offset terms, 3D {16, R_pad, nS}, box {16, q_rows, 1}, 32-byte swizzle
    CUtensorMap q;        // 4D {d, Hq, m, nL}, box {64, G, q_rows / G, 1}
};

struct TcSender {
    float2* stats;        // this sender's pass-1 partials [nS][n_chunk1][R]
    float* part;          // this sender's pass-2 partials [n_rc2][2][nS][T_pad]
    int64_t T, T_pad;
    int32_t R, halves;    // m * G query rows; 128-row halves of them
    int32_t q_rows;       // rows loaded of a half: 128, or R rounded up to 32 where there is one half
    int32_t n_chunk1;     // pass-1 partial slots: four per chunk of positions
    int32_t n_blk2;       // pass-2 blocks of positions
    int32_t n_rc1, n_rc2; // row chunks of each pass
    int32_t narrow;       // pass 2 takes blocks of one tile (k_narrow_tc)
    int32_t few;          // pass 2 hands its last half's columns out in eights (FEW)
    int32_t m_self;       // query tokens whose own keys join the softmax (m or 0)
    int32_t chunk1;       // pass-1 positions per chunk
    const int32_t* pages; // block table of a paged sender that pass 1 reads itself, else null
    int32_t n_pages, page_shift;
};

struct TcBatch {
    CUtensorMap omap;     // 2D {16, 128} block of ones columns, one box, 32-byte swizzle
    int32_t n;
    int32_t nL, Hq, Hkv, G, log2g;
    int32_t stages1, rows1;       // pass 1: K ring stages, Q rows held
    int32_t kbufs, rows2;         // pass 2: K blocks in flight (1 or 2, four tiles each; k_narrow_tc: K tiles), Q rows held
    int32_t max_rc1, max_rc2;
    float sl2e, p;
    int32_t p_inf, ph;
    int64_t weight1, weight2;     // work of each pass: 128-row halves over all units
    uint64_t wait_ns;     // limit of one bounded mbarrier wait
    int32_t few;          // some sender has `few`
    int32_t paged;        // some sender has `pages`: warp 3 of pass 1 stores its tiles
    int32_t stall;        // 1: CTA 0's pass-1 MMA issuer first waits on a barrier nothing arrives on
    uint32_t* err;
    TcMaps maps[kMaxTcSenders];   // (apart from the sizes: a tensor map is aligned to 128 bytes)
    TcSender s[kMaxTcSenders];
};

static_assert(sizeof(TcBatch) <= 32764, "kernel parameters");

// The launches of head dimension D.
template <int D>
cudaError_t launch_stats_d(const TcBatch& tb, int grid, cudaStream_t st);
template <int D>
cudaError_t launch_accum_d(const TcBatch& tb, int grid, cudaStream_t st);
template <int D>
cudaError_t launch_narrow_d(const TcBatch& tb, int grid, cudaStream_t st);
}  // namespace tc

namespace {
using namespace sm100;
using namespace tc;

// One unit of work: sender i, group s, row chunk rc, position chunk (pass 1) or block (pass 2) c.
struct Unit {
    int i, s, c, rc;
};


struct Ctl {
    uint64_t k_full[kMaxStages], k_empty[kMaxStages];
    uint64_t t_full[4], t_empty[4];   // ring of TMEM buffers of 128 columns
    uint64_t q_full, q_empty, drain[2], o_full;
    uint64_t q2_full[2], q2_empty[2];   // k_narrow_tc's two Q buffers
    uint64_t stall;         // failure-detection test: a barrier nothing arrives on
    uint64_t wait_ns;       // limit of one bounded wait
    uint64_t xb, xe;        // pass 2: a block's sums written by the epilogue and read by warp 3
    int32_t units;          // this CTA's units, the first of which is `first`
    Unit first;
    int32_t redo_lo, redo_hi;   // pass 1: first and last of them with a sum out of range
    uint32_t tmem_base;
    int abort;
};
static_assert(sizeof(Ctl) <= 512, "the epilogue exchange area starts 512 bytes after Ctl");

__device__ __forceinline__ uint64_t now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait: true when the phase completed, false on abort (set by anyone) or timeout.
// `tag` names the wait in the device error word (bit 8 + tag) when it times out.  The polling is
// out of line: the epilogue loops stay small enough for the instruction cache.
static __device__ __noinline__ bool wait_poll(uint64_t* bar, uint32_t parity, Ctl* ctl, uint32_t* err, int tag) {
    const uint64_t t0 = now_ns();
    for (uint32_t i = 1; i < (1u << 30); ++i) {
        if (mbar_try_wait_hint(bar, parity, kPollNs)) return true;
        if ((i & 63) == 0) {
            if (*reinterpret_cast<volatile int*>(&ctl->abort)) return false;
            if (now_ns() - t0 > ctl->wait_ns) {
                *reinterpret_cast<volatile int*>(&ctl->abort) = 1;
                atomicOr(err, kErrTimeout | (1u << (8 + tag)));
                return false;
            }
        }
    }
    *reinterpret_cast<volatile int*>(&ctl->abort) = 1;
    atomicOr(err, kErrTimeout);
    return false;
}

__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, Ctl* ctl, uint32_t* err, int tag) {
    return mbar_try_wait(bar, parity) || wait_poll(bar, parity, ctl, err, tag);
}

// Wait used only on the way out (drain): bounded by kWaitNs whatever the configured limit
// (the copies and MMAs it waits for always complete), ignores the abort flag.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
    const uint64_t t0 = now_ns();
    while (!mbar_try_wait(bar, parity))
        if (now_ns() - t0 > kWaitNs) return;
}

__device__ __forceinline__ uint8_t* align1024(uint8_t* p) {
    return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

// Row chunk rc of n holds the sender's 128-row halves [rc * halves / n, (rc + 1) * halves / n).
__device__ __forceinline__ int rc_begin(int halves, int n, int rc) { return rc * halves / n; }

template <int PASS>
__device__ __forceinline__ int n_rc(const TcSender& sd) { return PASS == 1 ? sd.n_rc1 : sd.n_rc2; }
template <int PASS>
__device__ __forceinline__ int n_c(const TcSender& sd) { return PASS == 1 ? sd.n_chunk1 / 4 : sd.n_blk2; }

// Units are ordered by row chunk, sender, group and position.  One unit weighs as much as its row
// chunk has halves.  Unit that begins at or after weight `w`, and its place in the order.
template <int PASS>
__device__ __forceinline__ int64_t unit_at(const TcBatch& bt, int64_t w, Unit* un) {
    const int nS = bt.nL * bt.Hkv, max_rc = PASS == 1 ? bt.max_rc1 : bt.max_rc2;
    int64_t u = 0;
    for (int rc = 0; rc < max_rc; ++rc)
        for (int i = 0; i < bt.n; ++i) {
            const TcSender& sd = bt.s[i];
            const int n = n_rc<PASS>(sd);
            if (rc >= n) continue;
            const int wt = rc_begin(sd.halves, n, rc + 1) - rc_begin(sd.halves, n, rc);
            const int64_t units = (int64_t)nS * n_c<PASS>(sd);
            if (w < units * wt) {
                const int64_t k = (w + wt - 1) / wt;
                if (k < units) {
                    *un = Unit{i, (int)(k / n_c<PASS>(sd)), (int)(k % n_c<PASS>(sd)), rc};
                    return u + k;
                }
                w = units * wt;   // rounds up to the next sender's first unit
            }
            w -= units * wt;
            u += units;
        }
    return u;
}

// This CTA's contiguous share of the units (by weight), into shared memory.
template <int PASS>
__device__ __forceinline__ void my_units(const TcBatch& bt, Ctl* ctl) {
    const int64_t total = PASS == 1 ? bt.weight1 : bt.weight2;
    Unit first{0, 0, 0, 0}, end;
    const int64_t b = unit_at<PASS>(bt, total * blockIdx.x / gridDim.x, &first);
    ctl->units = (int32_t)(unit_at<PASS>(bt, total * (blockIdx.x + 1) / gridDim.x, &end) - b);
    ctl->first = first;
}

// Tiles of the query tokens' own keys, which pass 1 takes after those of a group's last chunk.
__device__ __forceinline__ int self_tiles(const TcSender& sd) { return (sd.m_self + kTileRows - 1) / kTileRows; }

// The next unit in order, without a division.  `nc`: the sender's chunks or blocks, kept by the
// caller (an indexed read of the kernel parameters for every unit holds a role up).
template <int PASS>
__device__ __forceinline__ void next_unit(const TcBatch& bt, Unit& un, int nc) {
    if (++un.c < nc) return;
    un.c = 0;
    if (++un.s < bt.nL * bt.Hkv) return;
    un.s = 0;
    const int max_rc = PASS == 1 ? bt.max_rc1 : bt.max_rc2;
    do {
        if (++un.i == bt.n) {
            un.i = 0;
            if (++un.rc >= max_rc) {   // past the last unit
                un.rc = 0;
                return;
            }
        }
    } while (n_rc<PASS>(bt.s[un.i]) <= un.rc);
}

// Shared memory of pass 1: [Q: d / 64 blocks x rows1 x 128 B][K ring][Ctl]; of pass 2:
// [Q][offset terms: rows2 x 32 B][ones: 4 KB][K blocks of four tiles][Ctl][exchange of sums].
struct Smem {
    uint8_t* q;
    uint8_t* ext;     // pass 2: offset terms of Q's rows [rows2][32 B], 32-byte swizzle
    uint8_t* ones;    // pass 2: ones columns [128][32 B], 32-byte swizzle
    uint8_t* k;
    Ctl* ctl;
    float* epi;
};

template <int D, int PASS>
__device__ __forceinline__ Smem carve(uint8_t* raw, const TcBatch& bt) {
    constexpr int kTile = kTileRows * D * 2;
    Smem sm;
    uint8_t* base = align1024(raw);
    sm.q = base;
    if (PASS == 1) {
        sm.ext = sm.ones = nullptr;
        sm.k = base + (size_t)bt.rows1 * D * 2;
        sm.ctl = reinterpret_cast<Ctl*>(sm.k + (size_t)bt.stages1 * kTile);
    } else {
        sm.ext = base + (size_t)bt.rows2 * D * 2;
        sm.ones = sm.ext + (size_t)bt.rows2 * 32;
        sm.k = sm.ones + 128 * 32;
        sm.ctl = reinterpret_cast<Ctl*>(sm.k + (size_t)4 * bt.kbufs * kTile);
    }
    sm.epi = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(sm.ctl) + 512);
    return sm;
}

// `k_releasers`: roles that arrive on a K slot's empty barrier.
__device__ __forceinline__ void init_ctl(Ctl* ctl, int k_releasers, uint64_t wait_ns) {
    for (int k = 0; k < kMaxStages; ++k) {
        mbar_init(&ctl->k_full[k], 1);
        mbar_init(&ctl->k_empty[k], k_releasers);
    }
    for (int b = 0; b < 4; ++b) {
        mbar_init(&ctl->t_full[b], 1);
        mbar_init(&ctl->t_empty[b], kEpiWarps);
    }
    mbar_init(&ctl->xb, kEpiWarps);
    mbar_init(&ctl->xe, 1);
    mbar_init(&ctl->q_full, 1);
    mbar_init(&ctl->q_empty, 2);
    for (int b = 0; b < 2; ++b) {
        mbar_init(&ctl->q2_full[b], 1);
        mbar_init(&ctl->q2_empty[b], 2);
    }
    mbar_init(&ctl->drain[0], 1);
    mbar_init(&ctl->drain[1], 1);
    mbar_init(&ctl->o_full, 1);
    mbar_init(&ctl->stall, 1);
    ctl->wait_ns = wait_ns;
    ctl->abort = 0;
    ctl->redo_lo = INT32_MAX;
    ctl->redo_hi = -1;
    fence_barrier_init();
}

// Producer: the 128-row halves [h0, h0 + nh) of group s's Q (s = l * Hkv + g) into the Q region
// (column blocks of `rows` rows).  Pass 2 also brings the rows' offset terms.  Rows past the loaded ones
// of a half hold anything: pass 1 writes nothing of theirs, pass 2's MMA does not read them.
template <int D, int PASS>
__device__ __forceinline__ void load_q(const TcBatch& bt, const TcMaps& mp, const Smem& sm, int s, int h0, int nh,
                                       int q_rows, uint64_t* full) {
    const int l = s / bt.Hkv, g = s % bt.Hkv;
    const int rows = PASS == 1 ? bt.rows1 : bt.rows2;
    mbar_arrive_expect_tx(full, (uint32_t)(nh * q_rows) * (D * 2 + (PASS == 2 ? 32 : 0)));
    for (int h = 0; h < nh; ++h) {
        if (PASS == 2)
            tma_load_3d(sm.ext + (size_t)h * kRowHalf * 32, &mp.k[2], full, 0, (h0 + h) * kRowHalf, s);
        for (int kb = 0; kb < D / 64; ++kb)
            tma_load_4d(sm.q + ((size_t)kb * rows + h * kRowHalf) * 128, &mp.q, full, 64 * kb, g * bt.G,
                        (h0 + h) * kRowHalf / bt.G, l);
    }
}

// Low word of a shared-memory matrix descriptor (the address field); the high word is a constant
// of the swizzle, so a K-step or another row block only adds to the low word.
__device__ __forceinline__ uint64_t desc64(uint32_t lo, uint32_t hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
    return d;
}

// One contraction over d (d / 16 UMMA K-steps) into d_tmem: operand rows of 128 B in 64-column
// blocks that lie `a_blk` / `b_blk` (16-byte units) apart.
template <int D>
__device__ __forceinline__ void mma_d(uint32_t d_tmem, uint32_t a_lo, uint32_t a_blk, uint32_t b_lo, uint32_t b_blk,
                                      uint32_t hi, uint32_t idesc) {
#pragma unroll
    for (int k = 0; k < D / 16; ++k)
        umma_bf16(d_tmem, desc64(a_lo + (k / 4) * a_blk + (k & 3) * 2, hi), desc64(b_lo + (k / 4) * b_blk + (k & 3) * 2, hi),
                  idesc, k > 0 ? 1u : 0u);
}

// 32 columns of pass 1 for this lane's row: sum of exp2(c z - m), m the row's offset (log2 domain).
// The packed adds leave the loop bound by exp2 (584 cycles for a 128 x 128 buffer, 603 with scalar
// adds, against 512 for its exp2 alone).
__device__ __forceinline__ uint64_t stats_block(const float (&v)[32], uint64_t cc, float m) {
    const uint64_t nm = pack2(-m, -m);
    uint64_t p0 = 0, p1 = 0;
#pragma unroll
    for (int q = 0; q < 16; q += 2) {
        float a0, a1, b0, b1;
        unpack2(ffma2(pack2(v[2 * q], v[2 * q + 1]), cc, nm), a0, a1);
        unpack2(ffma2(pack2(v[2 * q + 2], v[2 * q + 3]), cc, nm), b0, b1);
        p0 = fadd2(p0, pack2(ex2(a0), ex2(a1)));
        p1 = fadd2(p1, pack2(ex2(b0), ex2(b1)));
    }
    return fadd2(p0, p1);
}

// ===========================================================================
// pass 1
// ===========================================================================
// Epilogue of pass 1 over the CTA's units: offset and sum of each row.  `n`: accumulator buffers
// consumed so far.  RISE: the second run, which replaces the sums that were out of range.
template <int NH, bool RISE>
__device__ __forceinline__ void stats_rows(const TcBatch& bt, Ctl* ctl, uint32_t tmem, uint32_t& n) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int q = (warp - kEpi0) >> 2;       // column quarter: positions 32 q .. +31 of each tile
    const int sp = warp & 3;                 // TMEM lane quarter
    const int L = sp * 32 + lane;
    const uint32_t ta = tmem + ((uint32_t)(sp * 32) << 16) + 32 * q;
    const float c = bt.sl2e;
    Unit un = ctl->first;
    const uint64_t cc = pack2(c, c);
    float M[NH];                             // per half: offset (log2 domain) and sum of exp2(c z - offset)
    uint64_t S[NH];
    bool ok = true;
    // One tile, one buffer a half: load its 32 columns, hand the buffer back, sum.  PART: `nvalid` of
    // the columns hold a position.  SELF: the columns are query tokens' own keys, of which row
    // (token r, head) has those up to r: `nvalid` there, `tok0` of them for the thread's first row
    // and one more for each token after its own.  FIRST: the chunk's first tile sets the offset to the
    // largest of its first 8 logits, or to -FLT_MAX where it has none (then the row's first self keys set
    // it).  RISE (the second run): the largest of all 32, and a logit more than kRaise above the offset
    // raises it.
    // (In the first run the largest of 32 costs 3 us of 124, a maximum in every buffer 14, a look at
    // every buffer's sum 9 to 18.)
    auto tile = [&](auto part, auto self, auto first, int nvalid, int nh, int tok0) {
        constexpr bool PART = decltype(part)::value, SELF = decltype(self)::value;
        constexpr bool FIRST = decltype(first)::value;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            if (h >= nh) break;
            const uint32_t buf = n & 3;
            if (!(ok = wait_bar(&ctl->t_full[buf], (n >> 2) & 1, ctl, bt.err, 5))) break;
            ++n;
            tc_fence_after();
            float v[32];
            tmem_ld32(ta + buf * 128, v);
            tmem_wait_ld(v);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->t_empty[buf]);
            if (PART) {
                const int nv = SELF ? min(nvalid, tok0 + (h * kRowHalf >> bt.log2g)) : nvalid;
#pragma unroll
                for (int e = 0; e < 32; ++e) v[e] = e < nv ? v[e] : -INFINITY;
            }
            if (RISE) {
                const float m = max_tree1(v) * c;
                if (FIRST) {
                    M[h] = fmaxf(m, -FLT_MAX);
                } else if (m > M[h] + kRaise) {
                    const float f = ex2(M[h] - m);
                    S[h] = fmul2(S[h], pack2(f, f));
                    M[h] = m;
                }
            } else if (FIRST || (SELF && M[h] == -FLT_MAX)) {
                const float m = fmax3(fmax3(v[0], v[1], v[2]), fmax3(v[3], v[4], v[5]), fmaxf(v[6], v[7]));
                M[h] = fmaxf(m * c, -FLT_MAX);
            }
            S[h] = fadd2(S[h], stats_block(v, cc, M[h]));
        }
    };
    for (int left = ctl->units; left > 0 && ok;) {
        // the run of chunks of one group and row chunk (nothing but positions changes in it)
        const TcSender& sd = bt.s[un.i];
        const int h0 = rc_begin(sd.halves, sd.n_rc1, un.rc);
        const int nh = rc_begin(sd.halves, sd.n_rc1, un.rc + 1) - h0;
        const int R = sd.R, rows = R - h0 * kRowHalf - L;   // rows: query rows from the thread's first on
        const int m_self = sd.m_self, tok = (h0 * kRowHalf + L) >> bt.log2g;   // the thread's first row's token
        const int chunk = sd.chunk1, nc = n_c<1>(sd), len_run = min(left, nc - un.c);
        int rest = (int)sd.T - un.c * chunk;   // positions from the chunk's first on
        float2* dst = sd.stats + ((int64_t)un.s * sd.n_chunk1 + 4 * un.c + q) * R + h0 * kRowHalf + L;
        left -= len_run;
        un.c += len_run - 1;
        next_unit<1>(bt, un, nc);
        for (int k = 0; k < len_run && ok; ++k, rest -= chunk, dst += 4 * (int64_t)R) {
            const int len = min(chunk, rest);
#pragma unroll
            for (int h = 0; h < NH; ++h) { M[h] = -INFINITY; S[h] = 0; }
            int t0 = 0;
            constexpr std::false_type no{};
            constexpr std::true_type yes{};
            if (len >= kTileRows) {
                tile(no, no, yes, 32, nh, 0);
                for (t0 = kTileRows; t0 + kTileRows <= len && ok; t0 += kTileRows) tile(no, no, no, 32, nh, 0);
                if (t0 < len && ok) tile(yes, no, no, len - t0 - 32 * q, nh, 0);
            } else {
                tile(yes, no, yes, len - 32 * q, nh, 0);
            }
            if (m_self > 0 && rest <= chunk)   // the query tokens' own keys join the last chunk
                for (int u0 = 32 * q; u0 - 32 * q < m_self && ok; u0 += kTileRows)
                    tile(yes, yes, no, m_self - u0, nh, tok + 1 - u0);
            if (!ok) break;
            // this warp's partial statistics for the chunk: slot 4 c + q (rows of positions past T
            // are (-FLT_MAX, 0), which adds nothing); the combine kernel merges all slots
#pragma unroll
            for (int h = 0; h < NH; ++h) {
                if (h >= nh || h * kRowHalf >= rows) break;
                float s0, s1;
                unpack2(S[h], s0, s1);
                // The combine kernel scales sums by powers of two down to 2^-126, below which exp2 is zero, and
                // the largest of a row's offsets has a sum of at least one.  A large sum's exponent goes into
                // the offset (what that rounds off, back into the sum), so that what is scaled to zero is nothing.
                float m = M[h], x = s0 + s1;
                if (x > 0x1p30f && x <= FLT_MAX) {
                    const int e = (__float_as_int(x) >> 23) - 127;
                    const float m1 = m + (float)e;
                    x = __int_as_float(__float_as_int(x) - (e << 23)) * ex2(m - (m1 - (float)e));
                    m = m1;
                }
                float2* at = dst + h * kRowHalf;
                if (RISE) {
                    if (at->y <= FLT_MAX) continue;   // in range in the first run
                } else if (!(x <= FLT_MAX)) {
                    const int unit = ctl->units - left - len_run + k;
                    atomicMin(&ctl->redo_lo, unit);
                    atomicMax(&ctl->redo_hi, unit);
                }
                *at = make_float2(m, x);
            }
        }
    }
}

// The warps' work over the CTA's units, and where each role stands at its end, for a second run:
// K tiles and Q loads issued or consumed, accumulator buffers filled or consumed, ring slot of the
// next K tile and its phase parity.
struct StatsAt {
    int64_t kt;
    uint32_t qn, n, ph;
    int st;
};

template <int D, int NH, bool AGAIN>
__device__ __forceinline__ StatsAt stats_run(const TcBatch& bt, const Smem& sm, uint32_t tmem, StatsAt at) {
    constexpr int kTile = kTileRows * D * 2;
    Ctl* ctl = sm.ctl;
    const int warp = threadIdx.x >> 5;
    const int stages = bt.stages1;
    int64_t kt = at.kt;
    uint32_t qn = at.qn, n = at.n, ph = at.ph;
    int st = at.st;
    const int n_units = ctl->units;
    Unit un = ctl->first;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (elect_one()) {
            bool ok = true;
            int nc = 0, l = 0, g = 0, n_self = 0, chunk = 0;
            int64_t T = 0;
            const int32_t* pages = nullptr;
            int32_t n_pages = 0, ps = 0;
            for (int u = 0; u < n_units && ok; ++u, next_unit<1>(bt, un, nc)) {
                const TcMaps& mp = bt.maps[un.i];
                if (u == 0 || un.c == 0) {   // another group or row chunk: its Q
                    const TcSender& sd = bt.s[un.i];
                    nc = n_c<1>(sd);
                    chunk = sd.chunk1;
                    n_self = self_tiles(sd);
                    pages = sd.pages;
                    n_pages = sd.n_pages;
                    ps = sd.page_shift;
                    T = sd.T;
                    l = un.s / bt.Hkv;
                    g = un.s % bt.Hkv;
                    if (!(ok = wait_bar(&ctl->q_empty, (uint32_t)((qn & 1) ^ 1), ctl, bt.err, 0))) break;
                    const int h0 = rc_begin(sd.halves, sd.n_rc1, un.rc);
                    load_q<D, 1>(bt, mp, sm, un.s, h0, rc_begin(sd.halves, sd.n_rc1, un.rc + 1) - h0, sd.q_rows,
                             &ctl->q_full);
                    ++qn;
                }
                const int64_t c0 = (int64_t)un.c * chunk;
                const int nt = (int)((min((int64_t)chunk, T - c0) + kTileRows - 1) / kTileRows);
                const int n_tiles = nt + (un.c + 1 == nc ? n_self : 0);
                for (int tile = 0; tile < n_tiles; ++tile) {
                    const bool self = tile >= nt;
                    const int32_t row = self ? (tile - nt) * kTileRows : (int32_t)(c0 + tile * kTileRows);
                    // a tile's block-table entries, all in flight together while its slot is waited for
                    const int box = ps < 7 ? 1 << ps : kTileRows;
                    int32_t entry[kTileRows >> kMinPageShift];
                    if (pages && !self) {
#pragma unroll
                        for (int r = 0; r < kTileRows >> kMinPageShift; ++r)
                            if (r * box < kTileRows && row + r * box < T) entry[r] = __ldg(pages + ((row + r * box) >> ps));
                    }
                    if (!(ok = wait_bar(&ctl->k_empty[st], ph ^ 1u, ctl, bt.err, 1))) break;
                    mbar_arrive_expect_tx(&ctl->k_full[st], kTile);
                    if (pages && !self) {
                        // one box a page (or 128 rows of one); a page past T, or outside the pool (recorded), is
                        // the coordinate past the last page, which reads as zeros
#pragma unroll
                        for (int r = 0; r < kTileRows >> kMinPageShift; ++r) {
                            if (r * box >= kTileRows) break;
                            int32_t pg = n_pages;
                            if (row + r * box < T) {
                                pg = entry[r];
                                if (pg < 0 || pg >= n_pages) {
                                    pg = n_pages;
                                    atomicOr(bt.err, kErrPageIndex);
                                }
                            }
                            for (int kb = 0; kb < D / 64; ++kb)
                                tma_load_5d(sm.k + (size_t)st * kTile + (kb * kTileRows + r * box) * 128, &mp.k[0],
                                            &ctl->k_full[st], 64 * kb, (row + r * box) & ((1 << ps) - 1), pg, g, l);
                        }
                    } else {
                        for (int kb = 0; kb < D / 64; ++kb)
                            tma_load_4d(sm.k + (size_t)st * kTile + kb * kTileRows * 128, &mp.k[self ? 1 : 0],
                                        &ctl->k_full[st], 64 * kb, row, g, l);
                    }
                    ++kt;
                    if (++st == stages) { st = 0; ph ^= 1u; }
                }
            }
            // drain: every issued load must land before the CTA exits
            for (int64_t k = kt - stages > 0 ? kt - stages : 0; k < kt; ++k)
                drain_wait(&ctl->k_full[k % stages], (uint32_t)((k / stages) & 1));
            if (qn > 0) drain_wait(&ctl->q_full, (uint32_t)((qn - 1) & 1));
        }
    } else if (warp <= 2) {
        // ---------------- MMA issuers ----------------
        if (elect_one()) {
            const uint32_t me = (uint32_t)warp - 1;
            bool ok = true;
            constexpr uint32_t idesc = idesc_bf16_f32(128, 128);
            const uint64_t qd = smem_desc_sw128(smem_u32(sm.q));
            const uint32_t hi = (uint32_t)(qd >> 32), q_lo = (uint32_t)qd;
            const uint32_t k_lo = (uint32_t)smem_desc_sw128(smem_u32(sm.k));
            const uint32_t q_blk = (uint32_t)bt.rows1 * 128 >> 4;
            // failure-detection test: wait on a barrier that nothing arrives on, so the bounded
            // wait gives up, sets the abort flag and every role of this CTA leaves
            if (!AGAIN && bt.stall && blockIdx.x == 0) ok = wait_bar(&ctl->stall, 0, ctl, bt.err, 6);
            uint32_t nh = 0;
            int nc = 0, n_self = 0, chunk = 0;
            int64_t T = 0;
            for (int u = 0; u < n_units && ok; ++u, next_unit<1>(bt, un, nc)) {
                if (u == 0 || un.c == 0) {   // another group or row chunk: its Q
                    const TcSender& sd = bt.s[un.i];
                    nc = n_c<1>(sd);
                    chunk = sd.chunk1;
                    n_self = self_tiles(sd);
                    T = sd.T;
                    nh = rc_begin(sd.halves, sd.n_rc1, un.rc + 1) - rc_begin(sd.halves, sd.n_rc1, un.rc);
                    if (u > 0) umma_commit(&ctl->q_empty);
                    if (!(ok = wait_bar(&ctl->q_full, qn & 1, ctl, bt.err, 2))) break;
                    ++qn;
                }
                const int64_t c0 = (int64_t)un.c * chunk;
                const int nt = (int)((min((int64_t)chunk, T - c0) + kTileRows - 1) / kTileRows) +
                               (un.c + 1 == nc ? n_self : 0);
                for (int tile = 0; tile < nt; ++tile) {
                    if (!(ok = wait_bar(&ctl->k_full[st], ph, ctl, bt.err, 3))) break;
                    const uint32_t kt_lo = k_lo + (uint32_t)st * (kTile >> 4);
                    for (uint32_t h = (n ^ me) & 1; h < nh; h += 2) {   // the tile's buffers n + h of my parity
                        const uint32_t x = n + h, buf = x & 3;
                        if (!(ok = wait_bar(&ctl->t_empty[buf], ((x >> 2) & 1) ^ 1, ctl, bt.err, 4))) break;
                        tc_fence_after();
                        mma_d<D>(tmem + buf * 128, q_lo + h * (kRowHalf * 128 >> 4), q_blk, kt_lo, kTileRows * 128 >> 4, hi,
                                 idesc);
                        umma_commit(&ctl->t_full[buf]);
                    }
                    if (!ok) break;
                    n += nh;
                    umma_commit(&ctl->k_empty[st]);
                    if (++st == stages) { st = 0; ph ^= 1u; }
                }
            }
            umma_commit(&ctl->q_empty);
            umma_commit(&ctl->drain[me]);
            drain_wait(&ctl->drain[me], AGAIN ? 1u : 0u);
        }
    } else if (warp < kEpi0) {
        // ---------------- paged senders: the staged tiles on into the contiguous copy ----------------
        if (bt.paged && elect_one()) {
            int prev = -1;            // slot of the tile before, whose stores may still read it
            bool ok = true;
            int nc = 0, l = 0, g = 0, n_self = 0, chunk = 0;
            int64_t T = 0;
            bool store = false;
            for (int u = 0; u < n_units && ok; ++u, next_unit<1>(bt, un, nc)) {
                if (u == 0 || un.c == 0) {
                    const TcSender& sd = bt.s[un.i];
                    nc = n_c<1>(sd);
                    chunk = sd.chunk1;
                    n_self = self_tiles(sd);
                    T = sd.T;
                    l = un.s / bt.Hkv;
                    g = un.s % bt.Hkv;
                    store = !AGAIN && sd.pages && un.rc == 0;   // once for all row chunks
                }
                const int64_t c0 = (int64_t)un.c * chunk;
                const int nt = (int)((min((int64_t)chunk, T - c0) + kTileRows - 1) / kTileRows);
                const int n_tiles = nt + (un.c + 1 == nc ? n_self : 0);
                for (int tile = 0; tile < n_tiles; ++tile) {
                    if (!(ok = wait_bar(&ctl->k_full[st], ph, ctl, bt.err, 3))) break;
                    if (store && tile < nt)
                        for (int kb = 0; kb < D / 64; ++kb)
                            tma_store_4d(&bt.maps[un.i].k[2], sm.k + (size_t)st * kTile + kb * kTileRows * 128, 64 * kb,
                                         (int32_t)(c0 + tile * kTileRows), g, l);
                    bulk_commit();
                    if (prev >= 0) {
                        bulk_wait_read<1>();
                        mbar_arrive(&ctl->k_empty[prev]);
                    }
                    prev = st;
                    if (++st == stages) { st = 0; ph ^= 1u; }
                }
            }
            if (prev >= 0) {
                bulk_wait_read<0>();
                mbar_arrive(&ctl->k_empty[prev]);
            }
            bulk_wait<0>();
        }
    } else {
        // ---------------- epilogue ----------------
        stats_rows<NH, AGAIN>(bt, ctl, tmem, n);
    }
    return StatsAt{kt, qn, n, ph, st};
}

// (out of line: the first run keeps its registers)
template <int D, int NH>
__device__ __noinline__ void stats_again(const TcBatch& bt, uint8_t* smem, uint32_t tmem, int64_t kt, uint32_t qn, uint32_t n,
                                         uint32_t ph, int st) {
    stats_run<D, NH, true>(bt, carve<D, 1>(smem, bt), tmem, StatsAt{kt, qn, n, ph, st});
}

// Epilogue: thread = TMEM lane = row 128 h + lane of every half h and a quarter of each tile's
// positions; it keeps the offset and sum of exp2 of its rows over the chunk and writes them as
// partial (chunk, quarter); the combine kernel merges all partials of a group s.  The two MMA
// issuers take alternate buffers.
// A chunk's offset is the largest of its first 8 logits, so a sum is in range unless a later logit
// lies 127 (log2 domain) above all of those: out of 6e8 normal logits, one does from a standard
// deviation of 10 (natural units) on.  Then the CTA runs the units from its first to its last such
// sum again with offsets that rise with the logits, and replaces those sums alone, so that they
// depend on nothing else in the call: 36 layers, T = 8192, 256 rows take 124 us at standard deviations
// up to 8, 142 at 10 and 248 from 14 on (recomputing such rows in the combine kernel took 14 ms and
// more).  Stretches of marked units in place of the one range gain nothing (275 us from 14 on).
// Bound by the epilogue, whose waits, TMEM loads, exp2 and packed adds take 115 us without the K
// loads for 36 layers, T = 8192, 256 rows (64 at the rate of exp2 alone); the K loads without the
// epilogue take 102 (89 at the copy rate).
// 124 us together, against 130 with two accumulator tiles of two epilogue groups each and one
// issuer; 3 x T = 16384 with 512 rows 1216 against 1448 us.  Chunks of 512, 640 or 768 positions
// take 119 to 122 us, but the combine kernel 2 to 4 more, and longer at 512 rows.
template <int D, int NH>
__global__ void __launch_bounds__(kThreadsTc, 1) k_stats_tc(const __grid_constant__ TcBatch bt) {
    extern __shared__ uint8_t smem_raw[];
    const Smem sm = carve<D, 1>(smem_raw, bt);
    Ctl* ctl = sm.ctl;
    const int warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        init_ctl(ctl, bt.paged ? 3 : 2, bt.wait_ns);
        my_units<1>(bt, ctl);
    }
    if (warp == 1) {
        tmem_alloc(&ctl->tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    const StatsAt at = stats_run<D, NH, false>(bt, sm, tmem, StatsAt{0, 0, 0, 0, 0});
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (ctl->redo_hi >= 0 && !ctl->abort) {
        if (threadIdx.x == 0) {
            Unit f = ctl->first;
            for (int u = 0; u < ctl->redo_lo; ++u) next_unit<1>(bt, f, n_c<1>(bt.s[f.i]));
            ctl->first = f;
            ctl->units = ctl->redo_hi - ctl->redo_lo + 1;
        }
        __syncthreads();
        stats_again<D, NH>(bt, smem_raw, tmem, at.kt, at.qn, at.n, at.ph, at.st);
        tc_fence_before();
        __syncthreads();
    }
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// ===========================================================================
// pass 2
// ===========================================================================
// Pool over positions: the thread holds x[0..3], four neighbouring positions; the lane before it
// the four before, the lane after it the four after.  o[k] = max over positions k - PH .. k + PH.
// The window of each position is the thread's own part of it and a suffix of the lane before or a
// prefix of the lane after: six shuffles for four positions (PH = 3).
template <int PH>
__device__ __forceinline__ void pool4(const float (&x)[4], float (&o)[4]) {
    constexpr unsigned kAll = 0xffffffffu;
    if (PH == 0) {
#pragma unroll
        for (int k = 0; k < 4; ++k) o[k] = x[k];
    } else if (PH == 1) {
        o[0] = fmax3(__shfl_up_sync(kAll, x[3], 1), x[0], x[1]);
        o[1] = fmax3(x[0], x[1], x[2]);
        o[2] = fmax3(x[1], x[2], x[3]);
        o[3] = fmax3(x[2], x[3], __shfl_down_sync(kAll, x[0], 1));
    } else if (PH == 2) {
        const float s23 = fmaxf(x[2], x[3]), p01 = fmaxf(x[0], x[1]);
        const float all = fmaxf(p01, s23);
        o[0] = fmax3(__shfl_up_sync(kAll, s23, 1), p01, x[2]);
        o[1] = fmaxf(__shfl_up_sync(kAll, x[3], 1), all);
        o[2] = fmaxf(all, __shfl_down_sync(kAll, x[0], 1));
        o[3] = fmax3(x[1], s23, __shfl_down_sync(kAll, p01, 1));
    } else {
        const float s23 = fmaxf(x[2], x[3]), p01 = fmaxf(x[0], x[1]);
        const float s123 = fmaxf(x[1], s23), p012 = fmaxf(p01, x[2]);
        const float all = fmaxf(p01, s23);
        o[0] = fmaxf(__shfl_up_sync(kAll, s123, 1), all);
        o[1] = fmax3(__shfl_up_sync(kAll, s23, 1), all, __shfl_down_sync(kAll, x[0], 1));
        o[2] = fmax3(__shfl_up_sync(kAll, x[3], 1), all, __shfl_down_sync(kAll, p01, 1));
        o[3] = fmaxf(all, __shfl_down_sync(kAll, p012, 1));
    }
}

__device__ __forceinline__ float pow_p(float x, float p) { return x > 0.f ? ex2(p * lg2(x)) : 0.f; }

// e0 + .. + e3 as (e0 + e2) + (e1 + e3): one packed add of neighbouring registers, one scalar add.
__device__ __forceinline__ float sum4(const float* e) {
    float p, q;
    unpack2(fadd2(pack2(e[0], e[1]), pack2(e[2], e[3])), p, q);
    return p + q;
}

// Head sums of C / G tokens from their C columns: a / G = exp2(c D - centre) per column, `nc` minus
// the centre, summed over each token's G heads, as pairs of tokens (2 i, 2 i + 1).
template <int G, int C>
__device__ __forceinline__ void head_sums(const float (&v)[C], uint64_t cc, uint64_t nc, uint64_t* b) {
    float e[C];
#pragma unroll
    for (int q = 0; q < C / 2; ++q) {
        float a0, a1;
        unpack2(ffma2(pack2(v[2 * q], v[2 * q + 1]), cc, nc), a0, a1);
        e[2 * q] = ex2(a0);
        e[2 * q + 1] = ex2(a1);
    }
#pragma unroll
    for (int i = 0; i < C / (2 * G); ++i) {
        if (G == 1) b[i] = pack2(e[2 * i], e[2 * i + 1]);
        if (G == 2) b[i] = pack2(e[4 * i] + e[4 * i + 1], e[4 * i + 2] + e[4 * i + 3]);
        if (G == 4)
            b[i] = pack2(sum4(e + 8 * i), sum4(e + 8 * i + 4));
    }
}

// Epilogue: lane quarter w = warp % 4 of block c covers positions 480 c + 120 w - 4 .. + 127; its
// lane i holds positions 4 i .. 4 i + 3 of them, one in each of the block's four tiles.  Lanes 1
// to 30 are outputs, lanes 0 and 31 their Pool margin.  The four warps of a lane quarter take 32
// columns (query rows) each of every buffer; their sums meet in shared memory at the end of the
// block, where warp 3 does the adding: an epilogue warp that waited for its three neighbours would
// hold up the next block's buffers (28 us of this pass).  MMA issuer i fills the buffers of tiles i
// and i + 2.
// Bound by the epilogue: 138 us alone for 36 layers, T = 8192, 256 rows (of about 3700 cycles for
// four buffers, exp2 takes 2420 and Pool 780), 155 with the K loads (+12) and the MMA (+5).
// Against one position a thread, tiles of 104 outputs in 128 rows and Pool through a shuffle for
// every position and shift: 155 against 170 us; 3 x T = 16384 with 512 rows 1627 against 1867;
// 24 layers, 2 x T = 7001, 200 rows of d = 64, where the mma.sync kernel ran, 137 against 769.
// Blocks of fewer lane quarters gain nothing where there are fewer blocks than SMs (16.2 us either
// way for 32 groups of T = 2106): a lane quarter's warps share one scheduler, so a block takes as
// long with one quarter as with four.
// P: how N adds up the pooled values.  kPowSquare p = 2, kPowAny another p, kPowInf maxima (an
// instantiation each: choosing inside the loops spilled registers).
// FEW: some sender of the batch has a half of few query rows (kFewRows; an instantiation of its own: the
// others' loops are 2 % faster without the code for it).
enum { kPowSquare, kPowAny, kPowInf };

template <int D, int G, int PH, int P, bool FEW>
__global__ void __launch_bounds__(kThreadsTc, 1) k_accum_tc(const __grid_constant__ TcBatch bt) {
    constexpr int kTile = kTileRows * D * 2;
    extern __shared__ uint8_t smem_raw[];
    const Smem sm = carve<D, 2>(smem_raw, bt);
    Ctl* ctl = sm.ctl;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        init_ctl(ctl, 1, bt.wait_ns);
        my_units<2>(bt, ctl);
    }
    if (warp == 1) {
        tmem_alloc(&ctl->tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    const int n_units = ctl->units;
    Unit un = ctl->first;
    const int slots = 4 * bt.kbufs;

    if (warp == 0) {
        if (elect_one()) {
            int64_t kt = 0, qn = 0;   // K tiles and Q loads issued
            int st = 0;               // slot of the next K tile and its phase parity
            uint32_t ph = 0;
            bool ok = true;
            // the ones columns of the offset K-step, once per CTA
            mbar_arrive_expect_tx(&ctl->o_full, 128 * 32);
            tma_load_2d(sm.ones, &bt.omap, &ctl->o_full, 0, 0);
            int nc = 0, l = 0, g = 0, T = 0;
            for (int u = 0; u < n_units && ok; ++u, next_unit<2>(bt, un, nc)) {
                const TcMaps& mp = bt.maps[un.i];
                if (u == 0 || un.c == 0) {   // another group or row chunk: its Q
                    const TcSender& sd = bt.s[un.i];
                    nc = sd.n_blk2;
                    T = (int)sd.T;
                    l = un.s / bt.Hkv;
                    g = un.s % bt.Hkv;
                    if (!(ok = wait_bar(&ctl->q_empty, (uint32_t)((qn & 1) ^ 1), ctl, bt.err, 8))) break;
                    const int h0 = rc_begin(sd.halves, sd.n_rc2, un.rc);
                    load_q<D, 2>(bt, mp, sm, un.s, h0, rc_begin(sd.halves, sd.n_rc2, un.rc + 1) - h0, sd.q_rows,
                                 &ctl->q_full);
                    ++qn;
                }
                const int32_t t0 = un.c * kOut2 - kMargin;
                // the 5D map serves every tile (a change of map costs the TMA unit time: 150 against
                // 115 us for the loads of this pass with a map a tile); a last block that ends on one of the last
                // T mod 4 positions takes them through the other map, at half the rate
                const int32_t i0 = t0 / 4;
                const bool whole = t0 + kOut2 + 2 * kMargin <= T / 4 * 4 || T % 4 == 0;
                for (int j = 0; j < 4; ++j) {
                    if (!(ok = wait_bar(&ctl->k_empty[st], ph ^ 1u, ctl, bt.err, 9))) break;
                    // lane quarter w: positions t0 + 120 w + j + 4 i, i = 0 .. 31 (t0 a multiple of four)
                    uint8_t* dst = sm.k + (size_t)st * kTile;
                    mbar_arrive_expect_tx(&ctl->k_full[st], kTile);
                    if (whole) {
                        // (unrolled, one map: the issue time of these loads is on the path of the next block)
#pragma unroll
                        for (int w = 0; w < 4; ++w)
#pragma unroll
                            for (int kb = 0; kb < D / 64; ++kb)
                                tma_load_5d(dst + kb * kTileRows * 128 + w * 32 * 128, &mp.k[0], &ctl->k_full[st], 64 * kb,
                                            i0 + kOutW / 4 * w, j, g, l);
                    } else {
                        for (int w = 0; w < 4; ++w)
                            for (int kb = 0; kb < D / 64; ++kb)
                                tma_load_4d(dst + kb * kTileRows * 128 + w * 32 * 128, &mp.k[1], &ctl->k_full[st], 64 * kb,
                                            t0 + kOutW * w + j, g, l);
                    }
                    ++kt;
                    if (++st == slots) { st = 0; ph ^= 1u; }
                }
            }
            for (int64_t k = kt - slots > 0 ? kt - slots : 0; k < kt; ++k)
                drain_wait(&ctl->k_full[k % slots], (uint32_t)((k / slots) & 1));
            if (qn > 0) drain_wait(&ctl->q_full, (uint32_t)((qn - 1) & 1));
            drain_wait(&ctl->o_full, 0);
        }
    } else if (warp <= 2) {
        if (elect_one()) {
            const int me = warp - 1;
            uint32_t qn = 0;             // Q loads consumed
            uint32_t n = 0;              // rounds of the four accumulator buffers issued
            int st0 = 0;                 // slot of the block's first K tile and its phase parity
            uint32_t ph = 0;
            bool ok = wait_bar(&ctl->o_full, 0, ctl, bt.err, 15);
            const uint64_t ones_desc = smem_desc_sw32(smem_u32(sm.ones)), ext_desc = smem_desc_sw32(smem_u32(sm.ext));
            const uint32_t ext_hi = (uint32_t)(ext_desc >> 32), ext_lo = (uint32_t)ext_desc;
            const uint64_t qd = smem_desc_sw128(smem_u32(sm.q));
            const uint32_t hi = (uint32_t)(qd >> 32), q_lo = (uint32_t)qd;
            const uint32_t k_lo = (uint32_t)smem_desc_sw128(smem_u32(sm.k));
            const uint32_t q_blk = (uint32_t)bt.rows2 * 128 >> 4;
            constexpr uint32_t idesc = idesc_bf16_f32(128, 128);
            int nc = 0, nh = 0;
            uint32_t id_last = idesc;    // of the row chunk's last half: columns up to the last query row's 32
            for (int u = 0; u < n_units && ok; ++u, next_unit<2>(bt, un, nc)) {
                if (u == 0 || un.c == 0) {   // another group or row chunk: its Q
                    const TcSender& sd = bt.s[un.i];
                    nc = sd.n_blk2;
                    const int h1 = rc_begin(sd.halves, sd.n_rc2, un.rc + 1);
                    nh = h1 - rc_begin(sd.halves, sd.n_rc2, un.rc);
                    id_last = idesc_bf16_f32(128, min(kRowHalf, (sd.R - (h1 - 1) * kRowHalf + 31) & ~31));
                    if (u > 0) umma_commit(&ctl->q_empty);
                    if (!(ok = wait_bar(&ctl->q_full, qn & 1, ctl, bt.err, 10))) break;
                    ++qn;
                }
                for (int h = 0; h < nh && ok; ++h, ++n) {
                    const uint32_t id = h == nh - 1 ? id_last : idesc;
                    for (int j = me; j < 4; j += 2) {
                        if (h == 0 && !(ok = wait_bar(&ctl->k_full[st0 + j], ph, ctl, bt.err, 11))) break;
                        if (!(ok = wait_bar(&ctl->t_empty[j], (n & 1) ^ 1, ctl, bt.err, 12))) break;
                        tc_fence_after();
                        mma_d<D>(tmem + j * 128, k_lo + (uint32_t)(st0 + j) * (kTile >> 4), kTileRows * 128 >> 4,
                                 q_lo + h * (kRowHalf * 128 >> 4), q_blk, hi, id);
                        // one more K-step: ones (positions) x offset terms (rows) adds (centre - offset) / scale
                        // to every logit, so the epilogue needs only exp2(scale * D - centre)
                        umma_bf16(tmem + j * 128, ones_desc, desc64(ext_lo + h * (kRowHalf * 32 >> 4), ext_hi), id, 1u);
                        umma_commit(&ctl->t_full[j]);
                        if (h == nh - 1) umma_commit(&ctl->k_empty[st0 + j]);
                    }
                }
                st0 += 4;
                if (st0 == slots) { st0 = 0; ph ^= 1u; }
            }
            umma_commit(&ctl->drain[me]);
            drain_wait(&ctl->drain[me], 0);
        }
    } else if (warp >= kEpi0) {
        const int q = (warp - kEpi0) >> 2, sp = warp & 3;   // column quarter, TMEM lane quarter
        const uint32_t ta = tmem + ((uint32_t)(sp * 32) << 16) + 32 * q;
        float4* xch = reinterpret_cast<float4*>(sm.epi) + q * 256 + sp * 32 + lane;   // [column quarter][U, N][lane quarter][lane]
        const uint64_t cc = pack2(bt.sl2e, bt.sl2e);
        uint32_t n = 0, nu = 0;                  // parities: rounds of the four buffers, blocks so far
        bool ok = true;
        for (int left = n_units; left > 0 && ok;) {
            // the run of blocks of one group and row chunk (nothing but positions changes in it)
            const TcSender& sd = bt.s[un.i];
            const int h0 = rc_begin(sd.halves, sd.n_rc2, un.rc);
            const int nh = rc_begin(sd.halves, sd.n_rc2, un.rc + 1) - h0;
            const int R = sd.R - h0 * kRowHalf;  // query rows from the row chunk's first on
            const bool few = FEW && sd.few;
            const int T = (int)sd.T, nc = sd.n_blk2, run = min(left, nc - un.c);
            const float cen = (float)offset_centre(T, G);
            const uint64_t ncen = pack2(-cen, -cen);
            int pos = un.c * kOut2 + kOutW * sp - kMargin + 4 * lane;
            left -= run;
            un.c += run - 1;
            next_unit<2>(bt, un, nc);
            for (int k = 0; k < run && ok; ++k, pos += kOut2) {
                const int first = pos - 4 * lane;
                const bool all_valid = first >= 0 && first + 128 <= T;
                float us[4] = {0.f, 0.f, 0.f, 0.f}, ns[4] = {0.f, 0.f, 0.f, 0.f};   // per position: sums over tokens
                // N of position j takes two tokens' pooled values
                auto add_n = [&](int j, float o0, float o1) {
                    if (P == kPowSquare) ns[j] = fmaf(o0, o0, fmaf(o1, o1, ns[j]));
                    else if (P == kPowInf) ns[j] = fmaxf(ns[j], fmaxf(o0, o1));
                    else ns[j] += pow_p(o0, bt.p) + pow_p(o1, bt.p);
                };
                // Pool and the sums of two tokens (one pair of each of the four positions)
                auto pool_pair = [&](const auto& b, int i) {
                    float x0[4], x1[4], o0[4], o1[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        unpack2(b[j][i], x0[j], x1[j]);
                        us[j] += x0[j] + x1[j];
                    }
                    pool4<PH>(x0, o0);
                    pool4<PH>(x1, o1);
#pragma unroll
                    for (int j = 0; j < 4; ++j) add_n(j, o0[j], o1[j]);
                };
                // One round of the four buffers: the first `chunks` chunks of the columns from `t` on, TOK tokens
                // each.  EDGE: positions outside [0, T) are masked.  LAP: exp2 of a chunk's four tiles
                // interleaved with Pool of the chunk before it.  Unpooled sums (PH = 0) need no neighbours and
                // are taken load by load.
                auto round = [&](auto edge, auto lap, auto tok, uint32_t t, int chunks) {
                    constexpr bool EDGE = decltype(edge)::value, LAP = decltype(lap)::value;
                    constexpr int kTok = decltype(tok)::value, kChunks = 32 / (kTok * G), kPairs = kTok / 2;
                    constexpr int kCols = kTok * G < 16 ? kTok * G : 16;   // columns of a load
                    uint64_t b[LAP ? 2 : 1][4][kPairs];
#pragma unroll(LAP ? kChunks : 1)
                    for (int c = 0; c < (LAP || kChunks == 1 ? kChunks : chunks); ++c) {
                        auto& bc = b[LAP ? c & 1 : 0];
                        const bool end = c == (LAP || kChunks == 1 ? kChunks : chunks) - 1;
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (c == 0) {
                                if (!(ok = wait_bar(&ctl->t_full[j], n, ctl, bt.err, 13))) return;
                                tc_fence_after();
                            }
#pragma unroll
                            for (int x = 0; x < kTok * G; x += kCols) {
                                float v[kCols];
                                tmem_ldn(t + j * 128 + c * kTok * G + x, v);
                                if (LAP && c > 0 && (j & 1)) pool_pair(b[LAP ? (c & 1) ^ 1 : 0], j >> 1);
                                tmem_wait_ld(v);
                                if (end && x + kCols == kTok * G) {   // registers hold the rest
                                    tc_fence_before();
                                    __syncwarp();
                                    if (lane == 0) mbar_arrive(&ctl->t_empty[j]);
                                }
                                uint64_t* bx = bc[j] + x / (2 * G);
                                head_sums<G>(v, cc, ncen, bx);
                                if (EDGE) {
                                    const bool valid = pos + j >= 0 && pos + j < T;
#pragma unroll
                                    for (int i = 0; i < kCols / (2 * G); ++i) bx[i] = valid ? bx[i] : 0ull;
                                }
                                if (PH == 0) {
#pragma unroll
                                    for (int i = 0; i < kCols / (2 * G); ++i) {
                                        float x0, x1;
                                        unpack2(bx[i], x0, x1);
                                        us[j] += x0 + x1;
                                        add_n(j, x0, x1);
                                    }
                                }
                            }
                        }
                        if (PH > 0 && (!LAP || c == kChunks - 1)) {
#pragma unroll
                            for (int i = 0; i < kPairs; ++i) pool_pair(bc, i);
                        }
                    }
                };
                for (int h = 0; h < nh; ++h, n ^= 1) {
                    // A half of more than kFewRows rows, or of a sender of many: 32 columns a warp.  For d = 128 a buffer's are read one
                    // after the other (eight tokens at a time for G < 4, 16 columns a load) and go back to the
                    // MMA, which takes as long as the reading, before the next buffer's.  For d = 64 the MMA takes
                    // half that, so buffers can be held longer: four tokens' columns at a time, interleaved
                    // with Pool (143 -> 137 us for d64; d = 128 156 -> 168).
                    // Fewer rows, or G = 1, where eight tokens fill eight columns: eights of columns, as many for each of
                    // the four warps of a lane quarter.
                    const int rows = R - h * kRowHalf;
                    constexpr bool kLap = D == 64 && PH > 0, kEights = G == 1 && !kLap;
                    constexpr std::integral_constant<int, kLap ? 4 : 8> tok{};
                    constexpr std::integral_constant<int, 8 / G> tok8{};
                    constexpr std::bool_constant<kLap> lap{};
                    constexpr std::false_type no{};
                    constexpr std::true_type yes{};
                    constexpr int kChunks = 32 / (tok.value * G);
                    const bool wide = !kEights && (!FEW || !few || rows > kFewRows);
                    const int eights = min(4, (rows + 31) >> 5), col = 8 * eights * q;
                    if (wide ? 32 * q >= rows : col >= rows) {   // no columns
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (!(ok = wait_bar(&ctl->t_full[j], n, ctl, bt.err, 13))) break;
                            if (lane == 0) mbar_arrive(&ctl->t_empty[j]);
                        }
                    } else if (wide) {
                        if (all_valid) round(no, lap, tok, ta, kChunks);
                        else round(yes, lap, tok, ta, kChunks);
                    } else if (FEW || kEights) {
                        const int n8 = min(eights, (rows - col + 7) >> 3);
                        if (all_valid) round(no, no, tok8, ta - 32 * q + col, n8);
                        else round(yes, no, tok8, ta - 32 * q + col, n8);
                    }
                    if (!ok) break;
                }
                // hand the block's sums to warp 3 (it has read the last block's long ago)
                if (!ok || !(ok = wait_bar(&ctl->xe, nu ^ 1, ctl, bt.err, 7))) break;
                xch[0] = make_float4(us[0], us[1], us[2], us[3]);
                xch[128] = make_float4(ns[0], ns[1], ns[2], ns[3]);
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->xb);
                nu ^= 1;
            }
        }
    } else {
        // ---------------- warp 3: the column quarters' sums of a block, added in a fixed order ----------------
        const float4* xch = reinterpret_cast<const float4*>(sm.epi) + lane;   // [column quarter][U, N][lane quarter][lane]
        const int nS = bt.nL * bt.Hkv;
        bool ok = true;
        float* part = nullptr;                   // U partials of the current group and row chunk
        int64_t nST = 0;                         // distance between the U and N partials
        int T = 0, nc = 0;
        for (int u = 0; u < n_units && ok; ++u, next_unit<2>(bt, un, nc)) {
            if (u == 0 || un.c == 0) {
                const TcSender& sd = bt.s[un.i];
                nST = (int64_t)nS * sd.T_pad;
                part = sd.part + 2 * un.rc * nST + (int64_t)un.s * sd.T_pad;
                T = (int)sd.T;
                nc = sd.n_blk2;
            }
            if (!(ok = wait_bar(&ctl->xb, (uint32_t)u & 1, ctl, bt.err, 14))) break;
            auto add = [](float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); };
            auto mx = [](float4 a, float4 b) {
                return make_float4(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z), fmaxf(a.w, b.w));
            };
            auto add_n = [&](float4 a, float4 b) { return P == kPowInf ? mx(a, b) : add(a, b); };
#pragma unroll
            for (int sp = 0; sp < 4; ++sp) {
                float4 x[4], y[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x[k] = xch[(8 * k + sp) * 32];
                    y[k] = xch[(8 * k + 4 + sp) * 32];
                }
                const float4 u4 = add(add(x[0], x[1]), add(x[2], x[3])), n4 = add_n(add_n(y[0], y[1]), add_n(y[2], y[3]));
                const int pos = un.c * kOut2 + kOutW * sp - kMargin + 4 * lane;
                if (lane >= 1 && lane <= 30 && pos < T) {   // rows are padded to a multiple of four positions
                    *reinterpret_cast<float4*>(part + pos) = u4;
                    *reinterpret_cast<float4*>(part + nST + pos) = n4;
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->xe);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// Pass 2 for senders of few blocks of 480 positions: blocks of one tile, a position a lane.  Lane
// quarter w of block c covers positions 104 c + 26 w - 3 .. + 31, lanes 3 to 28 its outputs.  Pool takes
// two to four shuffles a value where k_accum_tc takes six for four, and 104 of a tile's 128
// positions are outputs instead of 120, but four times as many blocks fill the SMs, and a sender of less than 480
// positions has no lane quarters without any.
// P is chosen inside (`mode`): these are calls of few exponentials, bound by latencies (K and Q of a
// block arriving, its MMA, its round of exponentials one after the other).
template <int PH>
__device__ __forceinline__ float pool1(float x) {
    constexpr unsigned kAll = 0xffffffffu;
    if (PH == 0) return x;
    const float y = fmax3(__shfl_up_sync(kAll, x, 1), x, __shfl_down_sync(kAll, x, 1));
    if (PH == 1) return y;
    return fmax3(__shfl_up_sync(kAll, y, PH - 1), y, __shfl_down_sync(kAll, y, PH - 1));
}

template <int D, int G, int PH>
__global__ void __launch_bounds__(kThreadsTc, 1) k_narrow_tc(const __grid_constant__ TcBatch bt) {
    constexpr int kTile = kTileRows * D * 2;
    extern __shared__ uint8_t smem_raw[];
    Smem sm;   // [Q, offset terms] twice, ones, K tiles, Ctl, exchange of sums
    const uint32_t q_bytes = (uint32_t)bt.rows2 * (D * 2 + 32);
    sm.q = align1024(smem_raw);
    sm.ext = sm.q + (size_t)bt.rows2 * D * 2;
    sm.ones = sm.q + 2 * q_bytes;
    sm.k = sm.ones + 128 * 32;
    sm.ctl = reinterpret_cast<Ctl*>(sm.k + (size_t)bt.kbufs * kTile);
    sm.epi = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(sm.ctl) + 512);
    Ctl* ctl = sm.ctl;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        init_ctl(ctl, 2, bt.wait_ns);
        my_units<2>(bt, ctl);
    }
    if (warp == 1) {
        tmem_alloc(&ctl->tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = ctl->tmem_base;
    const int n_units = ctl->units;
    Unit un = ctl->first;
    const int slots = bt.kbufs;

    if (warp == 0) {
        // ---------------- TMA producer ----------------
        if (elect_one()) {
            int64_t kt = 0, qn = 0;   // K tiles and Q loads issued
            int st = 0;               // slot of the next K tile and its phase parity
            uint32_t ph = 0;
            bool ok = true;
            mbar_arrive_expect_tx(&ctl->o_full, 128 * 32);
            tma_load_2d(sm.ones, &bt.omap, &ctl->o_full, 0, 0);
            int nc = 0, l = 0, g = 0;
            for (int u = 0; u < n_units && ok; ++u, next_unit<2>(bt, un, nc)) {
                const TcMaps& mp = bt.maps[un.i];
                if (u == 0 || un.c == 0) {   // another group or row chunk: its Q
                    const TcSender& sd = bt.s[un.i];
                    nc = sd.n_blk2;
                    l = un.s / bt.Hkv;
                    g = un.s % bt.Hkv;
                    const uint32_t b = (uint32_t)qn & 1;
                    if (!(ok = wait_bar(&ctl->q2_empty[b], (uint32_t)((qn >> 1) & 1) ^ 1u, ctl, bt.err, 8))) break;
                    const int h0 = rc_begin(sd.halves, sd.n_rc2, un.rc);
                    Smem to = sm;
                    to.q += b * q_bytes;
                    to.ext += b * q_bytes;
                    load_q<D, 2>(bt, mp, to, un.s, h0, rc_begin(sd.halves, sd.n_rc2, un.rc + 1) - h0, sd.q_rows,
                                 &ctl->q2_full[b]);
                    ++qn;
                }
                if (!(ok = wait_bar(&ctl->k_empty[st], ph ^ 1u, ctl, bt.err, 9))) break;
                mbar_arrive_expect_tx(&ctl->k_full[st], kTile);
                for (int w = 0; w < 4; ++w)
                    for (int kb = 0; kb < D / 64; ++kb)
                        tma_load_4d(sm.k + (size_t)st * kTile + kb * kTileRows * 128 + w * 32 * 128, &mp.k[1],
                                    &ctl->k_full[st], 64 * kb, un.c * kOutN + kOutNW * w - kMarginN, g, l);
                ++kt;
                if (++st == slots) { st = 0; ph ^= 1u; }
            }
            for (int64_t k = kt - slots > 0 ? kt - slots : 0; k < kt; ++k)
                drain_wait(&ctl->k_full[k % slots], (uint32_t)((k / slots) & 1));
            for (int64_t k = qn - 2 > 0 ? qn - 2 : 0; k < qn; ++k) drain_wait(&ctl->q2_full[k & 1], (uint32_t)((k >> 1) & 1));
            drain_wait(&ctl->o_full, 0);
        }
    } else if (warp <= 2) {
        // ---------------- MMA issuers: alternate buffers ----------------
        if (elect_one()) {
            const uint32_t me = (uint32_t)warp - 1;
            uint32_t qn = 0, n = 0;      // Q loads consumed; accumulator buffers filled by both issuers
            int st = 0;                  // slot of the next K tile and its phase parity
            uint32_t ph = 0;
            bool ok = wait_bar(&ctl->o_full, 0, ctl, bt.err, 15);
            const uint64_t ones_desc = smem_desc_sw32(smem_u32(sm.ones)), ext_desc = smem_desc_sw32(smem_u32(sm.ext));
            const uint32_t ext_hi = (uint32_t)(ext_desc >> 32), ext_lo = (uint32_t)ext_desc;
            const uint64_t qd = smem_desc_sw128(smem_u32(sm.q));
            const uint32_t hi = (uint32_t)(qd >> 32);
            uint32_t q_lo = 0, e_lo = 0;   // of the current Q buffer
            const uint32_t k_lo = (uint32_t)smem_desc_sw128(smem_u32(sm.k));
            const uint32_t q_blk = (uint32_t)bt.rows2 * 128 >> 4;
            constexpr uint32_t idesc = idesc_bf16_f32(128, 128);
            uint32_t nh = 0, id_last = idesc;
            int nc = 0;
            for (int u = 0; u < n_units && ok; ++u, next_unit<2>(bt, un, nc)) {
                if (u == 0 || un.c == 0) {   // another group or row chunk: its Q
                    const TcSender& sd = bt.s[un.i];
                    nc = sd.n_blk2;
                    const int h1 = rc_begin(sd.halves, sd.n_rc2, un.rc + 1);
                    nh = h1 - rc_begin(sd.halves, sd.n_rc2, un.rc);
                    id_last = idesc_bf16_f32(128, min(kRowHalf, (sd.R - (h1 - 1) * kRowHalf + 31) & ~31));
                    if (u > 0) umma_commit(&ctl->q2_empty[(qn - 1) & 1]);
                    if (!(ok = wait_bar(&ctl->q2_full[qn & 1], (qn >> 1) & 1, ctl, bt.err, 10))) break;
                    q_lo = (uint32_t)qd + (qn & 1) * (q_bytes >> 4);
                    e_lo = ext_lo + (qn & 1) * (q_bytes >> 4);
                    ++qn;
                }
                if (!(ok = wait_bar(&ctl->k_full[st], ph, ctl, bt.err, 11))) break;
                for (uint32_t h = (n ^ me) & 1; h < nh; h += 2) {
                    const uint32_t x = n + h, buf = x & 3, id = h == nh - 1 ? id_last : idesc;
                    if (!(ok = wait_bar(&ctl->t_empty[buf], ((x >> 2) & 1) ^ 1, ctl, bt.err, 12))) break;
                    tc_fence_after();
                    mma_d<D>(tmem + buf * 128, k_lo + (uint32_t)st * (kTile >> 4), kTileRows * 128 >> 4,
                             q_lo + h * (kRowHalf * 128 >> 4), q_blk, hi, id);
                    umma_bf16(tmem + buf * 128, ones_desc, desc64(e_lo + h * (kRowHalf * 32 >> 4), ext_hi), id, 1u);
                    umma_commit(&ctl->t_full[buf]);
                }
                if (!ok) break;
                n += nh;
                umma_commit(&ctl->k_empty[st]);
                if (++st == slots) { st = 0; ph ^= 1u; }
            }
            umma_commit(&ctl->drain[me]);
            drain_wait(&ctl->drain[me], 0);
        }
    } else if (warp >= kEpi0) {
        // ---------------- epilogue: a position a lane, a share of every buffer's columns a warp ----------------
        const int q = (warp - kEpi0) >> 2, sp = warp & 3;   // column share, TMEM lane quarter
        const uint32_t ta = tmem + ((uint32_t)(sp * 32) << 16);
        float* xch = sm.epi + q * 256 + sp * 32 + lane;     // [column share][U, N][lane quarter][lane]
        const uint64_t cc = pack2(bt.sl2e, bt.sl2e);
        const int mode = bt.p_inf ? kPowInf : (bt.p == 2.f ? kPowSquare : kPowAny);
        uint32_t n = 0;                          // accumulator buffers consumed
        bool ok = true;
        int nc = 0, nh = 0, R = 0, T = 0;
        uint64_t ncen = 0;
        for (int u = 0; u < n_units && ok; ++u, next_unit<2>(bt, un, nc)) {
            if (u == 0 || un.c == 0) {
                const TcSender& sd = bt.s[un.i];
                nc = sd.n_blk2;
                const int h0 = rc_begin(sd.halves, sd.n_rc2, un.rc);
                nh = rc_begin(sd.halves, sd.n_rc2, un.rc + 1) - h0;
                R = sd.R - h0 * kRowHalf;
                T = (int)sd.T;
                const float cen = (float)offset_centre(T, G);
                ncen = pack2(-cen, -cen);
            }
            const int pos = un.c * kOutN + kOutNW * sp - kMarginN + lane;
            const bool valid = pos >= 0 && pos < T;
            float us = 0.f, ns = 0.f;
            // COLS columns from `t` on: their tokens' values, Pool and the sums
            auto take = [&](auto cols, uint32_t t, uint32_t buf, bool last) {
                constexpr int kCols = decltype(cols)::value;
                float v[kCols];
                tmem_ldn(t, v);
                tmem_wait_ld(v);
                if (last) {   // registers hold the rest
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&ctl->t_empty[buf]);
                }
                uint64_t b[kCols / (2 * G)];
                head_sums<G>(v, cc, ncen, b);
#pragma unroll
                for (int i = 0; i < kCols / (2 * G); ++i) {
                    float x0, x1;
                    unpack2(valid ? b[i] : 0ull, x0, x1);
                    us += x0 + x1;
                    const float o0 = pool1<PH>(x0), o1 = pool1<PH>(x1);
                    if (mode == kPowSquare) ns = fmaf(o0, o0, fmaf(o1, o1, ns));
                    else if (mode == kPowInf) ns = fmaxf(ns, fmaxf(o0, o1));
                    else ns += pow_p(o0, bt.p) + pow_p(o1, bt.p);
                }
            };
            for (int h = 0; h < nh; ++h, ++n) {
                const uint32_t buf = n & 3;
                if (!(ok = wait_bar(&ctl->t_full[buf], (n >> 2) & 1, ctl, bt.err, 13))) break;
                tc_fence_after();
                // eights of columns, as many for each of the four warps of a lane quarter
                const int rows = R - h * kRowHalf, eights = min(4, (rows + 31) >> 5), col = 8 * eights * q;
                int n8 = min(eights, (rows - col + 7) >> 3);
                if (n8 <= 0 && lane == 0) mbar_arrive(&ctl->t_empty[buf]);   // none
                uint32_t t = ta + buf * 128 + col;
                for (; n8 >= 2; n8 -= 2, t += 16) take(std::integral_constant<int, 16>{}, t, buf, n8 == 2);
                if (n8 == 1) take(std::integral_constant<int, 8>{}, t, buf, true);
            }
            // hand the block's sums to warp 3 (it has read the last block's long ago)
            if (!ok || !(ok = wait_bar(&ctl->xe, ((uint32_t)u & 1) ^ 1, ctl, bt.err, 7))) break;
            xch[0] = us;
            xch[128] = ns;
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->xb);
        }
    } else {
        // ---------------- warp 3: the column shares' sums of a block, added in a fixed order ----------------
        const float* xch = sm.epi + lane;        // [column share][U, N][lane quarter][lane]
        const int nS = bt.nL * bt.Hkv;
        bool ok = true;
        float* part = nullptr;                   // U partials of the current group and row chunk
        int64_t nST = 0;                         // distance between the U and N partials
        int T = 0, nc = 0;
        for (int u = 0; u < n_units && ok; ++u, next_unit<2>(bt, un, nc)) {
            if (u == 0 || un.c == 0) {
                const TcSender& sd = bt.s[un.i];
                nST = (int64_t)nS * sd.T_pad;
                part = sd.part + 2 * un.rc * nST + (int64_t)un.s * sd.T_pad;
                T = (int)sd.T;
                nc = sd.n_blk2;
            }
            if (!(ok = wait_bar(&ctl->xb, (uint32_t)u & 1, ctl, bt.err, 14))) break;
#pragma unroll
            for (int sp = 0; sp < 4; ++sp) {
                float x[4], y[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    x[k] = xch[(8 * k + sp) * 32];
                    y[k] = xch[(8 * k + 4 + sp) * 32];
                }
                const int pos = un.c * kOutN + kOutNW * sp - kMarginN + lane;
                if (lane >= kMarginN && lane < kMarginN + kOutNW && pos < T) {
                    part[pos] = (x[0] + x[1]) + (x[2] + x[3]);
                    part[nST + pos] = bt.p_inf ? fmaxf(fmaxf(y[0], y[1]), fmaxf(y[2], y[3])) : (y[0] + y[1]) + (y[2] + y[3]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->xe);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) tmem_dealloc(tmem, kTmemCols);
}

// ---------------------------------------------------------------------------
// launches
// ---------------------------------------------------------------------------
constexpr size_t kSmemMax = 227 * 1024;

// Raises a kernel's dynamic shared-memory limit to the SM's, once per device (`done`: a bit each;
// the call takes about a microsecond of host time, and setting it twice is harmless).
template <typename K>
cudaError_t allow_smem(K kernel, std::atomic<uint64_t>& done) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev < 64 ? uint64_t(1) << dev : 0;
    if (done.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
    return e;
}

inline size_t smem1_bytes(int d, int rows, int stages) {
    return 1024 + (size_t)rows * d * 2 + (size_t)stages * kTileRows * d * 2 + 512;
}

inline size_t smem2_bytes(int d, int rows, int kbufs) {
    return 1024 + (size_t)rows * (d * 2 + 32) + 128 * 32 + (size_t)kbufs * 4 * kTileRows * d * 2 + 512 + 4 * 8 * 128 * 4;
}

inline size_t smem_narrow_bytes(int d, int rows, int tiles) {
    return 1024 + (size_t)2 * rows * (d * 2 + 32) + 128 * 32 + (size_t)tiles * kTileRows * d * 2 + 512 + 4 * 8 * 32 * 4;
}

template <int D, int G, int PH, int P, bool FEW>
cudaError_t launch_accum_few(const TcBatch& tb, int grid, cudaStream_t st) {
    const size_t smem = smem2_bytes(D, tb.rows2, tb.kbufs);
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = allow_smem(k_accum_tc<D, G, PH, P, FEW>, done);
    if (e != cudaSuccess) return e;
    k_accum_tc<D, G, PH, P, FEW><<<grid, kThreadsTc, smem, st>>>(tb);
    return cudaGetLastError();
}

template <int D, int G, int PH, int P>
cudaError_t launch_accum(const TcBatch& tb, int grid, cudaStream_t st) {
    return tb.few ? launch_accum_few<D, G, PH, P, true>(tb, grid, st) : launch_accum_few<D, G, PH, P, false>(tb, grid, st);
}

template <int D, int G, int P>
cudaError_t launch_accum_gp(const TcBatch& tb, int grid, cudaStream_t st) {
    switch (tb.ph) {
        case 0: return launch_accum<D, G, 0, P>(tb, grid, st);
        case 1: return launch_accum<D, G, 1, P>(tb, grid, st);
        case 2: return launch_accum<D, G, 2, P>(tb, grid, st);
        case 3: return launch_accum<D, G, 3, P>(tb, grid, st);
    }
    return cudaErrorInvalidValue;
}

template <int D, int G>
cudaError_t launch_accum_g(const TcBatch& tb, int grid, cudaStream_t st) {
    if (tb.p == 2.f) return launch_accum_gp<D, G, kPowSquare>(tb, grid, st);
    return tb.p_inf ? launch_accum_gp<D, G, kPowInf>(tb, grid, st) : launch_accum_gp<D, G, kPowAny>(tb, grid, st);
}

template <int D, int G, int PH>
cudaError_t launch_narrow(const TcBatch& tb, int grid, cudaStream_t st) {
    const size_t smem = smem_narrow_bytes(D, tb.rows2, tb.kbufs);
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = allow_smem(k_narrow_tc<D, G, PH>, done);
    if (e != cudaSuccess) return e;
    k_narrow_tc<D, G, PH><<<grid, kThreadsTc, smem, st>>>(tb);
    return cudaGetLastError();
}

template <int D, int G>
cudaError_t launch_narrow_g(const TcBatch& tb, int grid, cudaStream_t st) {
    switch (tb.ph) {
        case 0: return launch_narrow<D, G, 0>(tb, grid, st);
        case 1: return launch_narrow<D, G, 1>(tb, grid, st);
        case 2: return launch_narrow<D, G, 2>(tb, grid, st);
        case 3: return launch_narrow<D, G, 3>(tb, grid, st);
    }
    return cudaErrorInvalidValue;
}

template <int D, int NH>
cudaError_t launch_stats(const TcBatch& tb, int grid, cudaStream_t st) {
    const size_t smem = smem1_bytes(D, tb.rows1, tb.stages1);
    static std::atomic<uint64_t> done{0};
    const cudaError_t e = allow_smem(k_stats_tc<D, NH>, done);
    if (e != cudaSuccess) return e;
    k_stats_tc<D, NH><<<grid, kThreadsTc, smem, st>>>(tb);
    return cudaGetLastError();
}

}  // namespace

namespace tc {
template <int D>
cudaError_t launch_accum_d(const TcBatch& tb, int grid, cudaStream_t st) {
    if (tb.G == 4) return launch_accum_g<D, 4>(tb, grid, st);
    return tb.G == 2 ? launch_accum_g<D, 2>(tb, grid, st) : launch_accum_g<D, 1>(tb, grid, st);
}

template <int D>
cudaError_t launch_narrow_d(const TcBatch& tb, int grid, cudaStream_t st) {
    if (tb.G == 4) return launch_narrow_g<D, 4>(tb, grid, st);
    return tb.G == 2 ? launch_narrow_g<D, 2>(tb, grid, st) : launch_narrow_g<D, 1>(tb, grid, st);
}

template <int D>
cudaError_t launch_stats_d(const TcBatch& tb, int grid, cudaStream_t st) {
    if (tb.rows1 <= kRowHalf) return launch_stats<D, 1>(tb, grid, st);
    if (tb.rows1 <= 2 * kRowHalf) return launch_stats<D, 2>(tb, grid, st);
    return launch_stats<D, kHalves1>(tb, grid, st);
}

// This file is compiled in three parts, at the same time: with CB_TC_PART = 64 and 128 the kernels of
// that head dimension, with 0 everything else (without it, all in one).
#if !defined(CB_TC_PART) || CB_TC_PART == 64
template cudaError_t launch_stats_d<64>(const TcBatch&, int, cudaStream_t);
template cudaError_t launch_accum_d<64>(const TcBatch&, int, cudaStream_t);
template cudaError_t launch_narrow_d<64>(const TcBatch&, int, cudaStream_t);
#else
extern template cudaError_t launch_stats_d<64>(const TcBatch&, int, cudaStream_t);
extern template cudaError_t launch_accum_d<64>(const TcBatch&, int, cudaStream_t);
extern template cudaError_t launch_narrow_d<64>(const TcBatch&, int, cudaStream_t);
#endif
#if !defined(CB_TC_PART) || CB_TC_PART == 128
template cudaError_t launch_stats_d<128>(const TcBatch&, int, cudaStream_t);
template cudaError_t launch_accum_d<128>(const TcBatch&, int, cudaStream_t);
template cudaError_t launch_narrow_d<128>(const TcBatch&, int, cudaStream_t);
#else
extern template cudaError_t launch_stats_d<128>(const TcBatch&, int, cudaStream_t);
extern template cudaError_t launch_accum_d<128>(const TcBatch&, int, cudaStream_t);
extern template cudaError_t launch_narrow_d<128>(const TcBatch&, int, cudaStream_t);
#endif
}  // namespace tc

#if !defined(CB_TC_PART) || CB_TC_PART == 0
// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {
using namespace tc;

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
    std::call_once(g_encode_once, [] {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
        else
            cudaGetLastError();
    });
    return g_encode;
}

// bf16 tensor map of `rank` dimensions (innermost first); strides in bytes of dims 1..rank-1; of
// dimension 1 the box takes every step-th element.
bool encode_nd(CUtensorMap* m, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides_bytes,
               const cuuint32_t* box, CUtensorMapSwizzle swizzle, cuuint32_t step = 1) {
    auto fn = encoder();
    if (!fn || !base) return false;
    const cuuint32_t es[5] = {1, step, 1, 1, 1};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides_bytes, box,
              es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_4d(CUtensorMap* m, const void* base, const cuuint64_t dims[4], const cuuint64_t strides_bytes[3],
               const cuuint32_t box[4]) {
    return encode_nd(m, base, 4, dims, strides_bytes, box, CU_TENSOR_MAP_SWIZZLE_128B);
}

// Positions of a pass-1 chunk of a sender of T positions and nS groups.  Chunks of 2048 positions
// leave half as many partials to write and merge as chunks of 1024, but units too few to spread
// evenly over the SMs unless there are many.  The combine kernel takes 10.7 against 12.4 us for 288
// groups, T = 8192 (1152 units), 44 against 73 for three senders of T = 16384 with 512 rows, 13
// against 19 for 64 groups, T = 65536 (2048 units; pass 1 208 against 204 there, the same
// elsewhere); below the line pass 1 loses more: 135 against 126 us for 192 groups, 2 x T = 7001
// (768 units a sender), 146 against 139 for 96 groups, T = 6001 (288).  The rule reads the sender
// alone, so its scores do not depend on the call's others.
int32_t stats_chunk(int64_t T, int nS) {
    return nS * ((T + 2 * kChunk1 - 1) / (2 * kChunk1)) >= kLongChunkUnits ? 2 * kChunk1 : kChunk1;
}

// Whether pass 2 takes a sender of T positions in blocks of one tile, given its units (blocks of 480,
// groups and row chunks): a sender of few positions leaves lane quarters idle (d = 128, 20 layers x 8 groups,
// 5 x T = 103, 6 rows: 16 against 26 us; beyond the line, 29 x 8, T = 352, 389 rows 50 against 46; d = 64, whose
// rounds of 32 columns are better packed, beyond its line, 7 x 4, 5 x T = 212, 188 rows 17 against 16),
// and where four times as many blocks of one tile still fit a wave of 152 SMs they take a third of the time
// (2 x 4 groups, T = 952, 140 rows: pass 2 11.5 against 14).  The rule reads the sender alone, so its scores do
// not depend on the call's others; many senders of few units fill the SMs together, and then blocks of
// 480 would take up to a third less (8 of 4 x 8, T = 900, 240 rows: 64 units each, beyond the line, 34 against 39).
bool narrow_blocks(int head_dim, int64_t T, int64_t units) {
    return T <= (head_dim == 128 ? 3 : 2) * kOutN || units <= kNarrowUnits;
}

// CTAs of a pass of `units` units: one an SM, a multiple of the row-chunk count when every sender
// has the same one (CTAs k, k + grid / n_rc, ... then walk the same K tiles in step, so that a
// tile comes from DRAM once and from L2 for the other row chunks).
int pass_grid(int64_t units, int num_sms, int n_rc) {
    int g = num_sms;
    if (n_rc > 1 && n_rc <= g) g = g / n_rc * n_rc;
    return (int)(units < g ? units : g);
}

}  // namespace

bool tc_path_supported(int head_dim, int G, int pool_half) {
    return (head_dim == 64 || head_dim == 128) && (G == 1 || G == 2 || G == 4) && pool_half <= 3;
}

// Pass 1, combine, pass 2 on the tensor cores for senders [0, b.n) of `b`; the caller
// launches the finalize kernel.  `combine` is the shared statistics-combine launcher.
cudaError_t launch_score_tc(ScoreBatch& b, cudaStream_t st, int num_sms, uint32_t* err,
                            cudaError_t (*combine)(const ScoreBatch&, cudaStream_t)) {
    const int G = b.n_q_heads / b.n_kv_heads;
    const int nS = b.n_layers * b.n_kv_heads, d_head = b.head_dim;
    // Encode every tensor map first: if the driver rejects one (an unusual stride
    // pattern), nothing has been launched and the caller uses the mma.sync passes.
    std::vector<std::unique_ptr<TcBatch>> batches;
    std::vector<std::unique_ptr<TcMaps[]>> maps2;   // pass 2's tensor maps of each sub-batch
    // Sub-batches of at most kMaxTcSenders senders; paged senders are copied into the staging buffer
    // (contiguous [nL][Hkv][T][d]; by pass 1, or ahead of it where pages are short), which each
    // sub-batch reuses from its start, so a sub-batch also ends where its paged senders would
    // overflow the staging.
    std::vector<int> firsts;
    std::vector<std::unique_ptr<DepageBatch>> depages;
    for (int b0 = 0; b0 < b.n;) {
        int nb = 0;
        int64_t used = 0;
        while (b0 + nb < b.n && nb < kMaxTcSenders) {
            const ScoreSender& s = b.s[b0 + nb];
            const int64_t e = s.pm.pages ? (int64_t)nS * s.T * d_head : 0;
            if (e > 0 && (!b.stage || e > b.stage_elems)) {   // no room: the mma.sync passes read pages
                return cudaErrorNotSupported;
            }
            if (nb > 0 && used + e > b.stage_elems) break;
            used += e;
            ++nb;
        }
        firsts.push_back(b0);
        depages.emplace_back(new DepageBatch);   // (uninitialised, like the next: filled for its senders only)
        DepageBatch* dp = depages.back().get();
        dp->n = 0;
        dp->n_layers = b.n_layers;
        dp->n_kv_heads = b.n_kv_heads;
        dp->head_dim = d_head;
        dp->err = err;
        batches.emplace_back(new TcBatch);
        maps2.emplace_back(new TcMaps[nb]);
        TcBatch* tb = batches.back().get();
        tb->n = nb;
        b0 += nb;
        tb->nL = b.n_layers;
        tb->Hq = b.n_q_heads;
        tb->Hkv = b.n_kv_heads;
        tb->G = G;
        tb->log2g = G == 4 ? 2 : G - 1;
        tb->sl2e = b.scale_log2e;
        tb->p = b.p;
        tb->p_inf = b.p_inf;
        tb->ph = b.pool_half;
        tb->err = err;
        tb->max_rc1 = 1;
        tb->weight1 = 0;
        tb->paged = 0;
        int rows1 = kRowHalf;
        int64_t staged = 0;
        const int b_first = firsts.back();
        for (int k = 0; k < nb; ++k) {
            const ScoreSender& s = b.s[b_first + k];
            TcSender& d = tb->s[k];
            TcMaps &mp = tb->maps[k], &mp2 = maps2.back()[k];   // pass 1's and pass 2's maps
            // K as the passes read it: the sender's own tensor, or its staged copy (which pass 1 writes
            // itself when the pages are long enough)
            const uint16_t* kp = s.k;
            int64_t kl = s.ks_l, kh = s.ks_h, kpos = s.ks_p;
            const bool fused = s.pm.pages && s.pm.shift >= kMinPageShift && s.pm.n_pages < INT32_MAX;
            d.pages = fused ? s.pm.pages : nullptr;
            d.n_pages = fused ? (int32_t)s.pm.n_pages : 0;
            d.page_shift = s.pm.shift;
            tb->paged |= fused;
            if (s.pm.pages) {
                if (!fused) {
                    DepageSender& ds = dp->s[dp->n++];
                    ds.k = s.k;
                    ds.ks_l = s.ks_l;
                    ds.ks_h = s.ks_h;
                    ds.ks_p = s.ks_p;
                    ds.pm = s.pm;
                    ds.T = s.T;
                    ds.out = b.stage + staged;
                }
                kp = b.stage + staged;
                kpos = d_head;
                kh = s.T * d_head;
                kl = (int64_t)b.n_kv_heads * s.T * d_head;
                staged += kl * b.n_layers;
            }
            d.T = s.T;
            d.T_pad = part_row(s.T);
            d.m_self = s.kself ? s.m : 0;
            d.R = s.m * G;
            d.halves = (d.R + kRowHalf - 1) / kRowHalf;
            d.q_rows = d.halves > 1 ? kRowHalf : (d.R + 31) & ~31;
            d.chunk1 = stats_chunk(s.T, nS);
            d.n_chunk1 = (int32_t)(4 * ((s.T + d.chunk1 - 1) / d.chunk1));   // one partial per (chunk, column quarter)
            d.n_blk2 = (int32_t)((s.T + kOut2 - 1) / kOut2);
            d.n_rc1 = (d.halves + kHalves1 - 1) / kHalves1;
            d.n_rc2 = (d.halves + kHalves2 - 1) / kHalves2;
            d.narrow = narrow_blocks(d_head, s.T, (int64_t)nS * d.n_blk2 * d.n_rc2);
            d.few = (G > 1 || d_head == 64) && d.halves <= kFewHalves && d.R - (d.halves - 1) * kRowHalf <= kFewRows;
            if (d.narrow) d.n_blk2 = (int32_t)((s.T + kOutN - 1) / kOutN);
            d.stats = b.stats + s.stats_off;
            d.part = b.part + s.part_off;
            tb->max_rc1 = tb->max_rc1 > d.n_rc1 ? tb->max_rc1 : d.n_rc1;
            const int r1 = (d.halves + d.n_rc1 - 1) / d.n_rc1 * kRowHalf;
            rows1 = rows1 > r1 ? rows1 : r1;
            tb->weight1 += (int64_t)nS * (d.n_chunk1 / 4) * d.halves;
            const cuuint64_t kd[4] = {(cuuint64_t)d_head, (cuuint64_t)s.T, (cuuint64_t)b.n_kv_heads,
                                      (cuuint64_t)b.n_layers};
            const cuuint64_t ks[3] = {(cuuint64_t)kpos * 2, (cuuint64_t)kh * 2, (cuuint64_t)kl * 2};
            const cuuint32_t kbox[4] = {64, kTileRows, 1, 1};
            const cuuint64_t qd[4] = {(cuuint64_t)d_head, (cuuint64_t)b.n_q_heads, (cuuint64_t)s.m, (cuuint64_t)b.n_layers};
            const cuuint64_t qs[3] = {(cuuint64_t)s.qs_h * 2, (cuuint64_t)s.qs_t * 2, (cuuint64_t)s.qs_l * 2};
            const cuuint32_t qbox[4] = {64, (cuuint32_t)G, (cuuint32_t)(d.q_rows / G), 1};
            // offset terms [nS][rows padded to 128][16] written by the combine kernel
            const cuuint64_t rpad = (cuuint64_t)d.halves * kRowHalf;
            const cuuint64_t ed[3] = {(cuuint64_t)kExtCols, rpad, (cuuint64_t)nS};
            const cuuint64_t es[2] = {(cuuint64_t)kExtCols * 2, rpad * kExtCols * 2};
            const cuuint32_t ebox[3] = {(cuuint32_t)kExtCols, (cuuint32_t)d.q_rows, 1};
            // positions (i, j) = 4 i + j of whole groups of four (a sender of fewer than four positions has
            // none: one row of any, which no block loads), and every fourth position up to the last
            const cuuint64_t k5d[5] = {kd[0], (cuuint64_t)(s.T / 4 > 0 ? s.T / 4 : 1), (cuuint64_t)(s.T < 4 ? s.T : 4),
                                       kd[2], kd[3]};
            const cuuint64_t k5s[4] = {4 * ks[0], ks[0], ks[1], ks[2]};
            const cuuint32_t k5box[5] = {64, 32, 1, 1, 1};
            const cuuint32_t k32box[4] = {64, 32, 1, 1};
            bool ok4;
            if (d.narrow) {
                ok4 = encode_4d(&mp2.k[1], kp, kd, ks, k32box);
            } else {
                ok4 = encode_nd(&mp2.k[0], kp, 5, k5d, k5s, k5box, CU_TENSOR_MAP_SWIZZLE_128B);
                if (s.T % 4 != 0) ok4 = ok4 && encode_nd(&mp2.k[1], kp, 4, kd, ks, kbox, CU_TENSOR_MAP_SWIZZLE_128B, 4);
            }
            bool ok1 = encode_4d(&mp.k[fused ? 2 : 0], kp, kd, ks, kbox);
            if (fused) {
                const cuuint64_t rows = (cuuint64_t)1 << s.pm.shift;
                const cuuint64_t pd[5] = {kd[0], rows, (cuuint64_t)s.pm.n_pages, kd[2], kd[3]};
                const cuuint64_t pst[4] = {(cuuint64_t)s.ks_p * 2, (cuuint64_t)s.pm.s_page * 2, (cuuint64_t)s.ks_h * 2,
                                           (cuuint64_t)s.ks_l * 2};
                const cuuint32_t pbox[5] = {64, (cuuint32_t)(rows < kTileRows ? rows : kTileRows), 1, 1, 1};
                ok1 = ok1 && encode_nd(&mp.k[0], s.k, 5, pd, pst, pbox, CU_TENSOR_MAP_SWIZZLE_128B);
            }
            if (!ok1 || !ok4 || !encode_4d(&mp.q, s.q, qd, qs, qbox) || !b.ext ||
                !encode_nd(&mp2.k[2], b.ext + s.ext_off, 3, ed, es, ebox, CU_TENSOR_MAP_SWIZZLE_32B)) {
                return cudaErrorNotSupported;
            }
            mp2.q = mp.q;
            if (s.kself) {
                const cuuint64_t sdm[4] = {kd[0], (cuuint64_t)s.m, kd[2], kd[3]};
                const cuuint64_t ss[3] = {(cuuint64_t)s.kss_t * 2, (cuuint64_t)s.kss_h * 2, (cuuint64_t)s.kss_l * 2};
                if (!encode_4d(&mp.k[1], s.kself, sdm, ss, kbox)) return cudaErrorNotSupported;
            }
        }
        const cuuint64_t od[2] = {(cuuint64_t)kExtCols, 128};
        const cuuint64_t os[1] = {(cuuint64_t)kExtCols * 2};
        const cuuint32_t obox[2] = {(cuuint32_t)kExtCols, 128};
        if (!encode_nd(&tb->omap, b.ones, 2, od, os, obox, CU_TENSOR_MAP_SWIZZLE_32B)) {
            return cudaErrorNotSupported;
        }
        tb->rows1 = rows1;
        tb->stages1 = 4;
        while (tb->stages1 > 2 && smem1_bytes(d_head, rows1, tb->stages1) > kSmemMax) --tb->stages1;
        tb->wait_ns = b.wait_ns;
        tb->stall = batches.size() == 1 ? b.stall : 0;   // the first launch only
    }
    cudaError_t e = cudaSuccess;
    for (size_t k = 0; k < batches.size() && e == cudaSuccess; ++k) {
        TcBatch* tb = batches[k].get();
        const int b0 = firsts[k];
        // row chunks in step only when all senders have the same number of them
        int rc1 = tb->max_rc1;
        int64_t units1 = 0;
        for (int j = 0; j < tb->n; ++j) {
            const TcSender& d = tb->s[j];
            if (d.n_rc1 != tb->max_rc1) rc1 = 1;
            units1 += (int64_t)nS * (d.n_chunk1 / 4) * d.n_rc1;
            b.s[b0 + j].n_rc = d.n_rc2;   // partials for the finalize kernel
        }
        stage_mark(b.timer, kStageStart, st);
        e = launch_depage(*depages[k], st, num_sms);   // timed with pass 1
        if (e == cudaSuccess) {
            const int g1 = pass_grid(units1, num_sms, rc1);
            e = d_head == 128 ? launch_stats_d<128>(*tb, g1, st) : launch_stats_d<64>(*tb, g1, st);
            stage_mark(b.timer, kStageStats, st);
        }
        if (e == cudaSuccess) {
            // combine reads this batch's partial-slot counts
            for (int j = 0; j < tb->n; ++j) b.s[b0 + j].n_chunk1 = tb->s[j].n_chunk1;
            if (tb->n == b.n) {
                e = combine(b, st);
            } else {
                const std::unique_ptr<ScoreBatch> sub(new ScoreBatch(b));
                sub->n = tb->n;
                for (int j = 0; j < tb->n; ++j) sub->s[j] = b.s[b0 + j];
                e = combine(*sub, st);
            }
            stage_mark(b.timer, kStageCombine, st);
        }
        // pass 2: the senders of blocks of four tiles, then those of one
        const std::vector<TcSender> all(tb->s, tb->s + tb->n);
        for (int narrow = 0; narrow < 2 && e == cudaSuccess; ++narrow) {
            tb->n = tb->few = 0;
            tb->weight2 = 0;
            tb->max_rc2 = 1;
            tb->rows2 = kRowHalf;
            bool same_rc = true;
            int64_t units2 = 0;
            for (size_t j = 0; j < all.size(); ++j) {
                const TcSender& d = all[j];
                if (d.narrow != narrow) continue;
                same_rc = same_rc && (tb->n == 0 || d.n_rc2 == tb->max_rc2);
                tb->max_rc2 = tb->max_rc2 > d.n_rc2 ? tb->max_rc2 : d.n_rc2;
                const int r2 = (d.halves + d.n_rc2 - 1) / d.n_rc2 * kRowHalf;
                tb->rows2 = tb->rows2 > r2 ? tb->rows2 : r2;
                tb->weight2 += (int64_t)nS * d.n_blk2 * d.halves;
                units2 += (int64_t)nS * d.n_blk2 * d.n_rc2;
                tb->few |= d.few;
                tb->maps[tb->n] = maps2[k][j];
                tb->s[tb->n++] = d;
            }
            if (tb->n == 0) continue;
            if (narrow) {
                tb->kbufs = kMaxStages;
                while (smem_narrow_bytes(d_head, tb->rows2, tb->kbufs) > kSmemMax) --tb->kbufs;
            } else {
                tb->kbufs = smem2_bytes(d_head, tb->rows2, 2) <= kSmemMax ? 2 : 1;
            }
            const int g2 = pass_grid(units2, num_sms, same_rc ? tb->max_rc2 : 1);
            if (narrow) e = d_head == 128 ? launch_narrow_d<128>(*tb, g2, st) : launch_narrow_d<64>(*tb, g2, st);
            else e = d_head == 128 ? launch_accum_d<128>(*tb, g2, st) : launch_accum_d<64>(*tb, g2, st);
        }
        if (e == cudaSuccess) stage_mark(b.timer, kStageAccum, st);
    }
    return e;
}

#endif

}  // namespace cbk
