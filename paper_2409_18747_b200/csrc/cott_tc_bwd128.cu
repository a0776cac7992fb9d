// Backward at d = 128 (bf16 I/O, fp32 accumulation and states; head sizes 72 .. 128 zero-filled to it):
// the three gradients and the dm sum in one launch of two kinds of CTAs.
//
// With q^, k^ the normalised rows (Eq. 2/3) and M the causal mask (Eq. 6), per chunk of 128 tokens:
//   Q walk, forward in time:    dQ^ = (dO V^T . M) K^ + dO Sq        Sq = sum over earlier chunks of V^T K^
//   K walk, backward in time:   dK^ = (V dO^T . M^T) Q^ + V Rt       Rt = sum over later chunks of dO^T Q^
//                               dV' = (K^ Q^^T . M^T) dO + K^ Rt^T
// (the formulas printed after Eq. 7).  dK and dV share one running sum -- the paper's reverse-time
// cumulative sum -- and all four input tiles, so one walk gives both; three such states, or all
// products of the three gradients, do not fit one SM's 512 tensor-memory columns and 227 KB next to
// tiles in flight at this head size, so dQ, whose sum runs the other way, has CTAs of its own.  With
// an all-ones mask (BIDIR) both sums are totals and only the products with them remain.
//
// What bounds it: the chain of one chunk (scores, mask, products, epilogue, state copy) on one SM, stretched
// where the other SMs load and store as well.  Stamps of every CTA, mean of a walk's chunks: K 4.3 us and Q 2.75
// with two (b, h) on an idle GPU, K 5.1 and Q 3.7 with 64 (N=2048), K 4.8 and Q 3.3 at B=3, H=16, N=2999, K 5.0 and
// Q 3.4 in 32 packed sequences.  The products alone would keep the tensor core busy for 1.8 and 1.1 us, and shared
// memory (operands of the products, tiles in and out, the workers' passes) for 3.4 and 2.5.
// Around its chunks a CTA spends 2 to 5 us until the first tile has landed and 2 us on dm and the exit, a walk that
// sums four partial states 14 us more in reading them (a row a lane, uncoalesced), and the call 7 us on its launches.
// So B=4, H=16, N=2048, one wave of 16 K chunks: 5 + 16 x 5.1 + 2 = 89 us of the kernel's 91; B=3, H=16, N=2999: 12 us
// until the state pass is over and read, 24 Q chunks of 3.3, 2 = 93 of 97.
// Measured, L2 cold: B=4, H=16, N=2048 99 us; B=3, H=16, N=2999 112 us; 32 packed sequences of 512 to
// 2048 tokens, H=16, 378 us; B=10, H=12, N=5349, d=96 411 us.  With one slot for P in the Q walk and three
// pairs of slots that took turns in the K walk, where every chunk waited for rows on their way out, and
// with eight warps for the masks: 103, 126, 400 and 441 us.
#include "cott_internal.h"
#include "cott_sm100.cuh"
#include "cott_tc_common.cuh"

namespace cott {

using namespace sm100;
using namespace tc;

namespace {

constexpr int kC = 128;
constexpr int kD = 128;
constexpr int kTile = kC * kD * 2;      // one 128 x 128 bf16 tile: two 64-column halves 16 KB apart
constexpr int kHalf = kTile / 2;
constexpr int kWarpsA = 16, kWarpsB = 8, kWorkerWarps = kWarpsA + kWarpsB;
constexpr int kGroupA = kWarpsA * 32, kGroupB = kWarpsB * 32;       // threads of the worker groups
constexpr int kThreads = (kWorkerWarps + 4) * 32;   // + score, product, state-update and copy threads

// Six tile slots, the bf16 copy of the state and the control block are all of the 227 KB.
// A walk has four tiles a chunk: X and A (scores X A^T), Bv (normalised in place) and the raw rows P
// that the projection needs.  Q walk: X = dO, A = V, Bv = K, P = Q.  K walk: X = V, A = dO, Bv = Q, P = K.
// A slot is asked for again when the last product or epilogue that reads it is done, and a slot that the
// chunk needs to its end, or that output rows are staged in, has a second one, so that no chunk waits for
// rows on their way out.  X is done first (scores and X State): one slot.  P is read by the epilogue, which
// stages its rows (dq, dk) over it: two.  Q walk: A is done with the state update, which goes ahead of the
// scores because Bv has two slots: one.  K walk: A is read by the chunk's last product, and dv is staged
// over it: two; Bv by its first: one.  (With an all-ones mask there is no A and no Bv; X has two, dv over X.)
struct L {
    static constexpr int kOffSb = 6 * kTile;
    static constexpr int kOffCtl = kOffSb + kTile;
    static constexpr int kOffDmRed = 640;            // float [8] + a flag
    static constexpr int kOffXch = 1024;             // float2 [2][128]: per-row partial sums of the two column halves
    static constexpr int kCtlBytes = 3072;
    static constexpr int kDynBytes = kOffCtl + kCtlBytes;   // (no slack: the base must be aligned, see the kernel)
};

struct Bwd128Params {
    // partial states of the groups, fp32 [BH, n * parts, 128 * 128]: V^T K^ of the Q walk's groups and
    // dO^T Q^ of the K walk's (or NULL: one group, nothing precedes it), raw (init_sum: summed here over
    // the groups before, after, or all, `parts` entries each) or already scanned
    const float* sq; const float* rt; int init_sum; int parts;
    float* dm_q; float* dm_k;           // [BH, n]: parts of the dm sum of the two walks
    float* dm_out; int* status;
    const float* m; const float* seq_len; float seq_len_scalar;
    int H; int N;
    int group_q, n_q, group_k, n_k;     // tokens per group and groups of the two walks
    int wait_limit_kcycles;
    int head_first_mask;                // bit i: in tensor map i (q, k, v, dO, dq, dk, dv) the head index comes before the token index
    const int* cu_seqlens;              // packed batch (VARLEN instances)
    void* out_rows[3]; long long out_sn[3], out_sh[3]; int out_w[3];
};

#ifdef COTT_TIMING
// Debug build only.  SM-clock stamps of the first K walk (0) and the first Q walk (1) of (b, h) 0, found by what they do
// and not by their place in the grid: up to 64 chunks, eight slots for each of six roles (0, 1: first thread of worker
// groups A, B; 2-5: score, product, state, copy threads).  Nanosecond stamps of every CTA: start, wait for the kernel before
// it over, first state written, first tile landed, last chunk done, exit.
__device__ long long g_b128_stamps[2 * 6 * 64 * 8];
__device__ long long g_b128_cta[8192 * 6];
__device__ __forceinline__ long long global_ns() { long long t; asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t)); return t; }
#define STAMP(role, c, slot)                                                                                 \
    do {                                                                                                     \
        if (bh == 0 && g == 0 && (c) < 64 && ((role) > 1 || threadIdx.x == ((role) ? kGroupA : 0)))          \
            g_b128_stamps[(((kw ? 0 : 1) * 6 + (role)) * 64 + (c)) * 8 + (slot)] = clock64();                \
    } while (0)
#define CTA_STAMP(thread, slot)                                                                              \
    do { if (threadIdx.x == (thread) && blockIdx.x < 8192) g_b128_cta[blockIdx.x * 6 + (slot)] = global_ns(); } while (0)
#else
#define STAMP(role, c, slot) do { } while (0)
#define CTA_STAMP(thread, slot) do { } while (0)
#endif

// tcgen05.mma chains (one thread).  K step kk of a K-major operand of 128 columns; of an MN-major
// operand: 16 rows = 2048 bytes.
__device__ __forceinline__ uint32_t kstep(int kk) { return ((kk >> 2) * (uint32_t)kHalf + (kk & 3) * 32u) >> 4; }

// P = X A^T, both K-major.
__device__ __forceinline__ void issue_scores(uint32_t tP, uint32_t x, uint32_t a) {
    constexpr uint32_t idesc = instr_desc_bf16(128, 128, false, false);
    const uint32_t xl = smem_desc_lo(x, 16), al = smem_desc_lo(a, 16);
#pragma unroll 2
    for (int kk = 0; kk < 8; ++kk) mma_ss_w(tP, xl + kstep(kk), kDescHi, al + kstep(kk), kDescHi, idesc, kk > 0);
}
// Out = X St, St MN-major (its rows are the contraction index).
__device__ __forceinline__ void issue_x_state(uint32_t tO, uint32_t x, uint32_t st) {
    constexpr uint32_t idesc = instr_desc_bf16(128, 128, false, true);
    const uint32_t xl = smem_desc_lo(x, 16), sl = smem_desc_lo(st, kHalf);
#pragma unroll 2
    for (int kk = 0; kk < 8; ++kk) mma_ss_w(tO, xl + kstep(kk), kDescHi, sl + kk * 128u, kDescHi, idesc, kk > 0);
}
// Out (+)= P~ B: P~ (bf16, two per column) in tensor memory, B MN-major.
__device__ __forceinline__ void issue_pt_b(uint32_t tO, uint32_t tPt, uint32_t bt, bool acc_first) {
    constexpr uint32_t idesc = instr_desc_bf16(128, 128, false, true);
    const uint32_t bl = smem_desc_lo(bt, kHalf);
#pragma unroll 2
    for (int kk = 0; kk < 8; ++kk) mma_ts_w(tO, tPt + kk * 8u, bl + kk * 128u, kDescHi, idesc, (acc_first || kk > 0) ? 1u : 0u);
}
// State (+)= A^T B, both MN-major.
__device__ __forceinline__ void issue_update(uint32_t tS, uint32_t a, uint32_t bt, bool acc_first) {
    constexpr uint32_t idesc = instr_desc_bf16(128, 128, true, true);
    const uint32_t al = smem_desc_lo(a, kHalf), bl = smem_desc_lo(bt, kHalf);
#pragma unroll 2
    for (int kk = 0; kk < 8; ++kk) mma_ss_w(tS, al + kk * 128u, kDescHi, bl + kk * 128u, kDescHi, idesc, (acc_first || kk > 0) ? 1u : 0u);
}

// Thread roles.  Warps 0-23 are row workers (warp w owns tensor-memory lanes / tile rows
// 32 (w % 4) .. + 31 and a part of the columns):
//   group A (16 warps, a quarter of the columns each): masks of the scores, row norms of Bv, bf16 copy
//           of the state -- one after the other the longest chain of a chunk, hence the larger group;
//   group B (8 warps, half of the columns each): epilogues.
// Lane 0 of warp 24 issues the scores, of warp 25 the output products, of warp 26 the state update,
// of warp 27 every TMA load and store.  The roles meet only through mbarriers, every wait bounded.
// Every barrier is a pair indexed by chunk parity; no role can be two chunks behind another: each
// chunk's tiles are requested only after the products (and, where a tile is staged over, the stores)
// of the chunk that held the slot before.
// Loops are kept rolled: five roles run different code on one SM, and with everything unrolled they
// ran out of the instruction caches (ncu: 8.7 warps per issue stalled on "no instruction" against
// 2.7 with the 16-column loops of the epilogues rolled: 141 us against 120 for B=4, H=16, N=2048;
// rolling the product chains, the row norms and the two masks took the same case from 113 to 93; figures of
// those steps, measured another way than the ones above).
// Which walk a CTA runs is a compile-time property of its code (KW).
template <bool KW, bool BIDIR, bool VARLEN>
__device__ __forceinline__ void walk(const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV,
                                     const CUtensorMap& tmDO, const CUtensorMap& tmDQ, const CUtensorMap& tmDK,
                                     const CUtensorMap& tmDV, const Bwd128Params& p) {
    // Tensor-memory columns: State 128 | SC1 128 | SC2 128 | O1 128.  The scores X A^T are in SC1,
    // packed in place to bf16 (columns 0-63).  K walk: K Q^^T in SC2, packed into columns 64-127 of
    // SC1, so that SC2 becomes the dV' accumulator; O1 holds dK^.  Q walk: dQ^ alternates between O1
    // and SC2 (chunk parity).
    constexpr uint32_t colS = 0, colSC1 = 128, colSC2 = 256, colO1 = 384;
    constexpr bool kw = KW;
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    const uint32_t base = smem_u32(smem_raw);
    uint8_t* gbase = smem_raw;
    const uint32_t bars = base + L::kOffCtl;
    enum { B_FX = 0, B_FA = 16, B_FB = 32, B_FP = 48 /* tiles landed */, B_NB = 64 /* Bv normalised */,
           B_S1 = 80, B_S2 = 112 /* scores done */, B_M1 = 96, B_M2 = 128 /* masked scores in tensor memory */,
           B_U = 144 /* state updated */, B_CP = 160 /* bf16 state copy written */, B_O1 = 176, B_O2 = 192 /* accumulators complete */,
           B_D1 = 208, B_D2 = 224 /* accumulators drained */, B_E1 = 240, B_E2 = 256 /* output rows staged */,
           B_XCH = 272, B_RD = 288 /* [4 quadrants][2] first scores read */, B_XF = 352 /* X State done */ };
    auto bar = [&](int which, int c) { return bars + which + 8 * (c & 1); };
    auto par = [&](int c) { return (uint32_t)((c >> 1) & 1); };
    const uint32_t tmem_slot = bars + kCtlTmemSlot;
    volatile uint32_t* tmem_slot_g = reinterpret_cast<volatile uint32_t*>(gbase + L::kOffCtl + kCtlTmemSlot);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + L::kOffCtl + kCtlAbort);
    float* dm_red = reinterpret_cast<float*>(gbase + L::kOffCtl + L::kOffDmRed);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    CTA_STAMP(0, 0);
    if (base & 1023u) {
        if (tid == 0 && atomicCAS(p.status, 0, 1) == 0) {
            p.status[1] = (int)0x80007FF0u;
            p.status[2] = (int)blockIdx.x | (8 << 24);
        }
        return;
    }
    const int n_groups = kw ? p.n_k : p.n_q, group = kw ? p.group_k : p.group_q;
    const int bh = blockIdx.x / (p.n_q + p.n_k), g = blockIdx.x % (p.n_q + p.n_k) - (kw ? 0 : p.n_k);
    const int bseq = bh / p.H, h = bh % p.H;
    const int b = VARLEN ? 0 : bseq;                   // batch coordinate of the tensor maps
    const int seq0 = VARLEN ? p.cu_seqlens[bseq] : 0, seq1 = VARLEN ? p.cu_seqlens[bseq + 1] : p.N;
    const int tok0 = seq0 + g * group;
    const int tok1 = min(seq1, tok0 + group);
    const int n_chunks = tok1 > tok0 ? (tok1 - tok0 + kC - 1) / kC : 0;
    // (a packed batch: the last chunk of a sequence may hold rows of the next one; they are normalised
    // to zero in Bv, which silences them in every product, and that chunk's rows are stored one by one)
    const bool ragged_last = VARLEN && ((tok1 - tok0) % kC) != 0;
    auto chunk_row = [&](int c) { return tok0 + (kw ? n_chunks - 1 - c : c) * kC; };
    auto is_ragged = [&](int c) { return ragged_last && c == (kw ? 0 : n_chunks - 1); };
    const bool is_score = warp == kWorkerWarps, is_out = warp == kWorkerWarps + 1;
    const bool is_upd = warp == kWorkerWarps + 2, is_copy = warp == kWorkerWarps + 3;

    if (is_score) {
        tmem_alloc(tmem_slot, 512);
        tmem_relinquish();
    }
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            const int o = 8 * i;
            for (int w : {(int)B_FX, (int)B_FA, (int)B_FB, (int)B_FP, (int)B_S1, (int)B_S2, (int)B_U, (int)B_O1, (int)B_O2, (int)B_XF}) mbar_init(bars + w + o, 1);
            for (int w : {(int)B_NB, (int)B_M1, (int)B_M2, (int)B_CP}) mbar_init(bars + w + o, kGroupA);
            for (int w : {(int)B_D1, (int)B_D2, (int)B_E1, (int)B_E2, (int)B_XCH}) mbar_init(bars + w + o, kGroupB);
            for (int qq = 0; qq < 4; ++qq) mbar_init(bars + B_RD + 16 * qq + o, kGroupA / 4);
        }
        *abort_flag = 0;
        abort_flag[3] = p.wait_limit_kcycles;
        mbar_fence_init();
        fence_proxy_async();
    }
    if (tid < 16) dm_red[tid] = 0.f;
    if (is_copy && lane == 0) {
        tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmDO);
        tma_prefetch_desc(kw ? &tmDK : &tmDQ);
        if (kw) tma_prefetch_desc(&tmDV);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_g;

    // Slots of the four tiles of chunk c (see L).
    auto off_x = [&](int c) { return BIDIR ? (c & 1) * kTile : 0; };
    auto off_a = [&](int c) { return kw ? (1 + (c & 1)) * kTile : kTile; };
    auto off_b = [&](int c) { return kw ? 3 * kTile : (2 + (c & 1)) * kTile; };
    auto off_p = [&](int c) { return (4 + (c & 1)) * kTile; };
    auto off_dv = [&](int c) { return BIDIR ? off_x(c) : off_a(c); };
    auto load = [&](int off, const CUtensorMap* tm, int which, uint32_t fb, int row) {
        const bool hf = (p.head_first_mask >> which) & 1;
        mbar_expect_tx(fb, kTile);
#pragma unroll 1
        for (int hh = 0; hh < 2; ++hh) tma_load_4d(base + off + hh * kHalf, tm, fb, hh * 64, hf ? h : row, hf ? row : h, b);
    };
    auto load_x = [&](int c) { load(off_x(c), kw ? &tmV : &tmDO, kw ? 2 : 3, bar(B_FX, c), chunk_row(c)); };
    auto load_a = [&](int c) { load(off_a(c), kw ? &tmDO : &tmV, kw ? 3 : 2, bar(B_FA, c), chunk_row(c)); };
    auto load_b = [&](int c) { load(off_b(c), kw ? &tmQ : &tmK, kw ? 0 : 1, bar(B_FB, c), chunk_row(c)); };
    auto load_p = [&](int c) { load(off_p(c), kw ? &tmK : &tmQ, kw ? 1 : 0, bar(B_FP, c), chunk_row(c)); };
    // A kernel of the same call, which writes none of the tensors loaded here, comes before this one: the
    // first tiles are requested before the wait for it.
    if (is_copy && lane == 0 && n_chunks > 0) {
        if (!BIDIR) { load_b(0); load_a(0); }
        load_x(0);
        load_p(0);
        if (n_chunks > 1) {
            if (BIDIR) load_x(1); else if (kw) load_a(1); else load_b(1);
            load_p(1);
        }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    CTA_STAMP(0, 1);

    const float s_b = p.seq_len ? p.seq_len[bseq]
                                : (p.seq_len_scalar > 0.f ? p.seq_len_scalar : (float)(VARLEN ? max(seq1 - seq0, 1) : p.N));
    const float cfac = stab_factor(p.m[h], s_b);

    const int q4 = warp & 3, hw = (warp >> 2) & 1, w8 = warp & 7;
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    const int row = q4 * 32 + lane;               // tile row / tensor-memory lane of a worker thread

    const float* part = kw ? p.rt : p.sq;
    const bool init_state = part != nullptr;
    // 32 columns of this thread's state row as bf16 into the copy (rows of 128 bytes, two column halves).
    auto write_sb = [&](const uint32_t (&r)[32], int c0) {
#pragma unroll
        for (int i = 0; i < 32; i += 8) {
            const int col = c0 + i;
            *reinterpret_cast<uint4*>(gbase + L::kOffSb + (col >> 6) * kHalf + swz(row, (col & 63) >> 3)) = pack8(&r[i]);
        }
    };
    if (init_state && warp < kWarpsA) {
        // The state before the group's first chunk: row `row`, columns 32 (warp / 4) .. + 31.
        const int cq = warp >> 2;
        const int entries = n_groups * p.parts;
        const float* src = part + (size_t)bh * entries * kD * kD + (size_t)row * kD + cq * 32;
        float acc[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) acc[i] = 0.f;
        const int g_lo = !p.init_sum ? g : (BIDIR ? 0 : (kw ? (g + 1) * p.parts : 0));
        const int g_hi = !p.init_sum ? g + 1 : (BIDIR ? entries : (kw ? entries : g * p.parts));
        for (int gg = g_lo; gg < g_hi; ++gg) {
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
                const float4 v = *reinterpret_cast<const float4*>(src + (size_t)gg * kD * kD + i);
                acc[i] += v.x; acc[i + 1] += v.y; acc[i + 2] += v.z; acc[i + 3] += v.w;
            }
        }
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) r[i] = __float_as_uint(acc[i]);
        if (!BIDIR) { tmem_st32(tmem + lane_base + colS + cq * 32, r); tmem_wait_st(); }
        write_sb(r, cq * 32);
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    CTA_STAMP(0, 2);
    float dm_acc = 0.f;
    if (is_copy) {
        // ------------------------------------------------------------------ copy thread
        if (lane == 0 && n_chunks > 0) {
            auto store = [&](const CUtensorMap* tm, int which, int off, int r0) {
                const bool hf = (p.head_first_mask >> which) & 1;
#pragma unroll 1
                for (int hh = 0; hh < 2; ++hh)
                    if (hh * 64 < p.out_w[which - 4]) tma_store_4d(tm, base + off + hh * kHalf, hh * 64, hf ? h : r0, hf ? r0 : h, b);
            };
            auto done = [&](int which, int c) { return wait_or_abort(bar(which, c), par(c), abort_flag); };
            for (int c = 0; c < n_chunks; ++c) {
                const bool by_rows = is_ragged(c);      // the workers stored this chunk's rows themselves
                // What chunk c + 1 lacks, in the order in which the slots come free.
                if (!BIDIR && c + 1 < n_chunks) {
                    if (!done(B_S1, c) || !done(B_XF, c)) break;
                    STAMP(5, c, 0);
                    load_x(c + 1);
                    if (!kw) {
                        if (!done(B_U, c)) break;
                        load_a(c + 1);
                    }
                    STAMP(5, c, 1);
                }
                // The rows staged a chunk ago have left their slots.
                if (c >= 1 && c + 1 < n_chunks) {
                    if (kw) {
                        tma_store_wait_read1();
                        if (BIDIR) load_x(c + 1); else load_a(c + 1);
                    }
                    tma_store_wait_read0();
                    load_p(c + 1);
                }
                STAMP(5, c, 2);
                if (!BIDIR && c + 1 < n_chunks) {
                    if (kw && (!done(B_U, c) || !done(B_S2, c))) break;
                    if (!done(B_O1, c)) break;
                    if (kw) load_b(c + 1); else if (c + 2 < n_chunks) load_b(c + 2);
                } else if (BIDIR && !kw && c + 2 < n_chunks) {
                    if (!done(B_O1, c)) break;
                    load_x(c + 2);
                }
                STAMP(5, c, 3);
                if (kw) {
                    if (!done(B_E2, c)) break;
                    if (!by_rows) store(&tmDV, 6, off_dv(c), chunk_row(c));
                    tma_store_commit();
                }
                if (!done(B_E1, c)) break;
                STAMP(5, c, 4);
                if (!by_rows) store(kw ? &tmDK : &tmDQ, kw ? 5 : 4, off_p(c), chunk_row(c));
                tma_store_commit();
            }
            tma_store_wait_all0();
        }
    } else if (is_score) {
        // ------------------------------------------------------------------ score thread
        if (lane == 0 && !BIDIR) {
            for (int c = 0; c < n_chunks; ++c) {
                if (!wait_or_abort(bar(B_FX, c), par(c), abort_flag)) break;
                if (!wait_or_abort(bar(B_FA, c), par(c), abort_flag)) break;
                STAMP(2, c, 0);
                // the products that read the packed scores in these columns have completed
                if (c >= 1 && !wait_or_abort(bar(B_O1, c - 1), par(c - 1), abort_flag)) break;
                if (kw && c >= 1 && !wait_or_abort(bar(B_O2, c - 1), par(c - 1), abort_flag)) break;
                STAMP(2, c, 1);
                tc_fence_after();
                issue_scores(tmem + colSC1, base + off_x(c), base + off_a(c));
                tc_commit(bar(B_S1, c));
                if (!kw) continue;
                if (!wait_or_abort(bar(B_FP, c), par(c), abort_flag)) break;
                if (!wait_or_abort(bar(B_NB, c), par(c), abort_flag)) break;
                STAMP(2, c, 2);
                if (c >= 1 && !wait_or_abort(bar(B_D2, c - 1), par(c - 1), abort_flag)) break;   // dV' drained
                STAMP(2, c, 3);
                tc_fence_after();
                issue_scores(tmem + colSC2, base + off_p(c), base + off_b(c));
                tc_commit(bar(B_S2, c));
            }
        }
    } else if (is_upd) {
        // ------------------------------------------------------------------ state-update thread
        // (the state after the last chunk is read by nobody)
        if (lane == 0 && !BIDIR) {
            for (int c = 0; c + 1 < n_chunks; ++c) {
                if (!wait_or_abort(bar(B_FA, c), par(c), abort_flag)) break;
                if (!wait_or_abort(bar(B_NB, c), par(c), abort_flag)) break;
                if (c >= 1 && !wait_or_abort(bar(B_CP, c - 1), par(c - 1), abort_flag)) break;
                STAMP(4, c, 0);
                tc_fence_after();
                issue_update(tmem + colS, base + off_a(c), base + off_b(c), init_state || c > 0);
                tc_commit(bar(B_U, c));
            }
        }
    } else if (is_out) {
        // ------------------------------------------------------------------ output-product thread
        if (lane == 0) {
            const uint32_t sb = base + L::kOffSb;
            for (int c = 0; c < n_chunks; ++c) {
                const bool acc = BIDIR || init_state || c > 0;
                const uint32_t tO = tmem + (!kw && (c & 1) ? colSC2 : colO1);
                if (!wait_or_abort(bar(B_FX, c), par(c), abort_flag)) break;
                if (c == 0) CTA_STAMP((kWorkerWarps + 1) * 32, 3);
                if (c >= 1 && !BIDIR && !wait_or_abort(bar(B_CP, c - 1), par(c - 1), abort_flag)) break;
                STAMP(3, c, 0);
                // the accumulator has been drained: one in the K walk, two in turn in the Q walk
                if (kw && c >= 1 && !wait_or_abort(bar(B_D1, c - 1), par(c - 1), abort_flag)) break;
                if (!kw && c >= 2 && !wait_or_abort(bar(B_D1, c - 2), par(c - 2), abort_flag)) break;
                STAMP(3, c, 1);
                tc_fence_after();
                if (acc) issue_x_state(tO, base + off_x(c), sb);
                if (!BIDIR) {
                    tc_commit(bar(B_XF, c));
                    if (!wait_or_abort(bar(B_M1, c), par(c), abort_flag)) break;
                    STAMP(3, c, 2);
                    if (!wait_or_abort(bar(B_NB, c), par(c), abort_flag)) break;
                    STAMP(3, c, 3);
                    tc_fence_after();
                    issue_pt_b(tO, tmem + colSC1, base + off_b(c), acc);
                }
                tc_commit(bar(B_O1, c));
                if (!kw) continue;
                if (BIDIR) {
                    if (!wait_or_abort(bar(B_FP, c), par(c), abort_flag)) break;
                    if (c >= 1 && !wait_or_abort(bar(B_D2, c - 1), par(c - 1), abort_flag)) break;
                } else if (!wait_or_abort(bar(B_M2, c), par(c), abort_flag)) break;
                STAMP(3, c, 4);
                tc_fence_after();
                // K Rt^T: the state copy read K-major (its columns are the contraction index)
                if (acc) issue_scores(tmem + colSC2, base + off_p(c), sb);
                if (!BIDIR) issue_pt_b(tmem + colSC2, tmem + colSC1 + 64, base + off_a(c), acc);
                tc_commit(bar(B_O2, c));
            }
        }
    } else {
        // ------------------------------------------------------------------ row workers
        bool alive = n_chunks > 0;
        auto wait = [&](uint32_t bar_, uint32_t parity) {
            if (alive && !wait_or_abort(bar_, parity, abort_flag)) alive = false;
            return alive;
        };
        if (warp < kWarpsA) {
            // -------------------------------------------------------------- group A
            const int cb = warp >> 2;                  // this warp's 32 columns
            // One 32 x 32 score block a warp (row block q4, column block cb), masked (Q walk: columns up
            // to the row, K walk: from the row on; diagonal kept, Eq. 6) and packed to bf16, two per
            // column, to the columns from tdst on.  The mask of a block is all-keep, all-zero or a
            // triangle; the first two are warp-uniform.  The packed scores go over the start of the
            // first fp32 ones: `rd` is the barrier on which the four warps of a row block meet when they
            // have read theirs (0: no need, they have).
            auto mask = [&](uint32_t tsc, uint32_t tdst, uint32_t rd, uint32_t rpar) {
                uint32_t r[32];
                if (kw ? cb >= q4 : cb <= q4) {
                    tmem_ld32(tsc + lane_base + cb * 32, r);
                    tmem_wait_ld();
                    if (cb == q4) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) r[j] = (kw ? j >= lane : j <= lane) ? r[j] : 0u;
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) r[j] = 0u;
                }
                if (rd) { tc_fence_before(); mbar_arrive(rd); }
#pragma unroll
                for (int j = 0; j < 16; ++j) r[j] = pack_bf16(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
                if (rd) {
                    if (!wait(rd, rpar)) return;
                    tc_fence_after();
                }
                tmem_st16(tdst + lane_base + cb * 16, r);
                tmem_wait_st();
                tc_fence_before();
            };
            // x^ = x / max(||x||, eps) on a quarter of a row of Bv, in place (lanes l, l ^ 8, l ^ 16, l ^ 24
            // share a row).
            auto normalise = [&](int c) {
                if (!wait(bar(B_FB, c), par(c))) return;
                const int nrow = warp * 8 + (lane & 7), part = lane >> 3;
                uint8_t* tile = gbase + off_b(c) + (part >> 1) * kHalf;
                uint4 w[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) w[j] = *reinterpret_cast<const uint4*>(tile + swz(nrow, (part & 1) * 4 + j));
                float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
                for (int i = 0; i < 16; i += 2) {
                    const float2 f0 = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[i]);
                    const float2 f1 = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[i + 1]);
                    s0 = __ffma2_rn(f0, f0, s0); s1 = __ffma2_rn(f1, f1, s1);
                }
                float ss = (s0.x + s0.y) + (s1.x + s1.y);
                ss += __shfl_xor_sync(0xffffffffu, ss, 8);
                ss += __shfl_xor_sync(0xffffffffu, ss, 16);
                float rn = 1.0f / fmaxf(sqrtf(ss), kEps);
                if (VARLEN && chunk_row(c) + nrow >= tok1) rn = 0.f;      // a row of the next sequence
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    __nv_bfloat162* e = reinterpret_cast<__nv_bfloat162*>(&w[j]);
#pragma unroll
                    for (int i = 0; i < 4; ++i) e[i] = scale_round(e[i], rn);
                    *reinterpret_cast<uint4*>(tile + swz(nrow, (part & 1) * 4 + j)) = w[j];
                }
                fence_proxy_async();
                mbar_arrive(bar(B_NB, c));
            };
            if (!BIDIR && !kw) normalise(0);
            for (int c = 0; !BIDIR && c < n_chunks && alive; ++c) {
                // K walk: Bv of this chunk was asked for during the chunk before.  Q walk: Bv of the next
                // chunk has been there for a while; its norms fill the wait for this chunk's products.
                STAMP(0, c, 0);
                if (kw) { normalise(c); if (!alive) break; }
                STAMP(0, c, 1);
                // (the second scores of the K walk are packed into columns 64-127 of SC1)
#pragma unroll 1
                for (int it = 0; it < (kw ? 2 : 1) && alive; ++it) {
                    if (!wait(bar(it ? B_S2 : B_S1, c), par(c))) break;
                    STAMP(0, c, 2 + 2 * it);
                    tc_fence_after();
                    mask(tmem + (it ? colSC2 : colSC1), tmem + colSC1 + it * 64, it ? 0u : bars + B_RD + 16 * q4 + 8 * (c & 1), par(c));
                    if (!alive) break;
                    mbar_arrive(bar(it ? B_M2 : B_M1, c));
                    STAMP(0, c, 3 + 2 * it);
                }
                if (!kw && alive && c + 1 < n_chunks) normalise(c + 1);
                if (!alive) break;
                // bf16 copy of the updated state for the next chunk, once this chunk's products
                // have read the previous copy.
                if (c + 1 < n_chunks) {
                    if (!wait(bar(B_U, c), par(c))) break;
                    if (!wait(bar(B_O1, c), par(c))) break;
                    if (kw && !wait(bar(B_O2, c), par(c))) break;
                    STAMP(0, c, 6);
                    tc_fence_after();
                    {
                        uint32_t r[32];
                        tmem_ld32(tmem + lane_base + colS + cb * 32, r);
                        tmem_wait_ld();
                        write_sb(r, cb * 32);
                    }
                    fence_proxy_async();
                    tc_fence_before();
                    mbar_arrive(bar(B_CP, c));
                    STAMP(0, c, 7);
                }
            }
        } else {
            // -------------------------------------------------------------- group B
            // (rows of a ragged last chunk of a packed batch leave one by one)
            auto put = [&](uint8_t* tile, int which, bool by_rows, int c, int i, uint4 o) {
                if (VARLEN && by_rows) {
                    const long long grow = (long long)chunk_row(c) + row;
                    const int col = hw * 64 + i;
                    if (grow < tok1 && col < p.out_w[which])
                        *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(p.out_rows[which]) + grow * p.out_sn[which] +
                                                  (long long)h * p.out_sh[which] + col) = o;
                } else {
                    *reinterpret_cast<uint4*>(tile + swz(row, i >> 3)) = o;
                }
            };
            float2* xch = reinterpret_cast<float2*>(gbase + L::kOffCtl + L::kOffXch);
            for (int c = 0; c < n_chunks && alive; ++c) {
                // ---- projection epilogue (chain rule through x^ = x / max(||x||, eps)), this thread's 64 columns
                STAMP(1, c, 0);
                if (!wait(bar(B_FP, c), par(c))) break;
                uint8_t* tile = gbase + off_p(c) + hw * kHalf;
                const uint32_t tacc = tmem + lane_base + (!kw && (c & 1) ? colSC2 : colO1) + hw * 64;
                if (!wait(bar(B_O1, c), par(c))) break;
                STAMP(1, c, 1);
                tc_fence_after();
                float2 s2 = make_float2(0.f, 0.f), d2 = s2;
#pragma unroll 1
                for (int pc = 0; pc < 4; ++pc) {
                    float2 r[8];
                    tmem_ld16(tacc + pc * 16, reinterpret_cast<uint32_t*>(r));
                    uint4 w[2];
#pragma unroll
                    for (int i = 0; i < 2; ++i) w[i] = *reinterpret_cast<const uint4*>(tile + swz(row, pc * 2 + i));
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const float2 f = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[i]);
                        s2 = __ffma2_rn(f, f, s2);
                        d2 = __ffma2_rn(f, r[i], d2);
                    }
                }
                // (every thread of the group has read the exchange area of the chunk before)
                if (c >= 1 && !wait(bar(B_D1, c - 1), par(c - 1))) break;
                xch[hw * 128 + row] = make_float2(s2.x + s2.y, d2.x + d2.y);
                mbar_arrive(bar(B_XCH, c));
                STAMP(1, c, 2);
                if (!wait(bar(B_XCH, c), par(c))) break;
                const float2 e0 = xch[row], e1 = xch[128 + row];
                const float dp = e0.y + e1.y, nrm = sqrtf(e0.x + e1.x);
                const float rp = 1.0f / fmaxf(nrm, kEps);
                const bool valid = !VARLEN || chunk_row(c) + row < tok1;
                // dm: the Q walk sums <q^_i, dQ^_i> of the unscaled accumulator.  That sum uses k^ rounded
                // to bf16; to first order the sum with the exact k^ is larger by
                // sum_j <k^_j - bf16(k^_j), dK^_j>, and the K walk has both factors.
                const bool use = valid && (!kw || nrm > kEps);
                if (use && hw == 0) dm_acc += dp * rp;
                const bool by_rows = is_ragged(c);
                const float sc = cfac * rp, mc = nrm > kEps ? -dp * cfac * rp * rp * rp : 0.f;
                const float2 sc2 = make_float2(sc, sc), mc2 = make_float2(mc, mc);
                if (kw) {
                    // ---- dV = (c / max(||k||, eps)) dV', ahead of the rows of dk: the next chunk's second
                    // scores wait for this accumulator.  (Its products and the state update are the last to read A.)
                    if (!wait(bar(B_O2, c), par(c))) break;
                    if (!BIDIR && c + 1 < n_chunks && !wait(bar(B_U, c), par(c))) break;
                    tc_fence_after();
                    STAMP(1, c, 3);
                    uint8_t* vt = gbase + off_dv(c) + hw * kHalf;
#pragma unroll 1
                    for (int pc = 0; pc < 4; ++pc) {
                        float2 r[8];
                        tmem_ld16(tmem + lane_base + colSC2 + hw * 64 + pc * 16, reinterpret_cast<uint32_t*>(r));
                        tmem_wait_ld();
                        uint4 o[2];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float2 v = __fmul2_rn(r[i], sc2);
                            reinterpret_cast<uint32_t*>(o)[i] = pack_bf16(v.x, v.y);
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) put(vt, 2, by_rows, c, (pc * 2 + i) * 8, o[i]);
                    }
                    tc_fence_before();
                    mbar_arrive(bar(B_D2, c));
                    fence_proxy_async();
                    mbar_arrive(bar(B_E2, c));
                }
                STAMP(1, c, 4);
                // ---- out = (c acc - x coef) / max(||x||, eps) over the raw rows
                const float ks = use ? rp : 0.f;
                float2 k2 = make_float2(0.f, 0.f);
#pragma unroll 1
                for (int pc = 0; pc < 4; ++pc) {
                    float2 r[8];
                    tmem_ld16(tacc + pc * 16, reinterpret_cast<uint32_t*>(r));
                    uint4 w[2];
#pragma unroll
                    for (int i = 0; i < 2; ++i) w[i] = *reinterpret_cast<const uint4*>(tile + swz(row, pc * 2 + i));
                    tmem_wait_ld();
                    uint4 o[2];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const __nv_bfloat162 e = reinterpret_cast<const __nv_bfloat162*>(w)[i];
                        if (kw) k2 = __ffma2_rn(__bfloat1622float2(scale_round(e, ks)), r[i], k2);
                        const float2 v = __ffma2_rn(__bfloat1622float2(e), mc2, __fmul2_rn(r[i], sc2));
                        reinterpret_cast<uint32_t*>(o)[i] = pack_bf16(v.x, v.y);
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i) put(tile, kw ? 1 : 0, by_rows, c, (pc * 2 + i) * 8, o[i]);
                }
                if (kw) dm_acc -= k2.x + k2.y;
                tc_fence_before();
                mbar_arrive(bar(B_D1, c));
                fence_proxy_async();
                mbar_arrive(bar(B_E1, c));
                STAMP(1, c, 5);
            }
            CTA_STAMP(kGroupA, 4);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dm_acc += __shfl_xor_sync(0xffffffffu, dm_acc, o);
            if (lane == 0) dm_red[w8] = dm_acc;
        }
    }

    tc_fence_before();
    __syncthreads();
    {
        int* last_flag = reinterpret_cast<int*>(&dm_red[8]);
        if (tid == 0) {
            if (!*abort_flag)
                (kw ? p.dm_k : p.dm_q)[(size_t)bh * n_groups + g] = ((dm_red[0] + dm_red[1]) + (dm_red[2] + dm_red[3])) +
                                                                   ((dm_red[4] + dm_red[5]) + (dm_red[6] + dm_red[7]));
            __threadfence();
            *last_flag = atomicAdd(&p.status[4], 1) == (int)gridDim.x - 1;
        }
        __syncthreads();
        if (*last_flag) {
            // Every CTA's partial sums are visible: dm_h = sum_b dc/dm(b,h) * sum_g T_{b,h,g}, T the sum
            // over rows of <q^, dQ^> plus the rounding term, dc/dm = -ln(s_b) sigma(m_h) (1 - sigma(m_h))
            // c_{b,h}; fixed order, so deterministic.  One warp per head.
            __threadfence();
            const int per_q = p.n_q + p.n_k, per = (int)gridDim.x / p.H;
            for (int hh = warp; hh < p.H; hh += kThreads / 32) {
                const float sg = 1.0f / (1.0f + expf(-p.m[hh]));
                float sum = 0.f;
                for (int i = lane; i < per; i += 32) {
                    const int bb = i / per_q, gg = i - bb * per_q;
                    const float sb2 = p.seq_len ? p.seq_len[bb]
                                                : (p.seq_len_scalar > 0.f ? p.seq_len_scalar
                                                   : (float)(VARLEN ? max(p.cu_seqlens[bb + 1] - p.cu_seqlens[bb], 1) : p.N));
                    const float ls = logf(sb2);
                    const size_t bh2 = (size_t)bb * p.H + hh;
                    const float part_sum = gg < p.n_q ? __ldcg(&p.dm_q[bh2 * p.n_q + gg]) : __ldcg(&p.dm_k[bh2 * p.n_k + gg - p.n_q]);
                    sum += part_sum * (-ls * sg * (1.0f - sg) * expf(-sg * ls));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (lane == 0) p.dm_out[hh] = sum;
            }
            if (tid == 0) p.status[4] = 0;
        }
    }
    if (*abort_flag) {
        // A wait gave up: let the copies and products still in flight land (microseconds), then report.
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
        __syncthreads();
        if (tid == 0 && atomicCAS(p.status, 0, 1) == 0) {
            p.status[1] = *abort_flag;
            p.status[2] = (int)blockIdx.x | (8 << 24);
        }
    }
    if (is_score) tmem_dealloc(tmem, 512);
    CTA_STAMP(0, 5);
}

template <bool BIDIR, bool VARLEN>
__global__ void __launch_bounds__(kThreads, 1)
tc_bwd128_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmDO,
                 const __grid_constant__ CUtensorMap tmDQ, const __grid_constant__ CUtensorMap tmDK,
                 const __grid_constant__ CUtensorMap tmDV, const __grid_constant__ Bwd128Params p) {
    // The walks of a (b, h) are neighbours in the grid; the longer ones, K, first.
    if ((int)(blockIdx.x % (p.n_q + p.n_k)) < p.n_k) walk<true, BIDIR, VARLEN>(tmQ, tmK, tmV, tmDO, tmDQ, tmDK, tmDV, p);
    else walk<false, BIDIR, VARLEN>(tmQ, tmK, tmV, tmDO, tmDQ, tmDK, tmDV, p);
}

}  // namespace

cudaError_t launch_tc_bwd128(const TcBwdFusedArgs& a, const Bwd128Groups& g, float* dm_k, int B, int H, int N, cudaStream_t st) {
    const void* ptrs[7] = {a.q, a.k, a.v, a.d_o, a.dq, a.dk, a.dv};
    const RowLayout lays[7] = {a.l_qkv, a.l_qkv, a.l_v, a.l_do, a.l_dqkv, a.l_dqkv, a.l_dv};
    const int wk = a.w_k > 0 ? a.w_k : kD, wv = a.w_v > 0 ? a.w_v : kD;
    const int dims[7] = {wk, wk, wv, wv, wk, wk, wv};
    if (wk > kD || wv > kD) return cudaErrorInvalidValue;
    CUtensorMap tm[7];
    Bwd128Params p;
    p.head_first_mask = 0;
    // A packed batch is one tensor of total_tokens rows per head (batch extent 1).
    const int map_B = a.cu_seqlens ? 1 : B, map_N = a.cu_seqlens ? a.total_tokens : N;
    for (int i = 0; i < 7; ++i) {
        bool hf = false;
        if (!make_tile_map(&tm[i], ptrs[i], map_B, H, map_N, dims[i], lays[i], &hf)) return cudaErrorInvalidValue;
        p.head_first_mask |= (hf ? 1 : 0) << i;
    }
    for (int i = 0; i < 3; ++i) {
        const RowLayout lo = resolve_layout(lays[4 + i], H, map_N, dims[4 + i]);
        p.out_rows[i] = const_cast<void*>(ptrs[4 + i]); p.out_sn[i] = lo.sn; p.out_sh[i] = lo.sh; p.out_w[i] = dims[4 + i];
    }
    p.sq = a.sq_part; p.rt = a.r_part; p.init_sum = g.init_sum; p.parts = g.parts;
    p.dm_q = a.dm_partial; p.dm_k = dm_k; p.dm_out = a.dm_out; p.status = a.status;
    p.m = a.m; p.seq_len = a.seq_len; p.seq_len_scalar = a.seq_len_scalar;
    p.H = H; p.N = N;
    p.group_q = g.group_q; p.n_q = g.n_q; p.group_k = g.group_k; p.n_k = g.n_k;
    p.wait_limit_kcycles = wait_limit_kcycles();
    p.cu_seqlens = a.cu_seqlens;
    if (a.bidir && (!a.sq_part || !a.r_part)) return cudaErrorInvalidValue;
    auto kern = a.cu_seqlens ? (a.bidir ? tc_bwd128_kernel<true, true> : tc_bwd128_kernel<false, true>)
                             : (a.bidir ? tc_bwd128_kernel<true, false> : tc_bwd128_kernel<false, false>);
    if (cudaError_t e = configure_smem_once(reinterpret_cast<const void*>(kern), L::kDynBytes); e != cudaSuccess)
        return e;
    const int prof = profile_begin_launch(3, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(B * H * (g.n_q + g.n_k)));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = L::kDynBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // (a packed batch reads cu_seqlens before anything else)
    cfg.numAttrs = a.cu_seqlens ? 0 : 1;
    cudaError_t le = cudaLaunchKernelEx(&cfg, kern, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], tm[6], p);
    profile_end_launch(prof, st);
    note_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
}

}  // namespace cott

#ifdef COTT_TIMING
extern "C" int cott_debug_b128_stamps(long long* out) {
    return (int)cudaMemcpyFromSymbol(out, cott::g_b128_stamps, sizeof(cott::g_b128_stamps));
}
extern "C" int cott_debug_b128_ctas(long long* out) {
    return (int)cudaMemcpyFromSymbol(out, cott::g_b128_cta, sizeof(cott::g_b128_cta));
}
#endif
