// Backward for sequences of at most 128 tokens (bf16 I/O, fp32 accumulation; causal or bidirectional,
// head sizes up to 128): the quadratic form, as in cott_tc_short.cu, several whole sequences per 128-row
// tile, no running state, no state pass.
//
// With rq, rk = 1 / max(||row||, eps), M the mask (same sequence; causal: j <= i), c the factor of Eq. 4:
//     P_ij = rq_i rk_j q_i . k_j   M_ij          G_ij = rq_i rk_j dO_i . v_j   M_ij
//     dV  = c P^T dO       a = G K,   dq_i = c (a_i - rq_i^2 <q_i, a_i> q_i)
//                          b = G^T Q, dk_j = c (b_j - rk_j^2 <k_j, b_j> k_j)
// (the second terms are absent where the norm is clamped).  Both norms ride on the scores, in fp32, so every
// operand is a tile as it was loaded: nothing is normalised in shared memory, and the rounding of P and G
// to bf16 is the only one before the outputs.  T = sum_ij P_ij dO_i . v_j of a sequence, which dm needs, is
// the element-wise product of the two score matrices, fp32.
//
// One CTA per tile: 16 warps of row workers (a quarter of a row's scores each, half of a row of dq or dk)
// and one warp for copies and products; where the tiles of D = 64 are more than one wave, eight, with 99.5 KB and
// 256 tensor-memory columns, so that two CTAs share an SM.  D = 64 keeps P and G in one buffer in turn, D = 128
// has one for each.  Bound by the chain of one tile (tiles land, norms, scores, masks, products, epilogues,
// rows out), which is most of the 12 to 16 us of a call of one wave.  Against the kernels for longer
// sequences, which take a CTA or two per (b, h): 39 x 12 sequences of 18 tokens, d = 128, bidirectional 119 ->
// 16.5 us, causal 63.7 -> 16.6, d = 64 causal 34.2 -> 13.3; 64 x 16 of 100 tokens, d = 128, 136 -> 103.
#include "cott_internal.h"
#include "cott_sm100.cuh"
#include "cott_tc_common.cuh"

namespace cott {

using namespace sm100;
using namespace tc;

namespace {

constexpr int kRows = 128;                    // rows of a tile

template <int D, int NW>
struct SBL {
    static constexpr int kWorkers = NW * 32, kThreads = kWorkers + 32;
    static constexpr int kParts = NW / 4;             // threads of a row in the scores
    static constexpr int kHalves = NW / 8;            // threads of a row of dq and of dk
    static constexpr int NH = D / 64;                 // 64-column half tiles
    static constexpr int kTile = kRows * D * 2;
    static constexpr int kOffQ = 0, kOffK = kTile, kOffV = 2 * kTile, kOffDO = 3 * kTile;
    static constexpr int kMat = kRows * kRows * 2;    // bf16 score matrix: two half tiles
    static constexpr bool kTwo = D == 128;            // P and G have a buffer each
    static constexpr int kOffP = 4 * kTile, kOffG = kTwo ? kOffP + kMat : kOffP;
    static constexpr int kOffCtl = kOffG + kMat;
    static constexpr int kOffRq = 512, kOffRk = 1024; // float [128], behind the barriers; negative where clamped
    static constexpr int kOffT = 1536;                // float [kParts][128]: <P_i, dO_i V^T> of the parts of a row
    static constexpr int kOffX = kOffT + kParts * 512;   // float [2][2][128]: <q_i, a_i>, <k_j, b_j> of the halves of a row
    static constexpr int kOffLast = 480, kOffBad = 484;
    static constexpr int kDynBytes = kOffCtl + kOffX + (kHalves > 1 ? 2048 : 0) + 1024;
    static constexpr int kTmemCols = D == 64 ? 256 : 512;
    static_assert(NW != 8 || (2 * (kDynBytes + 1024) <= 228 * 1024 && 2 * kTmemCols <= 512), "two CTAs an SM");
    // accumulators: scores P 0-127, G 128-255; D = 64: dV' over P (0-63), a 64-127, b 128-191; D = 128: dV' 256, a 384, b 0
    static constexpr uint32_t colP = 0, colG = 128, colV = D == 64 ? 0 : 256, colA = D == 64 ? 64 : 384, colB = D == 64 ? 128 : 0;
};

struct ShortBwdParams {
    float* dm_partial; float* dm_out; int* status;
    const float* m; const float* seq_len; float seq_len_scalar;
    int H; int N; int BH;
    int slot;                // rows of a sequence's place in a tile: N rounded up to eight (a swizzle atom)
    int seqs;                // sequences per tile
    int causal;
    int wk, wv;              // columns of q, k and of v, dO
    int head_first_mask;     // bit i: in tensor map i (q, k, v, dO, dq, dk, dv) the head index comes before the token index
    int wait_limit_kcycles;
};

template <int D, int NW>
__global__ void __launch_bounds__(SBL<D, NW>::kThreads, D == 64 && NW == 8 ? 2 : 1)
tc_short_bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmDO,
                    const __grid_constant__ CUtensorMap tmDQ, const __grid_constant__ CUtensorMap tmDK,
                    const __grid_constant__ CUtensorMap tmDV, const __grid_constant__ ShortBwdParams p) {
    using L = SBL<D, NW>;
    constexpr int NH = L::NH, kWorkers = L::kWorkers, kThreads = L::kThreads;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + L::kOffCtl;
    // (every barrier completes once a pass)
    enum { B_FULL = 0, B_NR = 8 /* norms known, other rows zeroed */, B_SF = 16 /* scores */, B_R1 = 24, B_R2 = 32 /* masked scores */,
           B_VF = 40 /* dV' done */, B_OF = 48 /* all products done */, B_XR = 56 /* halves of a row met */, B_ED = 64 /* rows staged */ };
    const uint32_t tmem_slot = bars + kCtlTmemSlot;
    volatile uint32_t* tmem_slot_g = reinterpret_cast<volatile uint32_t*>(gbase + L::kOffCtl + kCtlTmemSlot);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + L::kOffCtl + kCtlAbort);
    volatile int* bad_flag = reinterpret_cast<volatile int*>(gbase + L::kOffCtl + L::kOffBad);
    float* rq_buf = reinterpret_cast<float*>(gbase + L::kOffCtl + L::kOffRq);
    float* rk_buf = reinterpret_cast<float*>(gbase + L::kOffCtl + L::kOffRk);
    float* t_buf = reinterpret_cast<float*>(gbase + L::kOffCtl + L::kOffT);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool is_ctrl = warp == kWorkers / 32;
    const int pair0 = (int)blockIdx.x * p.seqs;               // first (b, h) of the tile
    const int n_seq = min(p.seqs, p.BH - pair0);

    if (is_ctrl) {
        tmem_alloc(tmem_slot, L::kTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(bars + B_FULL, 1);
        mbar_init(bars + B_NR, kWorkers);
        mbar_init(bars + B_SF, 1);
        mbar_init(bars + B_R1, kWorkers);
        mbar_init(bars + B_R2, kWorkers);
        mbar_init(bars + B_VF, 1);
        mbar_init(bars + B_OF, 1);
        mbar_init(bars + B_XR, kWorkers);
        mbar_init(bars + B_ED, kWorkers);
        *abort_flag = 0;
        *bad_flag = 0;
        abort_flag[3] = p.wait_limit_kcycles;
        mbar_fence_init();
        fence_proxy_async();
    }
    if (is_ctrl && lane == 0) {
        tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmDO);
        tma_prefetch_desc(&tmDQ); tma_prefetch_desc(&tmDK); tma_prefetch_desc(&tmDV);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_g;
    // Tiles of the sequences s0 .. s1 - 1 (all lanes of the last warp): one copy per sequence, tensor and half
    // tile, over the lanes; rows past N read as zero.
    auto load = [&](int s0, int s1) {
        if (lane == 0) mbar_expect_tx(bars + B_FULL, (uint32_t)((s1 - s0) * p.slot) * 128u * 4u * NH);
        __syncwarp();
        for (int i = lane; i < (s1 - s0) * 4 * NH; i += 32) {
            const int s = s0 + i / (4 * NH), t = i / NH & 3, hh = i % NH, pair = pair0 + s;
            const int b = pair / p.H, h = pair - b * p.H;
            const bool hf = (p.head_first_mask >> t) & 1;
            const CUtensorMap* tm = t == 0 ? &tmQ : t == 1 ? &tmK : t == 2 ? &tmV : &tmDO;
            tma_load_4d(base + t * L::kTile + hh * 16384 + s * p.slot * 128, tm, bars + B_FULL, hh * 64, hf ? h : 0, hf ? 0 : h, b);
        }
    };
    // The kernel before this one is the call's own, writes none of the tensors loaded here and started its
    // dependents behind its own wait: the tiles are requested before the wait for it.
    if (is_ctrl) load(0, n_seq);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // A pass takes the sequences s0 .. s1 - 1 of the tile: all of them, once.  Sequences that share a tile
    // meet in the products as zeros times each other's rows, which is no zero where a row is not finite:
    // then (some score, masked or not, is not finite) the first pass leaves nothing behind and every
    // sequence gets a pass of its own.
    int n_pass = 1;
    bool alive = true;
    auto wait = [&](int which, uint32_t parity) {
        if (alive && !wait_or_abort(bars + which, parity, abort_flag)) alive = false;
        return alive;
    };
    for (int pass = 0; pass < n_pass && alive; ++pass) {
        const uint32_t par = (uint32_t)(pass & 1);
        const int s0 = pass == 0 ? 0 : pass - 1, s1 = pass == 0 ? n_seq : pass;
        if (is_ctrl) {
            // -------------------------------------------------------------- copies and products
            if (pass > 0) load(s0, s1);
            if (lane == 0) {
                const uint32_t q = base + L::kOffQ, k = base + L::kOffK, v = base + L::kOffV, g_o = base + L::kOffDO;
                auto scores = [&](uint32_t t, uint32_t x, uint32_t a) {
                    constexpr uint32_t idesc = instr_desc_bf16(128, 128, false, false);
                    const uint32_t xl = smem_desc_lo(x, 16), al = smem_desc_lo(a, 16);
#pragma unroll 2
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint32_t off = ((kk >> 2) * 16384u + (kk & 3) * 32u) >> 4;
                        mma_ss_w(t, xl + off, kDescHi, al + off, kDescHi, idesc, kk > 0);
                    }
                };
                // rows of a score matrix (K-major), or its columns (MN-major), times a tile
                auto mat_b = [&](uint32_t t, uint32_t mat, uint32_t bt) {
                    constexpr uint32_t idesc = instr_desc_bf16(128, D, false, true);
                    const uint32_t ml = smem_desc_lo(mat, 16), bl = smem_desc_lo(bt, 16384);
#pragma unroll 2
                    for (int kk = 0; kk < kRows / 16; ++kk)
                        mma_ss_w(t, ml + (((kk >> 2) * 16384u + (kk & 3) * 32u) >> 4), kDescHi, bl + kk * 128u, kDescHi, idesc, kk > 0);
                };
                auto mat_t_b = [&](uint32_t t, uint32_t mat, uint32_t bt) {
                    constexpr uint32_t idesc = instr_desc_bf16(128, D, true, true);
                    const uint32_t ml = smem_desc_lo(mat, 16384), bl = smem_desc_lo(bt, 16384);
#pragma unroll 2
                    for (int kk = 0; kk < kRows / 16; ++kk) mma_ss_w(t, ml + kk * 128u, kDescHi, bl + kk * 128u, kDescHi, idesc, kk > 0);
                };
                if (wait(B_FULL, par) && wait(B_NR, par)) {
                    tc_fence_after();
                    scores(tmem + L::colP, q, k);
                    scores(tmem + L::colG, g_o, v);
                    tc_commit(bars + B_SF);
                }
                if (wait(B_R1, par)) {
                    tc_fence_after();
                    const bool skip = pass == 0 && n_seq > 1 && *bad_flag;
                    if (!skip) mat_t_b(tmem + L::colV, base + L::kOffP, g_o);
                    if (!L::kTwo) {
                        tc_commit(bars + B_VF);
                        if (wait(B_R2, par)) tc_fence_after();
                    }
                    if (alive) {
                        if (!skip) {
                            mat_b(tmem + L::colA, base + L::kOffG, k);
                            mat_t_b(tmem + L::colB, base + L::kOffG, q);
                        }
                        tc_commit(bars + B_OF);
                    }
                }
                wait(B_ED, par);
            }
            alive = __shfl_sync(0xffffffffu, alive ? 1 : 0, 0) != 0;
            // (long complete: the staged rows and the flag, which lane 0 alone has waited for, are shown to the lanes that store)
            if (!alive || !wait(B_ED, par)) break;
            const bool skip = pass == 0 && n_seq > 1 && *bad_flag;
            if (skip) {
                n_pass = 1 + n_seq;
            } else {
                for (int i = lane; i < (s1 - s0) * 3 * NH; i += 32) {
                    const int s = s0 + i / (3 * NH), r = i % (3 * NH), t = r / NH, hh = r % NH, pair = pair0 + s;
                    const int b = pair / p.H, h = pair - b * p.H;
                    const bool hf = (p.head_first_mask >> (4 + t)) & 1;
                    if (hh * 64 < (t == 2 ? p.wv : p.wk))
                        tma_store_4d(t == 0 ? &tmDQ : t == 1 ? &tmDK : &tmDV, base + t * L::kTile + hh * 16384 + s * p.slot * 128,
                                     hh * 64, hf ? h : 0, hf ? 0 : h, b);
                }
                tma_store_commit();
                tma_store_wait_read0();
            }
            __syncwarp();
        } else {
            // -------------------------------------------------------------- row workers
            const int q4 = warp & 3, part = warp >> 2, row = q4 * 32 + lane;
            const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
            // norms: the first half of the warps the rows of q, the second those of k, kHalves threads (lanes l and
            // l ^ 16) a row
            const int w0 = warp % (NW / 2), isk = warp / (NW / 2);
            const int nrow = L::kHalves == 1 ? w0 * 32 + lane : w0 * 16 + (lane & 15);
            constexpr int kCh = D / 8 / L::kHalves;
            const int ch0 = L::kHalves == 1 ? 0 : (lane >> 4) * kCh;
            // Rows that no copy writes are zeroed: in q or k by the threads that take their norm, which so read what they
            // wrote themselves, and in v or dO alike.
            // (After the first pass: once the copies are on their way, behind which the rows before them have left.)
            if (pass > 0 && !wait(B_FULL, par)) break;
            if (nrow < s0 * p.slot || nrow >= s1 * p.slot) {
#pragma unroll 1
                for (int t = isk; t < 4; t += 2)
#pragma unroll 1
                    for (int j = ch0; j < ch0 + kCh; ++j)
                        *reinterpret_cast<uint4*>(gbase + t * L::kTile + (j >> 3) * 16384 + swz(nrow, j & 7)) = make_uint4(0, 0, 0, 0);
            }
            // the row's sequence: (b, h), factor, first and last column it keeps
            const int seq = row / p.slot, tok = row - seq * p.slot, pair = pair0 + seq;
            const bool live = seq >= s0 && seq < s1 && tok < p.N;
            float cfac = 0.f;
            if (live) {
                const int b = pair / p.H;
                const float s_b = p.seq_len ? p.seq_len[b] : (p.seq_len_scalar > 0.f ? p.seq_len_scalar : (float)p.N);
                cfac = stab_factor(p.m[pair - b * p.H], s_b);
            }
            const int lo = seq * p.slot, hi = live ? (p.causal ? row : lo + p.N - 1) : -1;
            if (wait(B_FULL, par)) {
                uint8_t* tile = gbase + (isk ? L::kOffK : L::kOffQ);
                float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll 1
                for (int j = ch0; j < ch0 + kCh; j += 4) {
                    uint4 w[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const uint4*>(tile + (j >> 3) * 16384 + swz(nrow, (j & 7) + i));
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float2 f0 = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[i]);
                        const float2 f1 = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[i + 1]);
                        a0 = __ffma2_rn(f0, f0, a0); a1 = __ffma2_rn(f1, f1, a1);
                    }
                }
                float ss = (a0.x + a0.y) + (a1.x + a1.y);
                if (L::kHalves > 1) ss += __shfl_xor_sync(0xffffffffu, ss, 16);
                const float nrm = sqrtf(ss), r = 1.0f / fmaxf(nrm, kEps);
                // A row too long for fp32 has r = 0, that is a unit row of zeros, and its scores may be infinite: it
                // becomes zeros here, so that they are 0 as well.  (A row that is not finite stays.)
                const uint32_t too_long = __ballot_sync(0xffffffffu, !(ss <= 3.4028235e38f));
                if (too_long >> lane & 1) {
                    bool finite = true;
#pragma unroll 1
                    for (int j = ch0; j < ch0 + kCh; ++j) {
                        const uint4 w = *reinterpret_cast<const uint4*>(tile + (j >> 3) * 16384 + swz(nrow, j & 7));
                        for (uint32_t x : {w.x, w.y, w.z, w.w})
                            finite = finite && (x & 0x7f80u) != 0x7f80u && (x & 0x7f800000u) != 0x7f800000u;
                    }
                    if (L::kHalves > 1) finite = __shfl_xor_sync(too_long, finite ? 1 : 0, 16) && finite;
#pragma unroll 1
                    for (int j = ch0; j < ch0 + kCh && finite; ++j)
                        *reinterpret_cast<uint4*>(tile + (j >> 3) * 16384 + swz(nrow, j & 7)) = make_uint4(0, 0, 0, 0);
                }
                if (ch0 == 0) (isk ? rk_buf : rq_buf)[nrow] = nrm > kEps ? r : -r;
                fence_proxy_async();
                mbar_arrive(bars + B_NR);
            }
            // masked scores, this thread's columns: P to its buffer, G kept (or to its own)
            constexpr int kCols = 128 / L::kParts;
            const int col0 = part * kCols;
            uint32_t gk[kCols / 2];
            if (wait(B_NR, par) && wait(B_SF, par)) {
                tc_fence_after();
                const float rq = fabsf(rq_buf[row]);
                float2 all = make_float2(0.f, 0.f);      // not finite if any score is not
                float t_sum = 0.f;
#pragma unroll
                for (int pc = 0; pc < kCols / 16; ++pc) {
                    const int c0 = col0 + pc * 16;
                    float2 x[8], g[8];
                    tmem_ld16(tmem + lane_base + L::colP + c0, reinterpret_cast<uint32_t*>(x));
                    tmem_ld16(tmem + lane_base + L::colG + c0, reinterpret_cast<uint32_t*>(g));
                    tmem_wait_ld();
                    uint32_t pk[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int ja = c0 + 2 * i, jb = ja + 1;
                        all = __fadd2_rn(all, __fadd2_rn(x[i], g[i]));
                        const float2 rk = *reinterpret_cast<const float2*>(&rk_buf[ja]);
                        const float sa = rq * fabsf(rk.x), sb = rq * fabsf(rk.y);
                        const bool ka = ja >= lo && ja <= hi, kb = jb >= lo && jb <= hi;
                        const float pa = ka ? x[i].x * sa : 0.f, pb = kb ? x[i].y * sb : 0.f;
                        const float ga = ka ? g[i].x : 0.f, gb = kb ? g[i].y : 0.f;
                        t_sum = fmaf(pa, ga, t_sum);
                        t_sum = fmaf(pb, gb, t_sum);
                        pk[i] = pack_bf16(pa, pb);
                        gk[pc * 8 + i] = pack_bf16(ka ? ga * sa : 0.f, kb ? gb * sb : 0.f);
                    }
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        *reinterpret_cast<uint4*>(gbase + L::kOffP + (c0 >> 6) * 16384 + swz(row, ((c0 & 63) >> 3) + i)) =
                            make_uint4(pk[4 * i], pk[4 * i + 1], pk[4 * i + 2], pk[4 * i + 3]);
                }
                t_buf[part * 128 + row] = t_sum;
                if (!(fabsf(all.x) <= 3.4028235e38f && fabsf(all.y) <= 3.4028235e38f)) *bad_flag = 1;
                if (L::kTwo) {
#pragma unroll
                    for (int j = 0; j < kCols / 8; ++j)
                        *reinterpret_cast<uint4*>(gbase + L::kOffG + (col0 >> 6) * 16384 + swz(row, ((col0 & 63) >> 3) + j)) =
                            make_uint4(gk[4 * j], gk[4 * j + 1], gk[4 * j + 2], gk[4 * j + 3]);
                }
                fence_proxy_async();
                tc_fence_before();
                mbar_arrive(bars + B_R1);
            }
            if (!L::kTwo && wait(B_VF, par)) {
                // (the product that read P is done: G takes its buffer)
#pragma unroll
                for (int j = 0; j < kCols / 8; ++j)
                    *reinterpret_cast<uint4*>(gbase + L::kOffG + (col0 >> 6) * 16384 + swz(row, ((col0 & 63) >> 3) + j)) =
                        make_uint4(gk[4 * j], gk[4 * j + 1], gk[4 * j + 2], gk[4 * j + 3]);
                fence_proxy_async();
                mbar_arrive(bars + B_R2);
            }
            // (the flag and the sums of the other parts of a row are there with B_R1, which is long complete)
            if (wait(B_OF, par) && wait(B_R1, par)) {
                const bool skip = pass == 0 && n_seq > 1 && *bad_flag;
                if (skip) {
                    n_pass = 1 + n_seq;
                    if (L::kHalves > 1) mbar_arrive(bars + B_XR);
                } else {
                    tc_fence_after();
                    // ---- dq (first half of the warps), dk (second half), kHalves threads a row; over the raw row
                    const int half = part % L::kHalves;
                    constexpr int kEc = D / L::kHalves;                       // columns of a thread
                    uint8_t* tile = gbase + (isk ? L::kOffK : L::kOffQ);
                    const uint32_t tacc = tmem + lane_base + (isk ? L::colB : L::colA);
                    const float r = (isk ? rk_buf : rq_buf)[row];
                    float2 d2 = make_float2(0.f, 0.f);
#pragma unroll 1
                    for (int pc = 0; pc < kEc / 16; ++pc) {
                        const int c0 = half * kEc + pc * 16;
                        float2 a[8];
                        tmem_ld16(tacc + c0, reinterpret_cast<uint32_t*>(a));
                        uint4 w[2];
#pragma unroll
                        for (int i = 0; i < 2; ++i) w[i] = *reinterpret_cast<const uint4*>(tile + (c0 >> 6) * 16384 + swz(row, ((c0 & 63) >> 3) + i));
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            d2 = __ffma2_rn(__bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[i]), a[i], d2);
                    }
                    float dot = d2.x + d2.y;
                    if (L::kHalves > 1) {
                        float* x_buf = reinterpret_cast<float*>(gbase + L::kOffCtl + L::kOffX) + isk * 256;
                        x_buf[half * 128 + row] = dot;
                        mbar_arrive(bars + B_XR);
                        if (!wait(B_XR, par)) break;
                        dot = x_buf[row] + x_buf[128 + row];
                    }
                    const float mc = r > 0.f ? -cfac * dot * r * r : 0.f;
                    const float2 sc2 = make_float2(cfac, cfac), mc2 = make_float2(mc, mc);
#pragma unroll 1
                    for (int pc = 0; pc < kEc / 16; ++pc) {
                        const int c0 = half * kEc + pc * 16;
                        float2 a[8];
                        tmem_ld16(tacc + c0, reinterpret_cast<uint32_t*>(a));
                        uint4 w[2], o[2];
#pragma unroll
                        for (int i = 0; i < 2; ++i) w[i] = *reinterpret_cast<const uint4*>(tile + (c0 >> 6) * 16384 + swz(row, ((c0 & 63) >> 3) + i));
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float2 v = __ffma2_rn(__bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w)[i]), mc2, __fmul2_rn(a[i], sc2));
                            reinterpret_cast<uint32_t*>(o)[i] = pack_bf16(v.x, v.y);
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i) *reinterpret_cast<uint4*>(tile + (c0 >> 6) * 16384 + swz(row, ((c0 & 63) >> 3) + i)) = o[i];
                    }
                    // ---- dv, all threads of the row, over v
#pragma unroll 1
                    for (int pc = 0; pc < D / L::kParts / 16; ++pc) {
                        const int c0 = part * (D / L::kParts) + pc * 16;
                        float2 a[8];
                        tmem_ld16(tmem + lane_base + L::colV + c0, reinterpret_cast<uint32_t*>(a));
                        tmem_wait_ld();
                        uint4 o[2];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float2 v = __fmul2_rn(a[i], sc2);
                            reinterpret_cast<uint32_t*>(o)[i] = pack_bf16(v.x, v.y);
                        }
#pragma unroll
                        for (int i = 0; i < 2; ++i)
                            *reinterpret_cast<uint4*>(gbase + L::kOffV + (c0 >> 6) * 16384 + swz(row, ((c0 & 63) >> 3) + i)) = o[i];
                    }
                    // ---- T of every sequence of the pass, one warp each, fixed order
                    for (int s = s0 + warp; s < s1; s += NW) {
                        float t = 0.f;
                        for (int i = lane; i < p.N; i += 32)
#pragma unroll
                            for (int x = 0; x < L::kParts; ++x) t += t_buf[x * 128 + s * p.slot + i];
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                        if (lane == 0) p.dm_partial[pair0 + s] = t;
                    }
                    fence_proxy_async();
                }
                tc_fence_before();
                mbar_arrive(bars + B_ED);
            }
        }
    }
    if (is_ctrl) tma_store_wait_all0();
    tc_fence_before();
    __syncthreads();
    {
        volatile int* last_flag = reinterpret_cast<volatile int*>(gbase + L::kOffCtl + L::kOffLast);
        if (tid == 0) {
            __threadfence();
            *last_flag = atomicAdd(&p.status[4], 1) == (int)gridDim.x - 1;
        }
        __syncthreads();
        if (*last_flag) {
            // dm_h = sum_b dc/dm(b,h) T_{b,h}, dc/dm = -ln(s_b) sigma(m_h) (1 - sigma(m_h)) c_{b,h}; fixed order.
            __threadfence();
            const int n_b = p.BH / p.H;
            for (int hh = warp; hh < p.H; hh += kThreads / 32) {
                const float sg = 1.0f / (1.0f + expf(-p.m[hh]));
                float sum = 0.f;
                for (int b = lane; b < n_b; b += 32) {
                    const float ls = logf(p.seq_len ? p.seq_len[b] : (p.seq_len_scalar > 0.f ? p.seq_len_scalar : (float)p.N));
                    sum += __ldcg(&p.dm_partial[b * p.H + hh]) * (-ls * sg * (1.0f - sg) * expf(-sg * ls));
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
                if (lane == 0) p.dm_out[hh] = sum;
            }
            if (tid == 0) p.status[4] = 0;
        }
    }
    if (*abort_flag) {
        // A wait gave up: let the copies and products in flight land, then report where.
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
        __syncthreads();
        if (tid == 0 && atomicCAS(p.status, 0, 1) == 0) {
            p.status[1] = *abort_flag;
            p.status[2] = (int)blockIdx.x | (9 << 24);
        }
    }
    if (is_ctrl) tmem_dealloc(tmem, L::kTmemCols);
}

template <int D, int NW>
cudaError_t launch_d(const CUtensorMap* tm, const ShortBwdParams& p, int tiles, cudaStream_t st) {
    auto kern = tc_short_bwd_kernel<D, NW>;
    if (cudaError_t e = configure_smem_once(reinterpret_cast<const void*>(kern), SBL<D, NW>::kDynBytes); e != cudaSuccess) return e;
    const int prof = profile_begin_launch(8, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles);
    cfg.blockDim = dim3(SBL<D, NW>::kThreads);
    cfg.dynamicSmemBytes = SBL<D, NW>::kDynBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t le = cudaLaunchKernelEx(&cfg, kern, tm[0], tm[1], tm[2], tm[3], tm[4], tm[5], tm[6], p);
    profile_end_launch(prof, st);
    note_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
}

}  // namespace

cudaError_t launch_tc_short_bwd(const TcBwdFusedArgs& a, int B, int H, int N, int d, cudaStream_t st) {
    const void* ptrs[7] = {a.q, a.k, a.v, a.d_o, a.dq, a.dk, a.dv};
    const RowLayout lays[7] = {a.l_qkv, a.l_qkv, a.l_v, a.l_do, a.l_dqkv, a.l_dqkv, a.l_dv};
    const int wk = a.w_k > 0 ? a.w_k : d, wv = a.w_v > 0 ? a.w_v : d;
    const int dims[7] = {wk, wk, wv, wv, wk, wk, wv};
    if (N < 1 || N > kRows || (d != 64 && d != 128) || wk > d || wv > d) return cudaErrorInvalidValue;
    ShortBwdParams p;
    p.slot = (N + 7) / 8 * 8;
    p.seqs = kRows / p.slot;
    CUtensorMap tm[7];
    p.head_first_mask = 0;
    for (int i = 0; i < 7; ++i) {
        bool hf = false;
        if (!make_tile_map(&tm[i], ptrs[i], B, H, N, dims[i], lays[i], &hf, p.slot)) return cudaErrorInvalidValue;
        p.head_first_mask |= (hf ? 1 : 0) << i;
    }
    p.dm_partial = a.dm_partial; p.dm_out = a.dm_out; p.status = a.status;
    p.m = a.m; p.seq_len = a.seq_len; p.seq_len_scalar = a.seq_len_scalar;
    p.H = H; p.N = N; p.BH = B * H;
    p.causal = a.bidir ? 0 : 1;
    p.wk = wk; p.wv = wv;
    p.wait_limit_kcycles = wait_limit_kcycles();
    const int tiles = (p.BH + p.seqs - 1) / p.seqs;
    if (d == 128) return launch_d<128, 16>(tm, p, tiles, st);
    return tiles <= 148 ? launch_d<64, 16>(tm, p, tiles, st) : launch_d<64, 8>(tm, p, tiles, st);
}

}  // namespace cott
