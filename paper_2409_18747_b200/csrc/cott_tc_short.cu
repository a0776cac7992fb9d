// Short sequences (N <= 128 tokens, bf16 I/O, fp32 accumulation): the left-hand, quadratic side
// of Eq. 5 / the masked product of Eq. 6 with no running state at all.  The paper notes that
// this side is the cheaper one when the sequence is shorter than the head size; here the
// threshold is the 128-token tile of the tensor core.
//
// The rows of all (b, h) pairs of a dense [B,H,N,d] tensor are one long list of B H N rows, so a
// tile of 128 rows holds k = floor(128 / N) whole sequences of consecutive pairs.  In other memory
// orders (PLACES) a sequence is a copy of its own, in a place of N rows rounded up to eight (the
// swizzle pattern's period).  One CTA per tile: a single score product P = Q K^^T (128 x 128), a
// block-diagonal mask -- a row keeps the columns of its own sequence, up to and including its own
// position when causal --, a single product O = P~ V, rows scaled by c / max(||q||, eps) (Eq. 2-4) and
// stored.  No state update, no state copy, no second launch; B H / k CTAs instead of B H, four (d = 64)
// or two per SM.  A row that is not finite stays in its own sequence (the passes below).
// Bound by the chain of one CTA (tiles, norms, scores, mask, product, rows out), hence by how many share
// an SM: B=64, H=12, N=77, d=64 14.1 us (18.2 with two), B=256, H=12, N=100 45.6 (65).
// In [B,N,H,d] storage, against a CTA per (b, h): 39 x 12 sequences of 18 tokens, d = 128, bidirectional 50.6 ->
// 7.6 us, causal 22.7 -> 7.6; d = 64 18.1 -> 6.0.
#include "cott_internal.h"
#include "cott_sm100.cuh"
#include "cott_tc_common.cuh"

namespace cott {

using namespace sm100;
using namespace tc;

namespace {

constexpr int kRows = 128;                    // rows of a tile
constexpr int kWorkerWarps = 8;
constexpr int kThreads = (kWorkerWarps + 1) * 32;     // + control warp (copies and products)

template <int D>
struct SL {
    static constexpr int kTile = kRows * D * 2;       // D / 64 boxes of 128 rows x 64 columns
    static constexpr int kOffQ = 0, kOffK = kTile, kOffV = 2 * kTile;
    static constexpr int kOffCtl = 3 * kTile;
    static constexpr int kOffBad = 480;               // flag: some output of the first pass is not finite
    static constexpr int kOffRx = 1024;               // float [128]: 1 / max(||q||, eps), behind the barriers
    static constexpr int kDynBytes = kOffCtl + kOffRx + 512 + 1024;
    // D = 64: the masked scores are packed over the start of the scores and the output accumulator takes
    // their second half: 128 tensor-memory columns, so that four CTAs share an SM; D = 128, whose shared
    // memory allows two, keeps them apart.
    static constexpr int kTmemCols = D == 64 ? 128 : 256;
    static constexpr int kCtas = D == 64 ? 4 : 2;
};

struct ShortParams {
    int* status;
    const float* m; const float* seq_len; float seq_len_scalar;
    int H; int N; int BH;
    int seqs_per_tile;       // k
    int slot;                // rows of a sequence's place in a tile
    int head_first_mask;     // PLACES: bit i: in tensor map i (q, k, v, o) the head index comes before the token index
    int causal;
    int d_out;               // columns o really has
    int wait_limit_kcycles;
};

// What a tile holds: one sequence of dense tensors, several (which may have to be kept apart), or sequences in places
// of their own.
enum Tile { ONE, SEVERAL, PLACES };

template <int D, Tile TILE>
__global__ void __launch_bounds__(kThreads, SL<D>::kCtas)
tc_short_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO, ShortParams p) {
    using L = SL<D>;
    constexpr int NH = D / 64;
    constexpr bool SLOTS = TILE == PLACES;
    // Tensor-memory columns, D = 128: scores, later the output accumulator 0..127 | masked bf16 scores 128..191.
    // D = 64: scores 0..127, then masked bf16 scores 0..63 | output accumulator 64..127.
    constexpr uint32_t colP = 0, colPt = D == 64 ? 0 : 128, colO = D == 64 ? 64 : 0;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t bars = base + L::kOffCtl;
    enum { B_FULL = 0, B_KREADY = 8, B_PFULL = 16, B_PTREADY = 24, B_OFULL = 32, B_EDONE = 40, B_SIB = 48 /* [4 quadrants] */ };
    volatile int* bad_flag = reinterpret_cast<volatile int*>(gbase + L::kOffCtl + L::kOffBad);
    const uint32_t tmem_slot = bars + kCtlTmemSlot;
    volatile uint32_t* tmem_slot_g = reinterpret_cast<volatile uint32_t*>(gbase + L::kOffCtl + kCtlTmemSlot);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + L::kOffCtl + kCtlAbort);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool is_ctrl = warp == kWorkerWarps;
    const int row0 = (int)blockIdx.x * p.seqs_per_tile * p.N; // dense: first row of the tile in the list of B H N rows
    const int pair0 = (int)blockIdx.x * p.seqs_per_tile;
    const int n_seq = SLOTS ? min(p.seqs_per_tile, p.BH - pair0) : TILE == ONE ? 1 : p.seqs_per_tile;

    if (is_ctrl) {
        tmem_alloc(tmem_slot, L::kTmemCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(bars + B_FULL, 1);
        mbar_init(bars + B_KREADY, 256);
        mbar_init(bars + B_PFULL, 1);
        mbar_init(bars + B_PTREADY, 256);
        mbar_init(bars + B_OFULL, 1);
        mbar_init(bars + B_EDONE, 256);
        for (int i = 0; i < 4; ++i) mbar_init(bars + B_SIB + 8 * i, 32);
        *abort_flag = 0;
        *bad_flag = 0;
        abort_flag[3] = p.wait_limit_kcycles;
        mbar_fence_init();
        fence_proxy_async();
    }
    if (is_ctrl && lane == 0) {
        tma_prefetch_desc(&tmQ); tma_prefetch_desc(&tmK); tma_prefetch_desc(&tmV); tma_prefetch_desc(&tmO);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot_g;
    // The only kernel of its call: it may follow a kernel that produced its inputs.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0 && tid < 8) p.status[tid] = 0;

    // PLACES: a pass takes the sequences s0 .. s1 - 1 of the tile: all of them, once.  Sequences that share a tile
    // meet in the second product as zeros times each other's v rows, which is no zero where a row is not finite:
    // then (some output is not finite) the first pass is not stored and every sequence gets a pass of its own.
    // (Dense tensors, where one copy brings the rows of all sequences: one pass, and the second product again below.)
    int n_pass = 1;
    for (int pass = 0; pass < (SLOTS ? n_pass : 1); ++pass) {
        const uint32_t par = (uint32_t)(pass & 1);
        const int s0 = pass == 0 ? 0 : pass - 1, s1 = pass == 0 ? n_seq : pass;
        if (is_ctrl) {
            bool go = true;
            if (SLOTS) {
                // One copy per sequence, tensor and half tile, over the lanes (rows past N read as zero).
                if (lane == 0) mbar_expect_tx(bars + B_FULL, (uint32_t)((s1 - s0) * p.slot) * 128u * 3u * NH);
                __syncwarp();
                for (int i = lane; i < (s1 - s0) * 3 * NH; i += 32) {
                    const int sq = s0 + i / (3 * NH), r = i % (3 * NH), t = r / NH, hh = r % NH, pair = pair0 + sq;
                    const int b = pair / p.H, h = pair - b * p.H;
                    const bool hf = (p.head_first_mask >> t) & 1;
                    tma_load_4d(base + t * L::kTile + hh * 16384 + sq * p.slot * 128, t == 0 ? &tmQ : t == 1 ? &tmK : &tmV, bars + B_FULL,
                                hh * 64, hf ? h : 0, hf ? 0 : h, b);
                }
            }
            if (lane == 0) {
                if (!SLOTS) {
                    // The copies bring the rows of all sequences per box; the rows below them are zeroed by the workers.
                    const uint32_t fb = bars + B_FULL;
                    mbar_expect_tx(fb, 3u * NH * (uint32_t)(p.seqs_per_tile * p.N) * 128u);
#pragma unroll
                    for (int hh = 0; hh < NH; ++hh) {
                        tma_load_4d(base + L::kOffQ + hh * 16384, &tmQ, fb, hh * 64, row0, 0, 0);
                        tma_load_4d(base + L::kOffK + hh * 16384, &tmK, fb, hh * 64, row0, 0, 0);
                        tma_load_4d(base + L::kOffV + hh * 16384, &tmV, fb, hh * 64, row0, 0, 0);
                    }
                }
                bool ok = wait_or_abort(bars + B_KREADY, par, abort_flag);
                if (ok) {
                    // P = Q K^^T: both operands K-major
                    tc_fence_after();
                    constexpr uint32_t idesc = instr_desc_bf16(128, 128, false, false);
                    const uint32_t xl = smem_desc_lo(base + L::kOffQ, 16), al = smem_desc_lo(base + L::kOffK, 16);
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint32_t off = ((kk >> 2) * 16384u + (kk & 3) * 32u) >> 4;
                        mma_ss_w(tmem + colP, xl + off, kDescHi, al + off, kDescHi, idesc, kk > 0);
                    }
                    tc_commit(bars + B_PFULL);
                    ok = wait_or_abort(bars + B_PTREADY, par, abort_flag);
                }
                if (ok) {
                    // O = P~ V: P~ from tensor memory (8 columns per K = 16), V MN-major; the
                    // accumulator takes columns of the scores, which every worker has read
                    tc_fence_after();
                    constexpr uint32_t idesc = instr_desc_bf16(128, D, false, true);
                    const uint32_t bl = smem_desc_lo(base + L::kOffV, 16384);
#pragma unroll
                    for (int kk = 0; kk < kRows / 16; ++kk)
                        mma_ts_w(tmem + colO, tmem + colPt + kk * 8u, bl + kk * 128u, kDescHi, idesc, kk > 0);
                    tc_commit(bars + B_OFULL);
                    ok = wait_or_abort(bars + B_EDONE, par, abort_flag);
                }
                if (ok && !SLOTS && !(TILE == SEVERAL && *bad_flag)) {
#pragma unroll
                    for (int hh = 0; hh < NH; ++hh)
                        if (hh * 64 < p.d_out) tma_store_4d(&tmO, base + L::kOffQ + hh * 16384, hh * 64, row0, 0, 0);
                    tma_store_commit();
                    tma_store_wait_all0();
                }
                go = ok;
            }
            if (SLOTS) {
                if (!__shfl_sync(0xffffffffu, go ? 1 : 0, 0)) break;
                // (long complete: the staged rows and the flag, which lane 0 alone has waited for, are shown to the lanes that store)
                if (!wait_or_abort(bars + B_EDONE, par, abort_flag)) break;
                if (pass == 0 && n_seq > 1 && *bad_flag) {
                    n_pass = 1 + n_seq;
                } else {
                    for (int i = lane; i < (s1 - s0) * NH; i += 32) {
                        const int sq = s0 + i / NH, hh = i % NH, pair = pair0 + sq;
                        const int b = pair / p.H, h = pair - b * p.H;
                        const bool hf = (p.head_first_mask >> 3) & 1;
                        if (hh * 64 < p.d_out)
                            tma_store_4d(&tmO, base + L::kOffQ + hh * 16384 + sq * p.slot * 128, hh * 64, hf ? h : 0, hf ? 0 : h, b);
                    }
                    tma_store_commit();
                    tma_store_wait_read0();
                }
                __syncwarp();
            }
        } else {
            // ------------------------------------------------------------------ row workers
            // TMEM lane quadrant q4 = warp & 3, column half hf = warp >> 2: two threads per row.
            bool alive = true;
            auto wait = [&](uint32_t bar_, uint32_t parity) {
                if (alive && !wait_or_abort(bar_, parity, abort_flag)) alive = false;
                return alive;
            };
            const int q4 = warp & 3, hf = warp >> 2, row = q4 * 32 + lane;
            const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
            // rows the copies do not write: zero (a zero v row times a zero score must not be NaN)
            // (two lanes, l and l ^ 16, share a row here and in the row norms, half of it each)
            const int nrow = warp * 16 + (lane & 15), half = lane >> 4;
            if (pass > 0 && !wait(bars + B_FULL, par)) break;     // (behind which the rows of the pass before have left)
            if (nrow < s0 * p.slot || nrow >= s1 * p.slot) {
#pragma unroll
                for (int j = 0; j < 4 * NH; ++j) {
                    const int ch = half * 4 * NH + j;                     // 16-byte chunk of the row
                    const uint32_t off = (ch >> 3) * 16384u + swz(nrow, ch & 7);
                    *reinterpret_cast<uint4*>(gbase + L::kOffQ + off) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4*>(gbase + L::kOffK + off) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4*>(gbase + L::kOffV + off) = make_uint4(0, 0, 0, 0);
                }
            }
            // the row's sequence: pair index, scaling factor, first row of the sequence in the tile
            const int seq = row / p.slot, pair = pair0 + seq;
            const bool live = seq >= s0 && seq < s1 && row - seq * p.slot < p.N && pair < p.BH;
            float cfac = 0.f;
            if (live) {
                const int b = pair / p.H, h = pair % p.H;
                const float s_b = p.seq_len ? p.seq_len[b] : (p.seq_len_scalar > 0.f ? p.seq_len_scalar : (float)p.N);
                cfac = stab_factor(p.m[h], s_b);
            }
            const int lo = seq * p.slot, hi = live ? (p.causal ? row : lo + p.N - 1) : -1;
            float* rq_buf = reinterpret_cast<float*>(gbase + L::kOffCtl + L::kOffRx);
            if (wait(bars + B_FULL, par)) {
                // ||q|| and ||k||; k is normalised in place
                float2 sq = make_float2(0.f, 0.f), sk = sq;
#pragma unroll
                for (int j = 0; j < 4 * NH; ++j) {
                    const int ch = half * 4 * NH + j;
                    const uint32_t off = (ch >> 3) * 16384u + swz(nrow, ch & 7);
                    const uint4 wq = *reinterpret_cast<const uint4*>(gbase + L::kOffQ + off);
                    const uint4 wk = *reinterpret_cast<const uint4*>(gbase + L::kOffK + off);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 fq = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&wq)[i]);
                        const float2 fk = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&wk)[i]);
                        sq = __ffma2_rn(fq, fq, sq); sk = __ffma2_rn(fk, fk, sk);
                    }
                }
                float nq = sq.x + sq.y, nk = sk.x + sk.y;
                nq += __shfl_xor_sync(0xffffffffu, nq, 16);
                nk += __shfl_xor_sync(0xffffffffu, nk, 16);
                if (half == 0) rq_buf[nrow] = 1.0f / fmaxf(sqrtf(nq), kEps);
                const float rk = 1.0f / fmaxf(sqrtf(nk), kEps);
#pragma unroll
                for (int j = 0; j < 4 * NH; ++j) {
                    const int ch = half * 4 * NH + j;
                    uint4* pk = reinterpret_cast<uint4*>(gbase + L::kOffK + (ch >> 3) * 16384u + swz(nrow, ch & 7));
                    uint4 w = *pk;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        __nv_bfloat162& e = reinterpret_cast<__nv_bfloat162*>(&w)[i];
                        e = scale_round(e, rk);
                    }
                    *pk = w;
                }
                fence_proxy_async();
                mbar_arrive(bars + B_KREADY);
            }
            if (wait(bars + B_PFULL, par)) {
                // block-diagonal (causal) mask on this thread's 64 columns, packed to bf16 pairs
                tc_fence_after();
#pragma unroll 1
                for (int pc = 0; pc < 2; ++pc) {
                    const int c0 = hf * 64 + pc * 32;
                    uint32_t r[32];
                    tmem_ld32(tmem + lane_base + colP + c0, r);
                    tmem_wait_ld();
                    uint32_t pk[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const int ja = c0 + 2 * j, jb = ja + 1;
                        const float a = (ja >= lo && ja <= hi) ? __uint_as_float(r[2 * j]) : 0.f;
                        const float b2 = (jb >= lo && jb <= hi) ? __uint_as_float(r[2 * j + 1]) : 0.f;
                        pk[j] = pack_bf16(a, b2);
                    }
                    // (D = 64: columns 32-63, which the hf = 1 warp writes, hold scores of the hf = 0 warp)
                    if (D == 64 && hf == 0 && pc == 1) { tc_fence_before(); mbar_arrive(bars + B_SIB + 8 * q4); }
                    if (D == 64 && hf == 1 && pc == 0) { if (!wait(bars + B_SIB + 8 * q4, par)) break; tc_fence_after(); }
                    tmem_st16(tmem + lane_base + colPt + (c0 >> 1), pk);
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(bars + B_PTREADY);
            }
            if (wait(bars + B_OFULL, par)) {
                // this thread's D / 2 accumulator columns: scale, round, stage where q was
                tc_fence_after();
                const float rx = cfac * rq_buf[row];
                float finite = 0.f;
#pragma unroll 1
                for (int pc = 0; pc < D / 64; ++pc) {
                    const int c0 = hf * (D / 2) + pc * 32;
                    uint32_t a[32];
                    tmem_ld32(tmem + lane_base + colO + c0, a);
                    tmem_wait_ld();
                    if (TILE != ONE) {
                        const float2 zero = make_float2(0.f, 0.f);
                        float2 f0 = zero, f1 = zero;
#pragma unroll
                        for (int j = 0; j < 32; j += 4) {
                            f0 = __ffma2_rn(make_float2(__uint_as_float(a[j]), __uint_as_float(a[j + 1])), zero, f0);
                            f1 = __ffma2_rn(make_float2(__uint_as_float(a[j + 2]), __uint_as_float(a[j + 3])), zero, f1);
                        }
                        finite += (f0.x + f0.y) + (f1.x + f1.y);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint4 o;
                        o.x = pack_bf16(__uint_as_float(a[8 * j]) * rx, __uint_as_float(a[8 * j + 1]) * rx);
                        o.y = pack_bf16(__uint_as_float(a[8 * j + 2]) * rx, __uint_as_float(a[8 * j + 3]) * rx);
                        o.z = pack_bf16(__uint_as_float(a[8 * j + 4]) * rx, __uint_as_float(a[8 * j + 5]) * rx);
                        o.w = pack_bf16(__uint_as_float(a[8 * j + 6]) * rx, __uint_as_float(a[8 * j + 7]) * rx);
                        const int ch = (c0 >> 3) + j;
                        *reinterpret_cast<uint4*>(gbase + L::kOffQ + (ch >> 3) * 16384u + swz(row, ch & 7)) = o;
                    }
                }
                if (TILE != ONE && !(finite == 0.f)) *bad_flag = 1;
                fence_proxy_async();
                tc_fence_before();
                mbar_arrive(bars + B_EDONE);
            }
            if (SLOTS && n_seq > 1) {
                if (!wait(bars + B_EDONE, par)) break;
                if (pass == 0 && *bad_flag) n_pass = 1 + n_seq;
            }
        }
    }
    if (SLOTS && is_ctrl) tma_store_wait_all0();
    tc_fence_before();
    __syncthreads();
    if (TILE == SEVERAL && *bad_flag && !*abort_flag) {
        // The tile has not been stored: one sequence after the other, the masked scores, in tensor memory still, times
        // v with the rows of the other sequences zeroed.  (FULL and OFULL have completed one phase.)
        const int q4 = warp & 3, hf = warp >> 2, row = q4 * 32 + lane, pair = pair0 + row / p.N;
        bool ok = true;
        for (int sq = 0; sq < n_seq; ++sq) {
            const uint32_t par = (uint32_t)(~sq & 1);
            const int r0 = sq * p.N, r1 = r0 + p.N;
            if (is_ctrl && lane == 0) {
                mbar_expect_tx(bars + B_FULL, NH * (uint32_t)(n_seq * p.N) * 128u);
                for (int hh = 0; hh < NH; ++hh) tma_load_4d(base + L::kOffV + hh * 16384, &tmV, bars + B_FULL, hh * 64, row0, 0, 0);
            }
            ok = wait_or_abort(bars + B_FULL, par, abort_flag);
            if (!is_ctrl && (row < r0 || row >= r1))
                for (int ch = hf * 4 * NH; ch < (hf + 1) * 4 * NH; ++ch)
                    *reinterpret_cast<uint4*>(gbase + L::kOffV + (ch >> 3) * 16384u + swz(row, ch & 7)) = make_uint4(0, 0, 0, 0);
            fence_proxy_async();
            if (__syncthreads_or(!ok)) { ok = false; break; }
            if (is_ctrl && lane == 0) {
                tc_fence_after();
                constexpr uint32_t idesc = instr_desc_bf16(128, D, false, true);
                const uint32_t bl = smem_desc_lo(base + L::kOffV, 16384);
                for (int kk = 0; kk < kRows / 16; ++kk)
                    mma_ts_w(tmem + colO, tmem + colPt + kk * 8u, bl + kk * 128u, kDescHi, idesc, kk > 0);
                tc_commit(bars + B_OFULL);
            }
            ok = wait_or_abort(bars + B_OFULL, par, abort_flag);
            tc_fence_after();
            if (!is_ctrl) {
                float rx = 0.f;
                if (row >= r0 && row < r1 && pair < p.BH) {
                    const int b = pair / p.H;
                    const float s_b = p.seq_len ? p.seq_len[b] : (p.seq_len_scalar > 0.f ? p.seq_len_scalar : (float)p.N);
                    rx = stab_factor(p.m[pair - b * p.H], s_b) * reinterpret_cast<const float*>(gbase + L::kOffCtl + L::kOffRx)[row];
                }
#pragma unroll 1
                for (int pc = 0; pc < D / 32; ++pc) {
                    const int c0 = hf * (D / 2) + pc * 16;
                    float a[16];
                    __syncwarp();
                    tmem_ld16(tmem + ((uint32_t)(q4 * 32) << 16) + colO + c0, reinterpret_cast<uint32_t*>(a));
                    tmem_wait_ld();
                    uint4 o[2];
#pragma unroll
                    for (int j = 0; j < 8; ++j) reinterpret_cast<uint32_t*>(o)[j] = pack_bf16(a[2 * j] * rx, a[2 * j + 1] * rx);
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        if (row >= r0 && row < r1)
                            *reinterpret_cast<uint4*>(gbase + L::kOffQ + (c0 >> 6) * 16384u + swz(row, ((c0 & 63) >> 3) + j)) = o[j];
                }
            }
            fence_proxy_async();
            tc_fence_before();
            if (__syncthreads_or(!ok)) { ok = false; break; }
        }
        if (ok && is_ctrl && lane == 0) {
            for (int hh = 0; hh < NH; ++hh)
                if (hh * 64 < p.d_out) tma_store_4d(&tmO, base + L::kOffQ + hh * 16384, hh * 64, row0, 0, 0);
            tma_store_commit();
            tma_store_wait_all0();
        }
        __syncthreads();
    }
    if (*abort_flag) {
        // A wait gave up: let the copies and products in flight land, then report where.
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
        __syncthreads();
        if (tid == 0 && atomicCAS(p.status, 0, 1) == 0) {
            p.status[1] = *abort_flag;
            p.status[2] = (int)blockIdx.x | (6 << 24);
        }
    }
    if (is_ctrl) tmem_dealloc(tmem, L::kTmemCols);
}

template <int D, Tile TILE>
cudaError_t launch_d(const CUtensorMap* tm, const ShortParams& p, int tiles, cudaStream_t st) {
    auto kern = tc_short_fwd_kernel<D, TILE>;
    if (cudaError_t e = configure_smem_once(reinterpret_cast<const void*>(kern), SL<D>::kDynBytes); e != cudaSuccess)
        return e;
    const int prof = profile_begin_launch(5, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)tiles);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = SL<D>::kDynBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t le = cudaLaunchKernelEx(&cfg, kern, tm[0], tm[1], tm[2], tm[3], p);
    profile_end_launch(prof, st);
    note_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
}

}  // namespace

cudaError_t launch_tc_short_fwd(const void* q, const void* k, const void* v, void* o, const RowLayout& l_qk, const RowLayout& l_v,
                                const RowLayout& l_o, bool dense, int* status, const float* m, const float* seq_len,
                                float seq_len_scalar, int B, int H, int N, int d, int dk, int dv, int causal, cudaStream_t st) {
    if (N < 1 || N > kRows || (d != 64 && d != 128) || dk > d || dv > d) return cudaErrorInvalidValue;
    ShortParams p;
    p.status = status; p.m = m; p.seq_len = seq_len; p.seq_len_scalar = seq_len_scalar;
    p.H = H; p.N = N; p.BH = B * H;
    p.slot = dense ? N : (N + 7) / 8 * 8;
    p.seqs_per_tile = kRows / p.slot;
    p.causal = causal; p.d_out = dv;
    p.head_first_mask = 0;
    p.wait_limit_kcycles = wait_limit_kcycles();
    const void* ptrs[4] = {q, k, v, o};
    const int widths[4] = {dk, dk, dv, dv};
    const RowLayout lays[4] = {l_qk, l_qk, l_v, l_o};
    CUtensorMap tm[4];
    for (int i = 0; i < 4; ++i) {
        bool hf = false;
        if (dense ? !make_rows_map(&tm[i], ptrs[i], (long long)B * H * N, widths[i], p.seqs_per_tile * N)
                  : !make_tile_map(&tm[i], ptrs[i], B, H, N, widths[i], lays[i], &hf, p.slot)) return cudaErrorInvalidValue;
        p.head_first_mask |= (hf ? 1 : 0) << i;
    }
    const int tiles = (p.BH + p.seqs_per_tile - 1) / p.seqs_per_tile;
    if (!dense) return d == 64 ? launch_d<64, PLACES>(tm, p, tiles, st) : launch_d<128, PLACES>(tm, p, tiles, st);
    if (p.seqs_per_tile > 1) return d == 64 ? launch_d<64, SEVERAL>(tm, p, tiles, st) : launch_d<128, SEVERAL>(tm, p, tiles, st);
    return d == 64 ? launch_d<64, ONE>(tm, p, tiles, st) : launch_d<128, ONE>(tm, p, tiles, st);
}

}  // namespace cott
