// A block of at most 64 tokens per (b, h) on a caller-held state (bf16 I/O, fp32 state): the
// recurrence of Eq. 8 taken a block at a time,
//     o_t   = c ( q^_t^T S_in / c  +  sum_{j <= t in the block} (q^_t . k^_j) v_j ),
//     S_out = c ( S_in / c + K^^T V ) ,
// i.e. multi-token decode steps and short segments of a chunked prefill.  The state (d_k x d_v fp32,
// 64 KB at 128 x 128) is read and written once per block whatever the number of tokens, and it is
// almost all the traffic: what bounds the kernel is how many bytes of state are in flight.
//
// So the state goes from memory through registers to memory and never touches shared or tensor
// memory.  One CTA per (b, h), one warp per strip of 32 value columns; a warp streams its strip 16
// key rows at a time, up to four steps ahead.  The products have 16 to 64 rows, too few to fill a
// tcgen05 tile, and their operand and accumulator have to be the registers the state passes through:
// warp-level m16n8k16 products, transposed so that the fp32 accumulator of the update
// S^T += V^T K^ is, rounded to bf16, the right-hand operand of the read-out Q S.  With value
// column 4 g + j of a strip in row g of slot j every lane loads and stores 16 bytes of a state
// row (8 lanes = 128 contiguous bytes).  States of any d_k, d_v are used where the caller has them.
// B H = 1024, d = 128, 16 tokens: 31 us = 4.6 TB/s (56 with the state in tensor memory, one row per
// lane on the way in and out).
#include "cott_internal.h"
#include "cott_sm100.cuh"
#include "cott_tc_common.cuh"

namespace cott {

using namespace sm100;
using namespace tc;

namespace {

constexpr long long kL2Bytes = 126LL << 20;

struct BlockParams {
    const float* state_in;   // NULL (zero state) or [BH, dk, dv], contains c
    float* state_out;        // NULL or [BH, dk, dv]
    __nv_bfloat16* o; long long o_sb, o_sh, o_sn;
    int* status;
    const float* m; const float* seq_len; float seq_len_scalar;
    int H; int N;            // N <= 64 tokens
    int dk, dv;
    int wait_limit_kcycles;
    int head_first_mask;     // bit i: in tensor map i (q, k, v) the head index comes before the token index
};

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// D (16 x 8, fp32) += A (16 x 16) B (16 x 8), bf16 operands.
__device__ __forceinline__ void mma16816(float& c0, float& c1, float& c2, float& c3, uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(c0), "+f"(c1), "+f"(c2), "+f"(c3) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// TT: tiles of 16 tokens (N <= 16 TT).
template <int TT>
struct BL {
    static constexpr int kRows = 16 * TT;
    static constexpr int kBox = kRows * 128;                   // one box: 64 columns, 128-byte swizzle
    static constexpr int kOffQ = 0, kOffK = 2 * kBox, kOffV = 4 * kBox;
    static constexpr int kPitchV = 128 + 8;                    // permuted v rows (elements)
    static constexpr int kOffVp = 6 * kBox;
    static constexpr int kOffRq = kOffVp + kRows * kPitchV * 2;    // float [kRows]: c / max(||q||, eps)
    static constexpr int kOffCtl = (kOffRq + kRows * 4 + 15) / 16 * 16;
    static constexpr int kCtlBytes = kCtlAbort + 16;
    static constexpr int kDynBytes = kOffCtl + kCtlBytes + 1024;
    // steps of 16 key rows in flight per warp: four are 128 registers a thread and 16 warps an SM (eight:
    // 38 us against 33 at B H = 1024, d = 128, 16 tokens; two: 35); with 32 tokens two (40 us) beat four (43)
    static constexpr int kAhead = TT == 1 ? 4 : 2;
};

// STREAM: more state than L2 holds passes through, so loads and stores are marked for early eviction
// (B H = 1024, d = 128: 31 us against 33); otherwise the next call finds its state in L2 (B H = 512: 14.9
// against 15.8 with the marks).
template <int TT, bool STREAM>
__global__ void __launch_bounds__(128)
block_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                 const __grid_constant__ CUtensorMap tmV, const __grid_constant__ BlockParams p) {
    using L = BL<TT>;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* gbase = smem_raw + (base - smem_u32(smem_raw));
    const uint32_t full = base + L::kOffCtl;
    volatile int* abort_flag = reinterpret_cast<volatile int*>(gbase + L::kOffCtl + kCtlAbort);
    float* rq = reinterpret_cast<float*>(gbase + L::kOffRq);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, t = lane & 3;
    const int bh = blockIdx.x, b = bh / p.H, h = bh % p.H;
    if (tid == 0) {
        mbar_init(full, 1);
        *abort_flag = 0;
        abort_flag[3] = p.wait_limit_kcycles;
        mbar_fence_init();
        fence_proxy_async();
    }
    __syncthreads();
    // The only kernel of its call; the state and the rows may come from the kernel before it.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (blockIdx.x == 0 && tid < 8) p.status[tid] = 0;
    if (tid == 0) {
        const int nk = p.dk > 64 ? 2 : 1, nv = p.dv > 64 ? 2 : 1;
        // (the bound of the wait for these tiles counts from here: a bound of zero runs out whenever the
        // other warps get to their wait)
        const long long t0 = clock64();
        mbar_expect_tx(full, (uint32_t)((2 * nk + nv) * L::kBox));
        wait_expired(full, 0u, t0, abort_flag);
        auto load = [&](uint32_t dst, const CUtensorMap* tm, int which, int n) {
            const bool hf = (p.head_first_mask >> which) & 1;
            for (int hh = 0; hh < n; ++hh) tma_load_4d(dst + hh * L::kBox, tm, full, hh * 64, hf ? h : 0, hf ? 0 : h, b);
        };
        load(base + L::kOffQ, &tmQ, 0, nk);
        load(base + L::kOffK, &tmK, 1, nk);
        load(base + L::kOffV, &tmV, 2, nv);
    }
    // This lane's 16 bytes of the state rows 16 s + {2 t, 2 t + 1, 2 t + 8, 2 t + 9}, columns col0 .. + 3.
    const int col0 = warp * 32 + 4 * g;
    const bool has_col = col0 < p.dv;
    const size_t soff = (size_t)bh * p.dk * p.dv + col0;
    const int steps = (p.dk + 15) / 16;
    auto srow = [&](int s, int i) { return s * 16 + 2 * t + (i & 1) + (i >> 1) * 8; };
    float4 S[L::kAhead][4];
    auto load_state = [&](float4 (&d)[4], int s) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = srow(s, i);
            d[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (p.state_in && has_col && r < p.dk) {
                const float4* src = reinterpret_cast<const float4*>(p.state_in + soff + (size_t)r * p.dv);
                d[i] = STREAM ? __ldcs(src) : *src;
            }
        }
    };
#pragma unroll
    for (int i = 0; i < L::kAhead; ++i)
        if (i < steps) load_state(S[i], i);

    const float s_b = p.seq_len ? p.seq_len[b] : (p.seq_len_scalar > 0.f ? p.seq_len_scalar : (float)p.N);
    const float m_h = p.m[h];
    const bool landed = wait_polling(full, 0u, abort_flag);
    const float cfac = stab_factor(m_h, s_b), ic = 1.0f / cfac;
    if (landed) {
        // ---- eight lanes per row: c / ||q||, k^ in place, v with its columns permuted (column
        // 32 w + 4 g + j at 32 w + 8 j + g), 16 bytes at a time
        const int nw = blockDim.x >> 5;
#pragma unroll 1
        for (int r0 = warp * 4; r0 < L::kRows; r0 += nw * 4) {
            const int r = r0 + (lane >> 3), ch = lane & 7;
            float sq = 0.f, sk = 0.f;
            uint4 wk[2];
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                wk[hh] = make_uint4(0u, 0u, 0u, 0u);
                if (hh * 64 >= p.dk) continue;
                const uint32_t off = hh * (uint32_t)L::kBox + swz(r, ch);
                const uint4 wq = *reinterpret_cast<const uint4*>(gbase + L::kOffQ + off);
                wk[hh] = *reinterpret_cast<const uint4*>(gbase + L::kOffK + off);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float2 fq = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&wq)[i]);
                    const float2 fk = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(&wk[hh])[i]);
                    sq = fmaf(fq.x, fq.x, fmaf(fq.y, fq.y, sq));
                    sk = fmaf(fk.x, fk.x, fmaf(fk.y, fk.y, sk));
                }
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                sq += __shfl_xor_sync(0xffffffffu, sq, o);
                sk += __shfl_xor_sync(0xffffffffu, sk, o);
            }
            const float rk = 1.0f / fmaxf(sqrtf(sk), kEps);
            if (ch == 0) rq[r] = cfac / fmaxf(sqrtf(sq), kEps);
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                if (hh * 64 < p.dk) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        __nv_bfloat162& e = reinterpret_cast<__nv_bfloat162*>(&wk[hh])[i];
                        const float2 f = __bfloat1622float2(e);
                        e = __floats2bfloat162_rn(f.x * rk, f.y * rk);
                    }
                    *reinterpret_cast<uint4*>(gbase + L::kOffK + hh * L::kBox + swz(r, ch)) = wk[hh];
                }
                if (hh * 64 < p.dv) {
                    const uint4 wv = *reinterpret_cast<const uint4*>(gbase + L::kOffV + hh * L::kBox + swz(r, ch));
                    uint8_t* dst = gbase + L::kOffVp + (r * L::kPitchV + hh * 64 + (ch >> 2) * 32 + (ch & 3) * 2) * 2;
                    const uint32_t x[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j)          // columns j and j + 4 of the eight
                        *reinterpret_cast<uint32_t*>(dst + j * 16) = __byte_perm(x[j >> 1], x[2 + (j >> 1)], (j & 1) ? 0x7632 : 0x5410);
                }
            }
        }
    }
    __syncthreads();
    if (*abort_flag == 0) {
        // ldmatrix addresses: lane l points at row l % 8 of matrix l / 8.
        const int lr = lane & 7, lm = lane >> 3;
        // A operand of 16 tokens x 16 keys: matrices (tokens 0-7, 8-15) x keys 0-7, then keys 8-15
        auto row_key = [&](int off, int tile, int s) {
            const int r = tile * 16 + lr + (lm & 1) * 8, ch = 2 * s + (lm >> 1);
            return base + off + (ch >> 3) * (uint32_t)L::kBox + swz(r, ch & 7);
        };
        // B operand (keys x tokens): matrices (keys 0-7, 8-15) x tokens 0-7, then tokens 8-15
        auto key_row = [&](int off, int tile, int s) {
            const int r = tile * 16 + lr + (lm >> 1) * 8, ch = 2 * s + (lm & 1);
            return base + off + (ch >> 3) * (uint32_t)L::kBox + swz(r, ch & 7);
        };
        // V^T of this warp's strip: av[kt][mt] = A operand, value slots 2 mt, 2 mt + 1 x 16 tokens
        uint32_t av[TT][2][4];
#pragma unroll
        for (int kt = 0; kt < TT; ++kt)
#pragma unroll
            for (int mt = 0; mt < 2; ++mt) {
                const int r = kt * 16 + lr + (lm >> 1) * 8, col = warp * 32 + (2 * mt + (lm & 1)) * 8;
                ldsm4t(av[kt][mt], base + L::kOffVp + (r * L::kPitchV + col) * 2);
            }
        float O[TT][4][4];
#pragma unroll
        for (int i = 0; i < TT; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
                for (int c = 0; c < 4; ++c) O[i][j][c] = 0.f;
        // ---- within the block: masked scores (diagonal kept, Eq. 6) times v
#pragma unroll
        for (int tt = 0; tt < TT; ++tt) {
            float P[TT][2][4];
#pragma unroll
            for (int kt = 0; kt <= tt; ++kt)
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int c = 0; c < 4; ++c) P[kt][n][c] = 0.f;
#pragma unroll 1
            for (int s = 0; s < steps; ++s) {
                uint32_t a[4];
                ldsm4(a, row_key(L::kOffQ, tt, s));
#pragma unroll
                for (int kt = 0; kt <= tt; ++kt) {
                    uint32_t bk[4];
                    ldsm4(bk, key_row(L::kOffK, kt, s));
#pragma unroll
                    for (int n = 0; n < 2; ++n)
                        mma16816(P[kt][n][0], P[kt][n][1], P[kt][n][2], P[kt][n][3], a[0], a[1], a[2], a[3], bk[2 * n], bk[2 * n + 1]);
                }
            }
#pragma unroll
            for (int kt = 0; kt <= tt; ++kt) {
                if (kt == tt) {
#pragma unroll
                    for (int n = 0; n < 2; ++n)
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (8 * n + 2 * t + (c & 1) > g + (c >> 1) * 8) P[kt][n][c] = 0.f;
                }
                const uint32_t a0 = pack_bf16(P[kt][0][0], P[kt][0][1]), a1 = pack_bf16(P[kt][0][2], P[kt][0][3]);
                const uint32_t a2 = pack_bf16(P[kt][1][0], P[kt][1][1]), a3 = pack_bf16(P[kt][1][2], P[kt][1][3]);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    mma16816(O[tt][j][0], O[tt][j][1], O[tt][j][2], O[tt][j][3], a0, a1, a2, a3, av[kt][j >> 1][j & 1], av[kt][j >> 1][2 + (j & 1)]);
            }
        }
        // ---- the state, 16 key rows at a time: read out, then updated
#pragma unroll 1
        for (int s0 = 0; s0 < steps; s0 += L::kAhead) {
#pragma unroll
            for (int i = 0; i < L::kAhead; ++i) {
                const int s = s0 + i;
                if (s >= steps) break;
                float4 (&Sx)[4] = S[i];
                float* e[4] = {&Sx[0].x, &Sx[1].x, &Sx[2].x, &Sx[3].x};
#pragma unroll
                for (int k = 0; k < 4; ++k) { Sx[k].x *= ic; Sx[k].y *= ic; Sx[k].z *= ic; Sx[k].w *= ic; }
                uint32_t b0[4], b1[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) { b0[j] = pack_bf16(e[0][j], e[1][j]); b1[j] = pack_bf16(e[2][j], e[3][j]); }
#pragma unroll
                for (int tt = 0; tt < TT; ++tt) {
                    uint32_t a[4];
                    ldsm4(a, row_key(L::kOffQ, tt, s));
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        mma16816(O[tt][j][0], O[tt][j][1], O[tt][j][2], O[tt][j][3], a[0], a[1], a[2], a[3], b0[j], b1[j]);
                }
                if (p.state_out) {
#pragma unroll
                    for (int kt = 0; kt < TT; ++kt) {
                        uint32_t bk[4];
                        ldsm4t(bk, row_key(L::kOffK, kt, s));
#pragma unroll
                        for (int n = 0; n < 2; ++n)
#pragma unroll
                            for (int mt = 0; mt < 2; ++mt)
                                mma16816(e[2 * n][2 * mt], e[2 * n + 1][2 * mt], e[2 * n][2 * mt + 1], e[2 * n + 1][2 * mt + 1],
                                         av[kt][mt][0], av[kt][mt][1], av[kt][mt][2], av[kt][mt][3], bk[2 * n], bk[2 * n + 1]);
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int r = srow(s, k);
                        if (has_col && r < p.dk) {
                            float4* dst = reinterpret_cast<float4*>(p.state_out + soff + (size_t)r * p.dv);
                            const float4 w = make_float4(Sx[k].x * cfac, Sx[k].y * cfac, Sx[k].z * cfac, Sx[k].w * cfac);
                            if (STREAM) __stcs(dst, w); else *dst = w;
                        }
                    }
                }
                if (s + L::kAhead < steps) load_state(Sx, s + L::kAhead);
            }
        }
        // ---- output rows: lane (g, t) has columns 8 t .. + 7 of the strip for tokens g, g + 8 of a tile
        const int oc = warp * 32 + 8 * t;
#pragma unroll
        for (int tt = 0; tt < TT; ++tt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int n = tt * 16 + hf * 8 + g;
                if (n < p.N && oc < p.dv) {
                    const float r = rq[n];
                    uint4 w;
                    w.x = pack_bf16(O[tt][0][2 * hf] * r, O[tt][1][2 * hf] * r);
                    w.y = pack_bf16(O[tt][2][2 * hf] * r, O[tt][3][2 * hf] * r);
                    w.z = pack_bf16(O[tt][0][2 * hf + 1] * r, O[tt][1][2 * hf + 1] * r);
                    w.w = pack_bf16(O[tt][2][2 * hf + 1] * r, O[tt][3][2 * hf + 1] * r);
                    *reinterpret_cast<uint4*>(p.o + (long long)b * p.o_sb + (long long)h * p.o_sh + (long long)n * p.o_sn + oc) = w;
                }
            }
    } else {
        // The wait for the tiles gave up: give the copies time to land, then report.
        for (int i = 0; i < 100; ++i) __nanosleep(1000);
        if (tid == 0 && atomicCAS(p.status, 0, 1) == 0) {
            p.status[1] = *abort_flag;
            p.status[2] = (int)blockIdx.x | (7 << 24);
        }
    }
}

template <int TT>
cudaError_t launch_t(const CUtensorMap* tm, const BlockParams& p, int BH, cudaStream_t st) {
    const bool stream = ((p.state_in ? 4LL : 0LL) + (p.state_out ? 4LL : 0LL)) * BH * p.dk * p.dv > kL2Bytes;
    auto kern = stream ? block_fwd_kernel<TT, true> : block_fwd_kernel<TT, false>;
    if (cudaError_t e = configure_smem_once(reinterpret_cast<const void*>(kern), BL<TT>::kDynBytes); e != cudaSuccess)
        return e;
    const int prof = profile_begin_launch(6, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)BH);
    // (two warps at least: a second one without value columns shares the row passes; d_k = d_v = 32, 33 tokens,
    // 12 (b, h): 11 us with one)
    cfg.blockDim = dim3(32u * (unsigned)(p.dv > 64 ? (p.dv + 31) / 32 : 2));
    cfg.dynamicSmemBytes = BL<TT>::kDynBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t le = cudaLaunchKernelEx(&cfg, kern, tm[0], tm[1], tm[2], p);
    profile_end_launch(prof, st);
    note_launch();
    return le != cudaSuccess ? le : cudaGetLastError();
}

}  // namespace

cudaError_t launch_block_fwd(const void* q, const void* k, const void* v, void* o, const RowLayout& l_qk,
                                const RowLayout& l_v, const RowLayout& l_o, const float* state_in, float* state_out,
                                int* status, const float* m, const float* seq_len, float seq_len_scalar, int B, int H,
                                int N, int dk, int dv, cudaStream_t st) {
    if (N < 1 || N > 64 || dk < 8 || dv < 8 || dk > 128 || dv > 128) return cudaErrorInvalidValue;
    BlockParams p;
    p.state_in = state_in; p.state_out = state_out; p.status = status;
    p.m = m; p.seq_len = seq_len; p.seq_len_scalar = seq_len_scalar;
    p.H = H; p.N = N; p.dk = dk; p.dv = dv;
    const RowLayout lo = resolve_layout(l_o, H, N, dv);
    p.o = static_cast<__nv_bfloat16*>(o); p.o_sb = lo.sb; p.o_sh = lo.sh; p.o_sn = lo.sn;
    p.wait_limit_kcycles = wait_limit_kcycles();
    const int tiles = N <= 16 ? 1 : (N <= 32 ? 2 : 4);
    const void* ptrs[3] = {q, k, v};
    const RowLayout lays[3] = {l_qk, l_qk, l_v};
    const int widths[3] = {dk, dk, dv};
    CUtensorMap tm[3];
    p.head_first_mask = 0;
    for (int i = 0; i < 3; ++i) {
        bool hf = false;
        if (!make_tile_map(&tm[i], ptrs[i], B, H, N, widths[i], lays[i], &hf, 16 * tiles)) return cudaErrorInvalidValue;
        p.head_first_mask |= (hf ? 1 : 0) << i;
    }
    switch (tiles) {
        case 1: return launch_t<1>(tm, p, B * H, st);
        case 2: return launch_t<2>(tm, p, B * H, st);
        default: return launch_t<4>(tm, p, B * H, st);
    }
}

}  // namespace cott
