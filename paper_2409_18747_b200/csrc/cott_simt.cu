// fp32 SIMT kernels: the running-sum walk (Eq. 7 / Eq. 8), the scan over per-group partial
// states, the dm reduction and the recurrent decode step.  These serve fp32 I/O (tensor
// cores in TF32 cannot meet the fp32 tolerance) and every shape the tensor-core kernels do
// not cover.
#include <initializer_list>
#include "cott_internal.h"

namespace cott {

namespace {

constexpr int kThreads = 256;
constexpr int kChunk = kSimtChunk;

template <typename T> __device__ __forceinline__ float4 load4(const T* p);
template <> __device__ __forceinline__ float4 load4<float>(const float* p) {
    return *reinterpret_cast<const float4*>(p);
}
template <> __device__ __forceinline__ float4 load4<__nv_bfloat16>(const __nv_bfloat16* p) {
    uint2 v = *reinterpret_cast<const uint2*>(p);
    const float2 lo = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&v.x));
    const float2 hi = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&v.y));
    return make_float4(lo.x, lo.y, hi.x, hi.y);
}
template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) {
    return __bfloat162float(v);
}
template <typename T> __device__ __forceinline__ T from_f32(float v);
template <> __device__ __forceinline__ float from_f32<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float v) {
    return __float2bfloat16_rn(v);
}
template <typename T> __device__ __forceinline__ void store4(T* p, float4 f);
template <> __device__ __forceinline__ void store4<float>(float* p, float4 f) {
    *reinterpret_cast<float4*>(p) = f;
}
template <> __device__ __forceinline__ void store4<__nv_bfloat16>(__nv_bfloat16* p, float4 f) {
    __nv_bfloat162 lo = __floats2bfloat162_rn(f.x, f.y);
    __nv_bfloat162 hi = __floats2bfloat162_rn(f.z, f.w);
    uint2 v;
    v.x = *reinterpret_cast<uint32_t*>(&lo);
    v.y = *reinterpret_cast<uint32_t*>(&hi);
    *reinterpret_cast<uint2*>(p) = v;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float dot4(float4 a, float4 b) {
    return fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}
__device__ __forceinline__ void axpy4(float4& y, float a, float4 x) {
    const float2 a2 = make_float2(a, a);
    const float2 lo = __ffma2_rn(a2, make_float2(x.x, x.y), make_float2(y.x, y.y));
    const float2 hi = __ffma2_rn(a2, make_float2(x.z, x.w), make_float2(y.z, y.w));
    y = make_float4(lo.x, lo.y, hi.x, hi.y);
}

// y += a.x x0 + a.y x1 + a.z x2 + a.w x3, the four products summed among themselves first: a chain of D
// multiply-adds onto one accumulator rounds at the size of the whole sum D times, this D / 4 times.
__device__ __forceinline__ void axpy4x4(float4& y, float4 a, float4 x0, float4 x1, float4 x2, float4 x3) {
    float2 lo = __fmul2_rn(make_float2(a.x, a.x), make_float2(x0.x, x0.y)), hi = __fmul2_rn(make_float2(a.x, a.x), make_float2(x0.z, x0.w));
    lo = __ffma2_rn(make_float2(a.y, a.y), make_float2(x1.x, x1.y), lo); hi = __ffma2_rn(make_float2(a.y, a.y), make_float2(x1.z, x1.w), hi);
    lo = __ffma2_rn(make_float2(a.z, a.z), make_float2(x2.x, x2.y), lo); hi = __ffma2_rn(make_float2(a.z, a.z), make_float2(x2.z, x2.w), hi);
    lo = __ffma2_rn(make_float2(a.w, a.w), make_float2(x3.x, x3.y), lo); hi = __ffma2_rn(make_float2(a.w, a.w), make_float2(x3.z, x3.w), hi);
    lo = __fadd2_rn(make_float2(y.x, y.y), lo); hi = __fadd2_rn(make_float2(y.z, y.w), hi);
    y = make_float4(lo.x, lo.y, hi.x, hi.y);
}

// Shared memory of the walk: three chunk tiles (rows padded by four words: threads that read 16
// consecutive rows at the same column then hit different banks), the chunk's masked scores and
// the state.
template <int D> struct WalkSmem {
    static constexpr int kRow = D + 4, kScoreRow = kChunk + 4;
    static constexpr int kX = 0, kA = kX + kChunk * kRow, kB = kA + kChunk * kRow;
    static constexpr int kP = kB + kChunk * kRow, kS = kP + kChunk * kScoreRow;
    static constexpr int kBytes = (kS + D * D) * 4;
};

// One pass of the running-sum walk (WalkArgs) over one sequence group, 32 tokens at a time:
//     P = X A^T, masked to the pairs the running sum holds (Eq. 6) ;  Out = P Bv + X S ;  S += A^T Bv
// in fp32 multiply-adds (packed in pairs) throughout.  What bounds it is the multiply-add rate (per token 2 * 32 * d
// for the scores side, 2 d^2 for the state side), and for the small problems this path serves the
// chain of launches and the fill of the SMs; the token-by-token recurrence it replaces was one
// serial chain (0.35 us a token) on the same SMs.  32 tokens a chunk: a 64-token chunk does 1.3
// times the multiply-adds at d = 64 and halves the number of CTAs a short sequence gives.
// Measured, forward and backward at B=2, H=8, N=509, d=64: 303 us and 13 launches with the
// recurrence, 70 us and 4 launches (state pass and walk each way) here.
// Thread (ty, tx) owns columns 4 tx .. + 3 everywhere: rows ty, ty + TY, .. of the chunk (it loads,
// normalises and produces them; the TX threads of a row sit in one warp, so row sums are
// shuffles) and rows SR ty .. + SR - 1 of the state, which stays in its registers and is copied
// to shared memory once per chunk.  The next chunk's rows are loaded while this one is computed.
// blockIdx.y picks one of up to three streams (the three gradients of a backward call).
// Threads of a CTA: few, so that each has a tile of four rows (d = 64; 32: two) and shared memory feeds
// twice as many multiply-adds per load; three or four CTAs share an SM.  (Backward at B=2, H=8, N=509, d = 64:
// 43 us against 56 with 256 threads, B=32, H=12, N=100, d = 32: 57 against 90; 168 registers, 128 spill.)
template <int D> struct WalkThreads { static constexpr int n = D == 128 ? 256 : 128, ctas = D == 128 ? 1 : (D == 64 ? 3 : 4); };

template <int D, typename T>
__global__ void __launch_bounds__(WalkThreads<D>::n, WalkThreads<D>::ctas) walk_kernel(const __grid_constant__ WalkBatch batch) {
    using M = WalkSmem<D>;
    constexpr int NT = WalkThreads<D>::n;
    constexpr int TX = D / 4, TY = NT / TX;
    constexpr int RPT = kChunk / TY;      // chunk rows per thread
    constexpr int SR = D / TY;            // state rows per thread
    extern __shared__ __align__(16) float sm[];
    __shared__ float dm_red[NT / 32];
    __shared__ int last_flag;
    const WalkArgs& w = batch.w[blockIdx.y];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int tx = tid % TX, ty = tid / TX;
    const int g = blockIdx.x % w.n_groups;
    const int bh = blockIdx.x / w.n_groups;
    const int b = bh / w.H, h = bh % w.H;
    // (the walk of a call may start while its state pass drains)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!w.write_out) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (batch.clear_status && blockIdx.x == 0 && blockIdx.y == 0 && tid < 8) batch.status[tid] = 0;
    // (a packed batch: the rows of sequence b, one group)
    const int lo = w.cu_seqlens ? w.cu_seqlens[b] : g * w.group;
    const int hi = w.cu_seqlens ? w.cu_seqlens[b + 1] : min(w.N, lo + w.group);
    // (the launcher has resolved the layouts: strides are never all zero here)
    auto slice = [&](const RowLayout& l) { return (w.cu_seqlens ? (size_t)0 : (size_t)b * l.sb) + (size_t)h * l.sh; };
    const bool write_out = w.write_out, update = w.update;
    const T* X = write_out ? static_cast<const T*>(w.x) + slice(w.lx) : nullptr;
    const T* A = static_cast<const T*>(w.a) + slice(w.la);
    const T* Bv = static_cast<const T*>(w.bv) + slice(w.lbv);
    const T* P = w.proj ? static_cast<const T*>(w.proj) + slice(w.lproj) : nullptr;
    T* O = write_out ? static_cast<T*>(w.out) + slice(w.lout) : nullptr;

    const float s_b = w.seq_len ? w.seq_len[b]
                                : (w.seq_len_scalar > 0.f ? w.seq_len_scalar
                                                          : (float)(w.cu_seqlens ? max(hi - lo, 1) : w.N));
    const float c = stab_factor(w.m[h], s_b);

    const int n_chunks = (hi - lo + kChunk - 1) / kChunk;
    auto chunk_row = [&](int it) { return lo + (w.reverse ? n_chunks - 1 - it : it) * kChunk; };
    const float4 zero4 = make_float4(0.f, 0.f, 0.f, 0.f);
    auto load_rows = [&](float4 (&r)[RPT], const T* src, long long sn, int t0) {
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            const int t = t0 + ty + TY * u;
            r[u] = t < hi ? load4<T>(src + (long long)t * sn + tx * 4) : zero4;
        }
    };
    float4 rx[RPT], ra[RPT], rb[RPT];
    auto load_chunk = [&](int t0) {
        if (write_out) load_rows(rx, X, w.lx.sn, t0);
        if (update) { load_rows(ra, A, w.la.sn, t0); load_rows(rb, Bv, w.lbv.sn, t0); }
    };
    if (n_chunks > 0) load_chunk(chunk_row(0));

    // The state before this group's first chunk: the sum of the partial states before it in the
    // walk's direction of time (all of them when the mask is all ones), or what a scan launch has
    // left in the group's own place.
    float4 S[SR];
#pragma unroll
    for (int r = 0; r < SR; ++r) S[r] = zero4;
    bool have_state = false;
    auto add_state = [&](const float* src, bool transposed) {
        have_state = true;
        if (!transposed) {
#pragma unroll
            for (int r = 0; r < SR; ++r) {
                const float4 v = *reinterpret_cast<const float4*>(src + (size_t)(ty * SR + r) * D + tx * 4);
                S[r].x += v.x; S[r].y += v.y; S[r].z += v.z; S[r].w += v.w;
            }
        } else {
            const float* s0 = src + (size_t)(tx * 4) * D + ty * SR;
            if constexpr (SR >= 4) {
#pragma unroll
                for (int r = 0; r < SR; r += 4) {
                    const float4 v0 = *reinterpret_cast<const float4*>(s0 + r), v1 = *reinterpret_cast<const float4*>(s0 + D + r);
                    const float4 v2 = *reinterpret_cast<const float4*>(s0 + 2 * D + r), v3 = *reinterpret_cast<const float4*>(s0 + 3 * D + r);
                    S[r].x += v0.x; S[r].y += v1.x; S[r].z += v2.x; S[r].w += v3.x;
                    S[r + 1].x += v0.y; S[r + 1].y += v1.y; S[r + 1].z += v2.y; S[r + 1].w += v3.y;
                    S[r + 2].x += v0.z; S[r + 2].y += v1.z; S[r + 2].z += v2.z; S[r + 2].w += v3.z;
                    S[r + 3].x += v0.w; S[r + 3].y += v1.w; S[r + 3].z += v2.w; S[r + 3].w += v3.w;
                }
            } else {
#pragma unroll
                for (int r = 0; r < SR; ++r) {
                    S[r].x += s0[r]; S[r].y += s0[D + r]; S[r].z += s0[2 * D + r]; S[r].w += s0[3 * D + r];
                }
            }
        }
    };
    // A caller's state is added to the sum of the partial states, not they to it one by one; a single group
    // keeps it apart altogether, and the two meet where the state is read.
    const float* base = (w.init_extra && !w.init) ? w.init_extra + (size_t)bh * D * D : nullptr;
    if (w.init) {
        const float* part = w.init + (size_t)bh * w.n_groups * D * D;
        if (w.init_sum) {
            const int g0 = (w.reverse && update) ? g + 1 : 0, g1 = (w.reverse || !update) ? w.n_groups : g;
            for (int gg = g0; gg < g1; ++gg) add_state(part + (size_t)gg * D * D, w.init_transposed);
        } else {
            add_state(part + (size_t)g * D * D, w.init_transposed);
        }
        if (w.init_extra) add_state(w.init_extra + (size_t)bh * D * D, false);
    }
    if (base) have_state = true;
    // The total of several groups is what comes before the last one plus its partial state: the former goes
    // to its place now, the latter is added at the end (this walk's rows accumulate onto the whole sum).
    // Where a scan launch has left the sum of the partial states there, the caller's state is added.
    const bool total = w.init && w.final_state && update && g == (w.reverse ? 0 : w.n_groups - 1);
    auto final_row = [&](int r) {
        return reinterpret_cast<float4*>(w.final_state + (w.final_grouped ? ((size_t)bh * w.n_groups + g) : (size_t)bh) * D * D +
                                         (size_t)(ty * SR + r) * D + tx * 4);
    };
    if (total && w.init_sum) {
#pragma unroll
        for (int r = 0; r < SR; ++r) *final_row(r) = S[r];
    }
    auto add = [](float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); };
    auto state_row = [&](int r) {
        return base ? add(*reinterpret_cast<const float4*>(base + (size_t)(ty * SR + r) * D + tx * 4), S[r]) : S[r];
    };
    auto put_state = [&]() {
        constexpr int RB = SR < 4 ? SR : 4;
#pragma unroll
        for (int r0 = 0; r0 < SR; r0 += RB) {
            float4 v[RB];
#pragma unroll
            for (int r = 0; r < RB; ++r) v[r] = state_row(r0 + r);
#pragma unroll
            for (int r = 0; r < RB; ++r) *reinterpret_cast<float4*>(sm + M::kS + (ty * SR + r0 + r) * D + tx * 4) = v[r];
        }
    };
    if (write_out && have_state) put_state();

    // Row treatment of a loaded row piece: scale by c, or by 1 / max(||row||, eps).
    auto treat = [&](float4& v, int mode) {
        float s = 1.f;
        if (mode == ROW_SCALE) s = c;
        if (mode == ROW_NORM) {
            float ss = dot4(v, v);
#pragma unroll
            for (int o = TX / 2; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
            s = 1.0f / fmaxf(sqrtf(ss), kEps);
        }
        if (mode != ROW_RAW) { v.x *= s; v.y *= s; v.z *= s; v.w *= s; }
    };
    auto put_rows = [&](float4 (&r)[RPT], int off, int mode) {
        bool finite = true;
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
            treat(r[u], mode);
            *reinterpret_cast<float4*>(sm + off + (ty + TY * u) * M::kRow + tx * 4) = r[u];
            finite = finite && dot4(r[u], zero4) == 0.f;      // (infinity and NaN times zero are NaN)
        }
        return finite;
    };

    // (the state after the last chunk is read by nobody unless it is a partial state or a single group's total)
    const bool keep_state = w.final_state && (w.final_grouped || w.n_groups == 1);
    float dm_acc = 0.f;
    for (int it = 0; it < n_chunks; ++it) {
        const int t0 = chunk_row(it);
        const int n_rows = min(kChunk, hi - t0);     // (rows behind it are zero: the loops over tokens leave them out)
        if (write_out) put_rows(rx, M::kX, w.mode_x);
        bool finite = true;
        if (update) { put_rows(ra, M::kA, w.mode_a); finite = put_rows(rb, M::kB, w.mode_b); }
        // A masked score is zero, and zero times an infinity or a NaN is not: with one in a Bv row of this
        // chunk the masked pairs are left out of P Bv, not multiplied by zero.
        const bool skip_masked = __syncthreads_or(!finite);
        float4 rp[RPT];
        if (w.epilogue != EPI_PLAIN) load_rows(rp, P, w.lproj.sn, t0);
        if (it + 1 < n_chunks) load_chunk(chunk_row(it + 1));

        float4 out[RPT];
        if (write_out) {
            if (update) {
                // scores: SU rows pi + PY u against keys pj, pj + 16
                constexpr int PY = NT / 16, SU = kChunk / PY;
                const int pi = tid >> 4, pj = tid & 15;
                float2 acc[SU][2];
#pragma unroll
                for (int u = 0; u < SU; ++u) { acc[u][0] = make_float2(0.f, 0.f); acc[u][1] = acc[u][0]; }
#pragma unroll 2
                for (int k = 0; k < D; k += 8) {       // (eight products are summed among themselves first, as in axpy4x4)
                    const float4 a00 = *reinterpret_cast<const float4*>(sm + M::kA + pj * M::kRow + k);
                    const float4 a01 = *reinterpret_cast<const float4*>(sm + M::kA + pj * M::kRow + k + 4);
                    const float4 a10 = *reinterpret_cast<const float4*>(sm + M::kA + (pj + 16) * M::kRow + k);
                    const float4 a11 = *reinterpret_cast<const float4*>(sm + M::kA + (pj + 16) * M::kRow + k + 4);
                    auto part = [](float4 x0, float4 x1, float4 y0, float4 y1) {
                        float2 t = __fmul2_rn(make_float2(x0.x, x0.y), make_float2(y0.x, y0.y));
                        t = __ffma2_rn(make_float2(x0.z, x0.w), make_float2(y0.z, y0.w), t);
                        t = __ffma2_rn(make_float2(x1.x, x1.y), make_float2(y1.x, y1.y), t);
                        return __ffma2_rn(make_float2(x1.z, x1.w), make_float2(y1.z, y1.w), t);
                    };
#pragma unroll
                    for (int u = 0; u < SU; ++u) {
                        const float4 x0 = *reinterpret_cast<const float4*>(sm + M::kX + (pi + PY * u) * M::kRow + k);
                        const float4 x1 = *reinterpret_cast<const float4*>(sm + M::kX + (pi + PY * u) * M::kRow + k + 4);
                        acc[u][0] = __fadd2_rn(acc[u][0], part(x0, x1, a00, a01));
                        acc[u][1] = __fadd2_rn(acc[u][1], part(x0, x1, a10, a11));
                    }
                }
#pragma unroll
                for (int u = 0; u < SU; ++u)
#pragma unroll
                    for (int v = 0; v < 2; ++v) {
                        const int i = pi + PY * u, j = pj + 16 * v;
                        const bool keep = w.reverse ? j >= i : j <= i;
                        sm[M::kP + i * M::kScoreRow + j] = keep ? acc[u][v].x + acc[u][v].y : 0.f;
                    }
            }
#pragma unroll
            for (int u = 0; u < RPT; ++u) out[u] = zero4;
            if (have_state) {
#pragma unroll 4
                for (int k = 0; k < D; k += 4) {
                    float4 x[RPT];
#pragma unroll
                    for (int u = 0; u < RPT; ++u) x[u] = *reinterpret_cast<const float4*>(sm + M::kX + (ty + TY * u) * M::kRow + k);
                    const float* s0 = sm + M::kS + k * D + tx * 4;
                    const float4 v0 = *reinterpret_cast<const float4*>(s0), v1 = *reinterpret_cast<const float4*>(s0 + D);
                    const float4 v2 = *reinterpret_cast<const float4*>(s0 + 2 * D), v3 = *reinterpret_cast<const float4*>(s0 + 3 * D);
#pragma unroll
                    for (int u = 0; u < RPT; ++u) axpy4x4(out[u], x[u], v0, v1, v2, v3);
                }
            }
            if (update) {
                __syncthreads();
                if (skip_masked) {
#pragma unroll 1
                    for (int k = 0; k < kChunk; ++k) {
                        const float4 v = *reinterpret_cast<const float4*>(sm + M::kB + k * M::kRow + tx * 4);
#pragma unroll
                        for (int u = 0; u < RPT; ++u) {
                            const int i = ty + TY * u;
                            if (w.reverse ? k >= i : k <= i) axpy4(out[u], sm[M::kP + i * M::kScoreRow + k], v);
                        }
                    }
                } else
#pragma unroll 2
                for (int k = 0; k < n_rows; k += 4) {
                    float4 x[RPT];
#pragma unroll
                    for (int u = 0; u < RPT; ++u)
                        x[u] = *reinterpret_cast<const float4*>(sm + M::kP + (ty + TY * u) * M::kScoreRow + k);
                    const float* b0 = sm + M::kB + k * M::kRow + tx * 4;
                    const float4 v0 = *reinterpret_cast<const float4*>(b0), v1 = *reinterpret_cast<const float4*>(b0 + M::kRow);
                    const float4 v2 = *reinterpret_cast<const float4*>(b0 + 2 * M::kRow), v3 = *reinterpret_cast<const float4*>(b0 + 3 * M::kRow);
#pragma unroll
                    for (int u = 0; u < RPT; ++u) axpy4x4(out[u], x[u], v0, v1, v2, v3);
                }
            }
#pragma unroll
            for (int u = 0; u < RPT; ++u) {
                const int t = t0 + ty + TY * u;
                if (w.epilogue == EPI_PROJ) {
                    // dx = (dx^ - x^ <x^, dx^>) / ||x||, or dx^ / eps on the clamped branch
                    float ss = dot4(rp[u], rp[u]), dp = dot4(rp[u], out[u]);
#pragma unroll
                    for (int o = TX / 2; o > 0; o >>= 1) {
                        ss += __shfl_xor_sync(0xffffffffu, ss, o);
                        dp += __shfl_xor_sync(0xffffffffu, dp, o);
                    }
                    const float nrm = sqrtf(ss);
                    const float rinv = 1.0f / fmaxf(nrm, kEps);
                    const float coef = nrm > kEps ? dp * rinv * rinv : 0.f;  // <x^,dx^> * rinv
                    out[u].x = (out[u].x - rp[u].x * coef) * rinv; out[u].y = (out[u].y - rp[u].y * coef) * rinv;
                    out[u].z = (out[u].z - rp[u].z * coef) * rinv; out[u].w = (out[u].w - rp[u].w * coef) * rinv;
                } else if (w.epilogue == EPI_DV) {
                    dm_acc += dot4(rp[u], out[u]);  // (rows past the end are zero)
                    out[u].x *= c; out[u].y *= c; out[u].z *= c; out[u].w *= c;
                }
                if (t < hi) store4<T>(O + (long long)t * w.lout.sn + tx * 4, out[u]);
            }
        }
        if (update && (it + 1 < n_chunks || keep_state)) {
            have_state = true;
#pragma unroll 4
            for (int k = 0; k < n_rows; ++k) {
                const float4 v = *reinterpret_cast<const float4*>(sm + M::kB + k * M::kRow + tx * 4);
                const float* ap = sm + M::kA + k * M::kRow + ty * SR;
                if constexpr (SR >= 4) {
#pragma unroll
                    for (int r = 0; r < SR; r += 4) {
                        const float4 a = *reinterpret_cast<const float4*>(ap + r);
                        axpy4(S[r], a.x, v); axpy4(S[r + 1], a.y, v); axpy4(S[r + 2], a.z, v); axpy4(S[r + 3], a.w, v);
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < SR; ++r) axpy4(S[r], ap[r], v);
                }
            }
            // (every read of the previous copy came before this chunk's second barrier)
            if (write_out && it + 1 < n_chunks) put_state();
        }
        __syncthreads();
    }

    // The group's partial state, or the total: of a single group, or of all where the mask is all ones.
    if (total) {
        const float* rest = (w.init_sum ? w.init + ((size_t)bh * w.n_groups + g) * D * D : w.init_extra + (size_t)bh * D * D) +
                            (size_t)ty * SR * D + tx * 4;
        // (all loads before the first store: the compiler has to keep their order)
#pragma unroll
        for (int r = 0; r < SR; ++r) S[r] = add(*final_row(r), *reinterpret_cast<const float4*>(rest + r * D));
#pragma unroll
        for (int r = 0; r < SR; ++r) *final_row(r) = S[r];
    } else if (keep_state || (w.final_state && !update && g == 0)) {
#pragma unroll
        for (int r = 0; r < SR; ++r) S[r] = state_row(r);
#pragma unroll
        for (int r = 0; r < SR; ++r) *final_row(r) = S[r];
    }
    if (w.dm_partial) {
        dm_acc = warp_sum(dm_acc);
        if (lane == 0) dm_red[warp] = dm_acc;
        __syncthreads();
        if (tid == 0) {
            float t = 0.f;
            for (int i = 0; i < NT / 32; ++i) t += dm_red[i];
            w.dm_partial[(size_t)bh * w.n_groups + g] = t;
            __threadfence();
            last_flag = atomicAdd(&batch.status[4], 1) == (int)gridDim.x - 1;
        }
        __syncthreads();
        if (last_flag) {
            // dm_h = sum_b dc/dm * <dV', V>_{b,h},  dc/dm = -ln(s_b) sigma(m_h)(1-sigma(m_h)) c_{b,h}.
            // Fixed summation order (deterministic); one warp per head.
            __threadfence();
            const int n_b = (int)gridDim.x / (w.n_groups * w.H), per = n_b * w.n_groups;
            for (int hh = warp; hh < w.H; hh += NT / 32) {
                const float sg = 1.0f / (1.0f + expf(-w.m[hh]));
                float sum = 0.f;
                for (int i = lane; i < per; i += 32) {
                    const int bb = i / w.n_groups, gg = i - bb * w.n_groups;
                    const float sb2 = w.seq_len ? w.seq_len[bb]
                                                : (w.seq_len_scalar > 0.f ? w.seq_len_scalar
                                                   : (float)(w.cu_seqlens ? max(w.cu_seqlens[bb + 1] - w.cu_seqlens[bb], 1) : w.N));
                    const float ls = logf(sb2);
                    sum += __ldcg(&w.dm_partial[((size_t)bb * w.H + hh) * w.n_groups + gg]) * (-ls * sg * (1.0f - sg) * expf(-sg * ls));
                }
                sum = warp_sum(sum);
                if (lane == 0) w.dm_out[hh] = sum;
            }
            if (tid == 0) batch.status[4] = 0;
        }
    }
}

// Combine per-group partial states: exclusive prefix (forward), exclusive suffix (reverse
// time) or the total written to every group.  One thread per four consecutive state
// elements; groups are visited in batches whose loads are all issued before the first use.
__global__ void __launch_bounds__(256) scan_kernel(float* __restrict__ states,
                                                   float* __restrict__ total_out, int n_groups,
                                                   int dd, int mode, const float* scale_m,
                                                   const float* seq_len, float seq_len_scalar,
                                                   int H, int N, const float* __restrict__ init_in) {
    constexpr int kBatch = 8;
    const int e4 = blockIdx.x * blockDim.x + threadIdx.x;
    const int bh = blockIdx.y;
    // (started while the state pass drains; the walk behind it starts while this one does)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (e4 * 4 >= dd) return;
    float4* base = reinterpret_cast<float4*>(states + (size_t)bh * n_groups * dd) + e4;
    const size_t stride = (size_t)dd / 4;
    float4 run = make_float4(0.f, 0.f, 0.f, 0.f);
    // With scale_m the states being scanned are unscaled and the total is multiplied by c on
    // the way out; a caller's initial state (which contains c) enters divided by c.
    float c = 1.f;
    if (scale_m) {
        const float s_b = seq_len ? seq_len[bh / H]
                                  : (seq_len_scalar > 0.f ? seq_len_scalar : (float)N);
        c = stab_factor(scale_m[bh % H], s_b);
    }
    if (init_in) {
        const float4 v0 = reinterpret_cast<const float4*>(init_in + (size_t)bh * dd)[e4];
        const float ic = 1.0f / c;
        run = make_float4(v0.x * ic, v0.y * ic, v0.z * ic, v0.w * ic);
    }
    auto add = [](float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; };
    if (mode == SCAN_TOTAL) {
        for (int g0 = 0; g0 < n_groups; g0 += kBatch) {
            float4 v[kBatch];
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (g0 + i < n_groups) v[i] = base[(size_t)(g0 + i) * stride];
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (g0 + i < n_groups) add(run, v[i]);
        }
        for (int g = 0; g < n_groups; ++g) base[(size_t)g * stride] = run;
    } else {
        const bool rev = mode == SCAN_SUFFIX;
        for (int g0 = 0; g0 < n_groups; g0 += kBatch) {
            float4 v[kBatch];
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                const int g = rev ? n_groups - 1 - (g0 + i) : g0 + i;
                if (g0 + i < n_groups) v[i] = base[(size_t)g * stride];
            }
#pragma unroll
            for (int i = 0; i < kBatch; ++i) {
                const int g = rev ? n_groups - 1 - (g0 + i) : g0 + i;
                if (g0 + i < n_groups) {
                    base[(size_t)g * stride] = run;
                    add(run, v[i]);
                }
            }
        }
    }
    if (total_out) {
        if (scale_m) { run.x *= c; run.y *= c; run.z *= c; run.w *= c; }
        reinterpret_cast<float4*>(total_out + (size_t)bh * dd)[e4] = run;
    }
}

// dm_h = sum_b dc/dm * <dV', V>_{b,h},  dc/dm = -ln(s_b) sigma(m_h)(1-sigma(m_h)) c_{b,h}.
// Fixed summation order (deterministic).
__global__ void dm_finalize_kernel(const float* dm_partial, float* dm, const float* m,
                                   const float* seq_len, float seq_len_scalar, int B, int H,
                                   int n_groups, int N, const int* cu_seqlens) {
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= H) return;
    const float sg = 1.0f / (1.0f + expf(-m[h]));
    float total = 0.f;
    for (int b = 0; b < B; ++b) {
        const float s_b = seq_len ? seq_len[b]
                                  : (seq_len_scalar > 0.f ? seq_len_scalar
                                                          : (float)(cu_seqlens ? max(cu_seqlens[b + 1] - cu_seqlens[b], 1) : N));
        const float ls = logf(s_b);
        const float c = expf(-sg * ls);
        float acc = 0.f;
        for (int g = 0; g < n_groups; ++g) acc += dm_partial[((size_t)b * H + h) * n_groups + g];
        total += acc * (-ls * sg * (1.0f - sg) * c);
    }
    dm[h] = total;
}

// Recurrent decode step (Eq. 8): SPLIT CTAs per (b,h), each owning D / SPLIT value columns of
// the fp32 state, which streams through once with 128-bit loads and stores, update and
// read-out fused.  Every thread first issues all loads of its state elements (the CTA's whole
// share is then in flight), and only then normalises q and k, so the row norms hide behind
// the memory latency.  The column split keeps the per-thread share small (more CTAs resident,
// a shorter last wave); every CTA normalises q and k for itself and owns its columns of o.
template <int D, int SPLIT, typename T>
__global__ void __launch_bounds__(kThreads) decode_kernel(const T* q, const T* k, const T* v,
                                                          float* state, T* o, int H,
                                                          const float* m, const float* seq_len,
                                                          float seq_len_scalar) {
    constexpr int DC = D / SPLIT;         // value columns of this CTA
    constexpr int V4 = DC / 4;            // float4 per state row share
    constexpr int RG = kThreads / V4;     // rows covered per sweep
    constexpr int NIT = D / RG;
    __shared__ float qh[D], kh[D], vp[DC];
    __shared__ __align__(16) float red[RG][DC];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int bh = blockIdx.x / SPLIT, col0 = (blockIdx.x % SPLIT) * DC;
    const int b = bh / H, h = bh % H;
    const int c4 = tid % V4, r0 = tid / V4;
    float4* S = reinterpret_cast<float4*>(state + (size_t)bh * D * D + col0);   // row stride D / 4
    float4 sv[NIT];
#pragma unroll
    for (int i = 0; i < NIT; ++i) sv[i] = S[(size_t)(r0 + i * RG) * (D / 4) + c4];

    const float s_b = seq_len ? seq_len[b] : seq_len_scalar;
    const float c = stab_factor(m[h], s_b);
    if (tid < D) {
        qh[tid] = to_f32<T>(q[(size_t)bh * D + tid]);
        kh[tid] = to_f32<T>(k[(size_t)bh * D + tid]);
        if (tid < DC) vp[tid] = to_f32<T>(v[(size_t)bh * D + col0 + tid]) * c;
    }
    __syncthreads();
    if (warp < 2) {
        float* row = warp == 0 ? qh : kh;
        float ss = 0.f;
        for (int e = lane; e < D; e += 32) ss += row[e] * row[e];
        ss = warp_sum(ss);
        const float r = 1.0f / fmaxf(sqrtf(ss), kEps);
        for (int e = lane; e < D; e += 32) row[e] *= r;
    }
    __syncthreads();
    const float4 vv = *reinterpret_cast<const float4*>(&vp[c4 * 4]);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < NIT; ++i) {
        const int a = r0 + i * RG;
        const float ka = kh[a], qa = qh[a];
        sv[i].x += ka * vv.x; sv[i].y += ka * vv.y; sv[i].z += ka * vv.z; sv[i].w += ka * vv.w;
        S[(size_t)a * (D / 4) + c4] = sv[i];
        acc.x += qa * sv[i].x; acc.y += qa * sv[i].y; acc.z += qa * sv[i].z; acc.w += qa * sv[i].w;
    }
    *reinterpret_cast<float4*>(&red[r0][c4 * 4]) = acc;
    __syncthreads();
    if (tid < DC) {
        float t = 0.f;
#pragma unroll
        for (int r = 0; r < RG; ++r) t += red[r][tid];
        o[(size_t)bh * D + col0 + tid] = from_f32<T>(t);
    }
}

template <int D, typename T>
cudaError_t launch_walk_dt(const WalkBatch& wb, int n, int BH, cudaStream_t st, bool dependent) {
    if (cudaError_t e = configure_smem_once(reinterpret_cast<const void*>(walk_kernel<D, T>), WalkSmem<D>::kBytes); e != cudaSuccess)
        return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(BH * wb.w[0].n_groups), (unsigned)n);
    cfg.blockDim = dim3(WalkThreads<D>::n);
    cfg.dynamicSmemBytes = WalkSmem<D>::kBytes;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, walk_kernel<D, T>, wb);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <typename T>
cudaError_t launch_walk_t(const WalkBatch& wb, int n, int BH, int d, cudaStream_t st, bool dependent) {
    switch (d) {
        case 32: return launch_walk_dt<32, T>(wb, n, BH, st, dependent);
        case 64: return launch_walk_dt<64, T>(wb, n, BH, st, dependent);
        case 128: return launch_walk_dt<128, T>(wb, n, BH, st, dependent);
        default: return cudaErrorInvalidValue;
    }
}

template <typename T>
cudaError_t launch_decode_t(const void* q, const void* k, const void* v, float* state, void* o,
                            int B, int H, int d, const float* m, const float* seq_len,
                            float seq_len_scalar, cudaStream_t st) {
    const unsigned BH = (unsigned)(B * H);
    const T *qq = (const T*)q, *kk = (const T*)k, *vv = (const T*)v;
    T* oo = (T*)o;
    switch (d) {
        case 32: decode_kernel<32, 1, T><<<BH, kThreads, 0, st>>>(qq, kk, vv, state, oo, H, m, seq_len, seq_len_scalar); break;
        case 64: decode_kernel<64, 1, T><<<BH, kThreads, 0, st>>>(qq, kk, vv, state, oo, H, m, seq_len, seq_len_scalar); break;
        case 128: decode_kernel<128, 2, T><<<2 * BH, kThreads, 0, st>>>(qq, kk, vv, state, oo, H, m, seq_len, seq_len_scalar); break;
        default: return cudaErrorInvalidValue;
    }
    note_launch();
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_walk_simt(const WalkBatch& wb0, int n, int BH, int d, cott_dtype dt, cudaStream_t st, bool dependent) {
    WalkBatch wb = wb0;   // resolve "all zero = dense [B,H,N,d]" once, on the host
    for (int i = 0; i < n; ++i) {
        WalkArgs& w = wb.w[i];
        for (RowLayout* l : {&w.lx, &w.la, &w.lbv, &w.lproj, &w.lout}) *l = resolve_layout(*l, w.H, w.N, d);
    }
    return dt == COTT_F32 ? launch_walk_t<float>(wb, n, BH, d, st, dependent)
                          : launch_walk_t<__nv_bfloat16>(wb, n, BH, d, st, dependent);
}

// Zeroes the status words and the dm counter in front of a kernel that needs them zero on entry: unlike a
// memset it lets that kernel's prologue start while the one before drains (a backward call on 8 x 16 heads of
// 100 tokens: 14.5 us with a memset, 11.5 this way; 32 x 12 x 512 bidirectional: 62 against 60).  Its
// dependents start behind the wait, so they may read before their own what earlier kernels wrote.
__global__ void clear_status_kernel(int* status) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (threadIdx.x < 8) status[threadIdx.x] = 0;
}
cudaError_t launch_clear_status(int* status, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(32);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, clear_status_kernel, status);      // (stands for a memset: not counted)
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_scan(float* states, float* total_out, int BH, int n_groups, int d, int mode,
                        cudaStream_t st, const float* total_scale_m, const float* seq_len,
                        float seq_len_scalar, int H, int N, const float* init_in) {
    const int dd = d * d;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((dd / 4 + 255) / 256), (unsigned)BH);
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // Started while the state pass drains only where that pass leaves most SMs free (1 us): else the scan's CTAs
    // crowd onto the few that are (d = 128, 32 groups, B H = 4, N = 4096: 28 us a forward against 25 started
    // behind the pass; a readout 26 against 19).
    cfg.numAttrs = (long)BH * (n_groups - 1) <= 40 ? 1 : 0;
    if (cudaError_t e = cudaLaunchKernelEx(&cfg, scan_kernel, states, total_out, n_groups, dd, mode, total_scale_m, seq_len,
                                           seq_len_scalar, H, N, init_in); e != cudaSuccess)
        return e;
    note_launch();
    return cudaGetLastError();
}

// out[h] = sum over the n slices of parts[i][h], in slice order (deterministic).
__global__ void sum_slices_kernel(const float* parts, float* out, int n, int H) {
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= H) return;
    float acc = 0.f;
    for (int i = 0; i < n; ++i) acc += parts[(size_t)i * H + h];
    out[h] = acc;
}

cudaError_t launch_sum_slices(const float* parts, float* out, int n, int H, cudaStream_t st) {
    sum_slices_kernel<<<(H + 127) / 128, 128, 0, st>>>(parts, out, n, H);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_dm_finalize(const float* dm_partial, float* dm, const float* m,
                               const float* seq_len, float seq_len_scalar, int B, int H,
                               int n_groups, int N, cudaStream_t st, const int* cu_seqlens) {
    dm_finalize_kernel<<<(H + 127) / 128, 128, 0, st>>>(dm_partial, dm, m, seq_len,
                                                        seq_len_scalar, B, H, n_groups, N, cu_seqlens);
    note_launch();
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// Head sizes the tensor-core kernels run zero-padded (dk, dv <= their d): a caller's state
// [BH, dk, dv] enters and leaves through a padded [BH, d, d] copy in the workspace.
__global__ void pad_state_kernel(const float* __restrict__ src, float* __restrict__ dst, int dk, int dv, int d) {
    const size_t bh = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d * d; i += gridDim.x * blockDim.x) {
        const int r = i / d, c = i - r * d;
        dst[bh * d * d + i] = (r < dk && c < dv) ? src[bh * dk * dv + (size_t)r * dv + c] : 0.f;
    }
}
__global__ void unpad_state_kernel(const float* __restrict__ src, float* __restrict__ dst, int dk, int dv, int d) {
    const size_t bh = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < dk * dv; i += gridDim.x * blockDim.x) {
        const int r = i / dv, c = i - r * dv;
        dst[bh * dk * dv + i] = src[bh * d * d + (size_t)r * d + c];
    }
}
// dst[bh][c][r] = src[bh][r][c] for square d x d states.
__global__ void transpose_state_kernel(const float* __restrict__ src, float* __restrict__ dst, int d) {
    const size_t bh = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d * d; i += gridDim.x * blockDim.x) {
        const int r = i / d, c = i - r * d;
        dst[bh * d * d + (size_t)c * d + r] = src[bh * d * d + i];
    }
}
cudaError_t launch_transpose_state(const float* src, float* dst, int BH, int d, cudaStream_t st) {
    dim3 grid((unsigned)((d * d + 1023) / 1024), (unsigned)BH);
    transpose_state_kernel<<<grid, 256, 0, st>>>(src, dst, d);
    note_launch();
    return cudaGetLastError();
}
// dst = src (transposed if asked) times c[b,h] (scale_mode 1), divided by it (2) or as is (0):
// a caller's square state brought into the layout and scale a tensor-core stream starts from.
__global__ void state_prep_kernel(const float* __restrict__ src, float* __restrict__ dst, int d, int transpose, int scale_mode,
                                  const float* m, const float* seq_len, float seq_len_scalar, int H, int N) {
    const size_t bh = blockIdx.y;
    float f = 1.f;
    if (scale_mode) {
        const float s_b = seq_len ? seq_len[bh / H] : (seq_len_scalar > 0.f ? seq_len_scalar : (float)N);
        const float c = stab_factor(m[bh % H], s_b);
        f = scale_mode == 1 ? c : 1.0f / c;
    }
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d * d; i += gridDim.x * blockDim.x) {
        const int r = i / d, c2 = i - r * d;
        dst[bh * d * d + (transpose ? (size_t)c2 * d + r : (size_t)i)] = src[bh * d * d + i] * f;
    }
}
cudaError_t launch_state_prep(const float* src, float* dst, int BH, int d, int transpose, int scale_mode, const float* m,
                              const float* seq_len, float seq_len_scalar, int H, int N, cudaStream_t st) {
    dim3 grid((unsigned)((d * d + 1023) / 1024), (unsigned)BH);
    state_prep_kernel<<<grid, 256, 0, st>>>(src, dst, d, transpose, scale_mode, m, seq_len, seq_len_scalar, H, N);
    note_launch();
    return cudaGetLastError();
}

// Backward of a segment through the three tensor-core walks: what the streams' totals give.
//   tq_total [d_v][d_k] = state_in^T + c V^T K^        (the dQ^ stream's final sum, scaled)
//   tk_total [d_v][d_k] = c (d_state_out + Q^^T dO)^T  (the dK^ stream's)
// With S = K^^T V and R = Q^^T dO of the segment:
//   d_state_in = d_state_out + R = tk_total^T / c
//   the dm sum over the query rows, <q^_i, dQ^_i>, contains q^_i^T (state_in / c) dO_i, which is no
//   derivative with respect to c, and lacks <d_state_out, S>:  T = T_q - <state_in / c, R> + <d_state_out, S>.
// One CTA per (b, h); the correction (and the dK^ stream's partial sums `fold`, if any) is added to
// dm_partial[bh * n_groups], which the dm finaliser sums afterwards.
__global__ void __launch_bounds__(256) segment_finish_kernel(const float* __restrict__ state_in, const float* __restrict__ d_state_out,
                                                             const float* __restrict__ tq_total, const float* __restrict__ tk_total,
                                                             float* __restrict__ d_state_in, float* dm_partial, const float* fold,
                                                             int n_groups, int d, const float* m, const float* seq_len,
                                                             float seq_len_scalar, int H, int N) {
    const size_t bh = blockIdx.x;
    const float s_b = seq_len ? seq_len[bh / H] : (seq_len_scalar > 0.f ? seq_len_scalar : (float)N);
    const float ic = 1.0f / stab_factor(m[bh % H], s_b);
    const size_t o = bh * (size_t)d * d;
    float acc = 0.f;
    for (int i = threadIdx.x; i < d * d; i += blockDim.x) {
        const int a = i / d, b = i - a * d;                    // element [a][b] of a [d_k][d_v] state
        const size_t t = o + (size_t)b * d + a;                // its place in a transposed total
        const float dsi = tk_total[t] * ic;                    // d_state_out + R
        const float dso = d_state_out ? d_state_out[o + i] : 0.f;
        const float sin = state_in ? state_in[o + i] : 0.f;
        if (d_state_in) d_state_in[o + i] = dsi;
        const float r = dsi - dso, sl = (tq_total[t] - sin) * ic;
        acc += dso * sl - sin * ic * r;
    }
    __shared__ float red[8];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < 8; ++w) t += red[w];
        float f = 0.f;
        if (fold) for (int g = 0; g < n_groups; ++g) f += fold[bh * n_groups + g];
        dm_partial[bh * n_groups] += t + f;
    }
}
cudaError_t launch_segment_finish(const float* state_in, const float* d_state_out, const float* tq_total, const float* tk_total,
                                  float* d_state_in, float* dm_partial, const float* fold, int BH, int n_groups, int d,
                                  const float* m, const float* seq_len, float seq_len_scalar, int H, int N, cudaStream_t st) {
    segment_finish_kernel<<<(unsigned)BH, 256, 0, st>>>(state_in, d_state_out, tq_total, tk_total, d_state_in, dm_partial, fold,
                                                        n_groups, d, m, seq_len, seq_len_scalar, H, N);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_pad_state(const float* src, float* dst, int BH, int dk, int dv, int d, cudaStream_t st) {
    dim3 grid((unsigned)((d * d + 1023) / 1024), (unsigned)BH);
    pad_state_kernel<<<grid, 256, 0, st>>>(src, dst, dk, dv, d);
    note_launch();
    return cudaGetLastError();
}
cudaError_t launch_unpad_state(const float* src, float* dst, int BH, int dk, int dv, int d, cudaStream_t st) {
    dim3 grid((unsigned)((dk * dv + 1023) / 1024), (unsigned)BH);
    unpad_state_kernel<<<grid, 256, 0, st>>>(src, dst, dk, dv, d);
    note_launch();
    return cudaGetLastError();
}

// One step of Eq. 8 for any head sizes (dk keys, dv values, dv a multiple of 4): one CTA per
// (b, h); thread t owns the four state columns 4 (t % (dv/4)) .. +3 of the rows
// t / (dv/4), + 256 / (dv/4), ...: 128-bit state loads and stores, coalesced along a row; the
// per-column partial sums of o meet in shared memory.
//   S <- S + k^ (c v)^T ;  o = S^T q^      (update first, then observe)
template <typename T>
__global__ void __launch_bounds__(256) decode_generic_kernel(const T* __restrict__ q, const T* __restrict__ k,
                                                             const T* __restrict__ v, float* __restrict__ state,
                                                             T* __restrict__ o, int H, int dk, int dv,
                                                             const float* __restrict__ m, const float* __restrict__ seq_len,
                                                             float seq_len_scalar) {
    extern __shared__ float sm[];            // q^ [dk] | k^ [dk] | c v [dv] | partial o [slices][dv] | 2 norms
    float* qh = sm; float* kh = sm + dk; float* cv = kh + dk; float* part = cv + dv;
    const size_t bh = blockIdx.x;
    const int b = (int)(bh / H), h = (int)(bh % H), tid = threadIdx.x;
    const int cgs = dv / 4, slices = 256 / cgs;          // column groups, row slices (>= 1 since dv <= 1024)
    __shared__ float red[2][8];
    float sq = 0.f, sk = 0.f;
    for (int i = tid; i < dk; i += 256) {
        const float a = to_f32(q[bh * dk + i]), c2 = to_f32(k[bh * dk + i]);
        qh[i] = a; kh[i] = c2; sq = fmaf(a, a, sq); sk = fmaf(c2, c2, sk);
    }
    for (int off = 16; off; off >>= 1) { sq += __shfl_xor_sync(0xffffffffu, sq, off); sk += __shfl_xor_sync(0xffffffffu, sk, off); }
    if ((tid & 31) == 0) { red[0][tid >> 5] = sq; red[1][tid >> 5] = sk; }
    const float s_b = seq_len ? seq_len[b] : seq_len_scalar;
    const float cfac = stab_factor(m[h], s_b);
    for (int i = tid; i < dv; i += 256) cv[i] = cfac * to_f32(v[bh * dv + i]);
    __syncthreads();
    float nq = 0.f, nk = 0.f;
    for (int w = 0; w < 8; ++w) { nq += red[0][w]; nk += red[1][w]; }
    const float rq = 1.0f / fmaxf(sqrtf(nq), kEps), rk = 1.0f / fmaxf(sqrtf(nk), kEps);
    const int cg = tid % cgs, sl = tid / cgs;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    if (sl < slices) {
        const float4 vv = *reinterpret_cast<const float4*>(cv + 4 * cg);
        float4* S = reinterpret_cast<float4*>(state + bh * (size_t)dk * dv) + cg;
        for (int r = sl; r < dk; r += slices) {
            float4 x = S[(size_t)r * cgs];
            const float kr = kh[r] * rk, qr = qh[r] * rq;
            x.x = fmaf(kr, vv.x, x.x); x.y = fmaf(kr, vv.y, x.y); x.z = fmaf(kr, vv.z, x.z); x.w = fmaf(kr, vv.w, x.w);
            S[(size_t)r * cgs] = x;
            acc.x = fmaf(qr, x.x, acc.x); acc.y = fmaf(qr, x.y, acc.y); acc.z = fmaf(qr, x.z, acc.z); acc.w = fmaf(qr, x.w, acc.w);
        }
        *reinterpret_cast<float4*>(part + (size_t)sl * dv + 4 * cg) = acc;
    }
    __syncthreads();
    for (int i = tid; i < dv; i += 256) {
        float a = 0.f;
        for (int s2 = 0; s2 < slices; ++s2) a += part[(size_t)s2 * dv + i];
        o[bh * dv + i] = from_f32<T>(a);
    }
}

cudaError_t launch_decode_generic(const void* q, const void* k, const void* v, float* state, void* o,
                                  int B, int H, int dk, int dv, cott_dtype dt, const float* m,
                                  const float* seq_len, float seq_len_scalar, cudaStream_t st) {
    if (dk < 1 || dv < 4 || (dv & 3) || dv > 1024 || dk > 1024) return cudaErrorInvalidValue;
    const int cgs = dv / 4, slices = 256 / cgs;
    const size_t smem = sizeof(float) * ((size_t)2 * dk + dv + (size_t)slices * dv);
    const unsigned BH = (unsigned)(B * H);
    if (dt == COTT_F32)
        decode_generic_kernel<float><<<BH, 256, smem, st>>>((const float*)q, (const float*)k, (const float*)v, state,
                                                            (float*)o, H, dk, dv, m, seq_len, seq_len_scalar);
    else
        decode_generic_kernel<__nv_bfloat16><<<BH, 256, smem, st>>>((const __nv_bfloat16*)q, (const __nv_bfloat16*)k,
                                                                    (const __nv_bfloat16*)v, state, (__nv_bfloat16*)o, H,
                                                                    dk, dv, m, seq_len, seq_len_scalar);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_decode(const void* q, const void* k, const void* v, float* state, void* o,
                          int B, int H, int d, cott_dtype dt, const float* m,
                          const float* seq_len, float seq_len_scalar, cudaStream_t st) {
    return dt == COTT_F32
               ? launch_decode_t<float>(q, k, v, state, o, B, H, d, m, seq_len, seq_len_scalar, st)
               : launch_decode_t<__nv_bfloat16>(q, k, v, state, o, B, H, d, m, seq_len,
                                                seq_len_scalar, st);
}

}  // namespace cott
