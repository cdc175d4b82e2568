// Single-token decode over the grouped key cache and the latent value cache (App. B.1.3).
// HBM-bound: every live cache byte is read exactly once with 16-byte vector loads.
//
//   decode_partial_kernel : grid (chunk, sequence).  One CTA streams one chunk of one
//       sequence: the K rows of every key group (scores of all n_q maps), a local softmax,
//       then the latent rows C, applied to up to eight of the maps that share them at a time.
//       Writes per-(chunk, map) partials (max, sum, unnormalised latent sum) to workspace.
//   decode_chunk_merge_kernel : log-sum-exp merge of the chunk partials into the normalised latent L.
//   decode_finish_kernel  : gate pre-activation x_t W_G, decoder L W_P,i, sigmoid, store, 8 sequences
//       x 16 columns per CTA; the gate half runs before the kernel's dependency wait.
// The kernels are chained by programmatic dependent launch.
#include <float.h>

#include <type_traits>

#include "gta_common.cuh"
#include "sm100_ptx.cuh"

namespace gta {

constexpr int kDecodeThreads = 256;
constexpr int kFinishSeqs = 8;      // sequences per finish CTA
constexpr int kFinishCols = 16;     // output columns per finish CTA

struct DecodePlan {
    int chunk;       // tokens per partial CTA
    int n_chunks;    // ceil(S_cap / chunk)
    size_t off_ml, total;  // byte offsets inside the workspace (part_o at 0)
};

static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

static DecodePlan plan_of(const Dims& d, long long chunks, int chunk, int S_cap) {
    DecodePlan p;
    p.chunk = chunk;
    p.n_chunks = S_cap > 0 ? (S_cap + chunk - 1) / chunk : 1;
    p.off_ml = align256((size_t)chunks * d.n_q * d.d_l * sizeof(float));
    p.total = p.off_ml + align256((size_t)chunks * d.n_q * 2 * sizeof(float));
    return p;
}
static DecodePlan plan_of(const Dims& d, int chunk, int S_cap) {
    return plan_of(d, (long long)d.B * (S_cap > 0 ? (S_cap + chunk - 1) / chunk : 1), chunk, S_cap);
}
// Aim at >= 8 chunk CTAs per SM over the whole batch, chunks of 64..256 tokens.
static DecodePlan least_plan(const Dims& d, int S_cap) {
    const long long want = (long long)d.B * (S_cap > 0 ? S_cap : 1) / (148 * 8);
    const int chunk = (int)((want + 63) / 64) * 64;
    return plan_of(d, chunk < 64 ? 64 : chunk > 256 ? 256 : chunk, S_cap);
}
// ... and of 32 where 64 would not give every SM two CTAs (a chunk's time is then latency, not its bytes), the partial sums
// take 4 MB at the most and the workspace has room for them.
constexpr long long kSmallTokens = 148 * 2 * 64, kSmallPart = 1 << 25;
static DecodePlan make_plan(const Dims& d, int S_cap, size_t room) {
    const long long tokens = (long long)d.B * (S_cap > 0 ? S_cap : 1);
    if (tokens < kSmallTokens && tokens * d.n_q * d.d_l <= kSmallPart) {
        const DecodePlan p = plan_of(d, 32, S_cap);
        if (p.total <= room) return p;
    }
    return least_plan(d, S_cap);
}
// Room for the plan of every smaller batch and capacity too, so that a buffer for the largest call serves the others.  The
// chunks of a call are at most tokens / chunk + batch: 592 + batch of 32 tokens (fewer where their sums would pass 4 MB),
// 1203 + batch of 64 (a chunk is 64 up to 65 x 1184 tokens) and of 128 and 192 likewise, and what 256 tokens each make.
static size_t plan_bound(const Dims& d, int S_cap) {
    const long long S = S_cap > 0 ? S_cap : 1, small = kSmallPart / 32 / ((long long)d.n_q * d.d_l);
    const auto least = [](long long a, long long b) { return a < b ? a : b; };
    const long long n32 = least(d.B * ((S + 31) / 32), least(kSmallTokens / 32, small) + d.B);
    const long long n64 = least(d.B * ((S + 63) / 64), 1203 + d.B), n256 = d.B * ((S + 255) / 256);
    const long long most = n32 > n64 ? n32 : n64;
    return plan_of(d, most > n256 ? most : n256, 64, S_cap).total;
}

// The kernel family is a function of shape, dtype and page size only, so the sizes are that family's -- but over small pages
// (which had no other kernels once) the plain-ALU kernels take what the stream kernel's workspace is too much for.
static bool small_pages(int page_size) { return page_size % 64 != 0; }
size_t decode_workspace_bytes(const Dims& d, int dtype, int S_cap, int page_size) {
    if (decode_fast_supported(d, dtype, page_size) && S_cap > 0) return decode_fast_workspace_bytes(d, page_size);
    return plan_bound(d, S_cap);
}
size_t decode_least_workspace(const Dims& d, int dtype, int S_cap, int page_size) {
    const size_t plain = least_plan(d, S_cap).total;
    if (!decode_fast_supported(d, dtype, page_size) || S_cap <= 0) return plain;
    const size_t fast = decode_fast_workspace_bytes(d, page_size);
    return small_pages(page_size) && plain < fast ? plain : fast;
}

// ---- 16-byte vector of storage elements, widened to fp32 ----
template <typename T> struct Vec16;
template <> struct Vec16<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ void widen(const uint4& r, float (&v)[4]) {
        v[0] = __uint_as_float(r.x); v[1] = __uint_as_float(r.y); v[2] = __uint_as_float(r.z); v[3] = __uint_as_float(r.w);
    }
    static __device__ __forceinline__ void load(const float* p, float (&v)[4]) {
        widen(__ldg(reinterpret_cast<const uint4*>(p)), v);
    }
};
template <> struct Vec16<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ void widen(const uint4& r, float (&v)[8]) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // bf16 is the upper half of an fp32
            v[2 * i] = __uint_as_float(w[i] << 16);
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    static __device__ __forceinline__ void load(const __nv_bfloat16* p, float (&v)[8]) {
        widen(__ldg(reinterpret_cast<const uint4*>(p)), v);
    }
};

// e4m3 codes (1 sign, 4 exponent, 3 mantissa bits, bias 7): the seven low bits, put where fp32 keeps the low four
// exponent bits and the top three mantissa bits, are the value times 2^-120 -- for the subnormal codes too --,
// so one exact multiplication by 2^120 finishes the conversion.
struct Fp8 { uint8_t bits; };
__device__ __forceinline__ float e4m3_to_f32(uint32_t b) {
    return __uint_as_float(((b & 0x80u) << 24) | ((b & 0x7fu) << 20)) * 1.329227995784916e36f;   // 2^120
}
template <> struct Vec16<Fp8> {
    static constexpr int N = 16;
    static __device__ __forceinline__ void widen(const uint4& r, float (&v)[16]) {
        const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) v[4 * i + j] = e4m3_to_f32(w[i] >> (8 * j));
    }
    static __device__ __forceinline__ void load(const Fp8* p, float (&v)[16]) {
        widen(__ldg(reinterpret_cast<const uint4*>(p)), v);
    }
};

template <typename T> __device__ __forceinline__ float exp_fn(float x);
template <> __device__ __forceinline__ float exp_fn<float>(float x) { return expf(x); }
template <> __device__ __forceinline__ float exp_fn<__nv_bfloat16>(float x) { return __expf(x); }

// What a thread keeps of a latent row: 16 bytes, or 8 codes of an 8-bit cache (16 would take 128 accumulators for eight
// maps).
template <typename CT> struct LatentVec { using Raw = uint4; static constexpr int N = Vec16<CT>::N; };
template <> struct LatentVec<Fp8> { using Raw = uint2; static constexpr int N = 8; };
__device__ __forceinline__ void widen_latent(const float*, const uint4& r, float (&v)[4]) { Vec16<float>::widen(r, v); }
__device__ __forceinline__ void widen_latent(const __nv_bfloat16*, const uint4& r, float (&v)[8]) { Vec16<__nv_bfloat16>::widen(r, v); }
__device__ __forceinline__ void widen_latent(const Fp8*, const uint2& r, float (&v)[8]) {
    const uint32_t w[2] = {r.x, r.y};
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) v[4 * i + j] = e4m3_to_f32(w[i] >> (8 * j));
}

// Dynamic shared memory of decode_partial_kernel (floats): q_s [n_q][d_h] | p_s [chunk][n_q] | red [CM][R][d_l]
static size_t partial_smem(const Dims& d, int chunk, int cm, int vec) {
    const int R = kDecodeThreads / (d.d_l / vec);
    return ((size_t)d.n_q * d.d_h + (size_t)((chunk * d.n_q + 3) & ~3) + (size_t)cm * R * d.d_l) * sizeof(float);
}

// Tokens of a sequence that a step attends over: those of the cache, and the new one where the step appends it and it fits.
__device__ __forceinline__ int step_len(int len, int S_cap, bool append) {
    if (append && len >= 0 && len < S_cap) return len + 1;
    return len < 0 ? 0 : (len > S_cap ? S_cap : len);
}

// A piece of a cached row; kAppend: of a row that this CTA may have written.
template <bool kAppend, typename V> __device__ __forceinline__ V cache_load(const V* p) {
    if constexpr (kAppend) return *p;
    else return __ldg(p);
}

// CT: storage type of the caches (T, or Fp8 with one fp32 scale per cached row in k_scale / c_scale).  CM: maps of a
// latent group that a pass over its rows serves (the last pass may have fewer).
// Every key row is loaded once, whatever the number of maps of its group, and a latent row once per CM maps: the caches
// may sit behind the host link, where a row that is loaded again crosses the link again.  The first latent rows are
// fetched ahead of the scores.  What bounds it on device memory at small batches is the chain of latencies -- length,
// rows, scores, CTA barriers, sums -- and the length of a warp's instruction stream, on host memory the link.  (Four fp32
// sequences of about 1100 tokens, five maps, under the profiler: 16.8 us with the loops over maps unrolled and predicated,
// 9.4 us now; a pass over the latent rows and a pair of barriers per map took about the former.)
// kAppend: a fused step, whose new rows the CTA of their chunk puts into the caches and then reads like the others, with loads that see
// what the CTA has written.  (Rows told apart at every load cost the long contexts more than the launch that is saved: 16 sequences
// of 8000 tokens, eight maps, 285 -> 305 us; a body of its own for that CTA 2 us of code that is fetched late.)
template <typename T, typename CT, int CM, bool kAppend>
__global__ void __launch_bounds__(kDecodeThreads)
decode_partial_kernel(Dims d, int chunk, int n_chunks, int S_cap, const T* __restrict__ q,
                      std::conditional_t<kAppend, CT*, const CT*> k_cache, std::conditional_t<kAppend, CT*, const CT*> c_cache,
                      const int32_t* __restrict__ seq_lens, float* __restrict__ part_o,
                      float* __restrict__ part_ml, PageMap pm, int32_t* status_word,
                      const float* __restrict__ k_scale, const float* __restrict__ c_scale,
                      const CT* __restrict__ k_new, const CT* __restrict__ c_new) {
    constexpr int VEC = Vec16<CT>::N, CV = LatentVec<CT>::N;
    constexpr bool kScaled = !std::is_same<CT, T>::value;
    using Raw = typename LatentVec<CT>::Raw;
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int b = blockIdx.y, ck = blockIdx.x;
    const int old = seq_lens[b];
    // (a thread's first piece of the new rows is asked for beside the length)
    uint4 piece = make_uint4(0u, 0u, 0u, 0u);
    const int k_vecs = d.n_k * d.d_h / VEC, new_vecs = kAppend ? k_vecs + d.n_c * d.d_l / VEC : 0;
    const auto new_piece = [&](int i) {
        return __ldg(i < k_vecs ? reinterpret_cast<const uint4*>(k_new) + (size_t)b * k_vecs + i
                                : reinterpret_cast<const uint4*>(c_new) + (size_t)b * (new_vecs - k_vecs) + i - k_vecs);
    };
    if (kAppend && (int)threadIdx.x < new_vecs) piece = new_piece(threadIdx.x);
    const int len = step_len(old, S_cap, kAppend);
    const int j_begin = ck * chunk;
    if (kAppend && ck == 0 && threadIdx.x == 0 && (old < 0 || old >= S_cap)) raise_status(status_word, GTA_ERR_CACHE_FULL);
    if (j_begin >= len) return;
    const int n_tok = min(chunk, len - j_begin);
    if constexpr (kAppend) {
        if (len == old + 1 && j_begin + n_tok == len) {
            for (int i = threadIdx.x; i < new_vecs; i += kDecodeThreads) {
                const bool key = i < k_vecs;
                const int e = (key ? i : i - k_vecs) * VEC, width = key ? d.d_h : d.d_l, grp = e / width;
                CT* plane = key ? k_cache + (size_t)b * d.n_k * S_cap * d.d_h : c_cache + (size_t)b * d.n_c * S_cap * d.d_l;
                *reinterpret_cast<uint4*>(plane + ((size_t)grp * S_cap + old) * width + (e - grp * width)) = piece;
                if (i + kDecodeThreads < new_vecs) piece = new_piece(i + kDecodeThreads);
            }
            __syncthreads();
        }
    }

    extern __shared__ __align__(16) float smem[];
    float* q_s = smem;
    float* p_s = q_s + d.n_q * d.d_h;
    float* red = p_s + ((chunk * d.n_q + 3) & ~3);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr int kWarps = kDecodeThreads / 32;

    // row of token j_begin + j (a block-table entry outside the pool raises the status word; row 0 of the pool stands in)
    auto row_of = [&](int groups, int grp, int j) -> size_t {
        if (pm.table == nullptr) return ((size_t)b * groups + grp) * S_cap + j_begin + j;
        const long long i = cache_row(pm, b, groups, grp, S_cap, j_begin + j, status_word);
        return (size_t)(i < 0 ? 0 : i);
    };

    // ---- latent rows: tpr threads per row, R rows of the CTA at once, U of them per thread in flight
    constexpr int U = 8;
    const int tpr = d.d_l / CV, R = kDecodeThreads / tpr;
    const bool active = tid < R * tpr;
    const int r = tid / tpr, v = tid % tpr;
    Raw raw[U];
    float cs[U];
    auto fetch = [&](int cg, int j0) {      // rows j0 + r, j0 + r + R, ...
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = j0 + r + u * R;
            if (active && j < n_tok) {
                const size_t idx = row_of(d.n_c, cg, j);
                raw[u] = cache_load<kAppend>(reinterpret_cast<const Raw*>(c_cache + idx * d.d_l + v * CV));
                cs[u] = kScaled ? c_scale[idx] : 1.f;
            }
        }
    };
    fetch(0, 0);

    for (int e = tid; e < d.n_q * d.d_h; e += kDecodeThreads)
        q_s[e] = to_f32(q[(size_t)b * d.n_q * d.d_h + e]);
    __syncthreads();

    // ---- scores: 2^lg lanes share one K row, a 16-byte vector per lane and step; the rows' loads ahead of the maps' loop
    {
        constexpr int kScoreRows = 4;                       // rows per lane group whose loads are issued together
        constexpr int kSlots = (256 / VEC + 31) / 32;       // vectors per lane and row (d_h <= 256): 2 for fp32, else 1
        const int vecs_per_row = d.d_h / VEC;
        int lg = 0;
        while ((1 << lg) < vecs_per_row && lg < 5) ++lg;
        const int lpr = 1 << lg, rows_per_warp = 32 >> lg, sub = lane >> lg, sl = lane & (lpr - 1);
        const int q_per_k = d.n_q / d.n_k, step = kWarps * rows_per_warp;
        for (int kg = 0; kg < d.n_k; ++kg) {
            for (int w0 = warp * rows_per_warp; w0 < n_tok; w0 += step * kScoreRows) {
                const int j0 = w0 + sub;
                uint4 kraw[kScoreRows][kSlots];
                float row_scale[kScoreRows];
#pragma unroll
                for (int u = 0; u < kScoreRows; ++u) {
                    const int j = j0 + u * step;
                    row_scale[u] = d.scale;
#pragma unroll
                    for (int s = 0; s < kSlots; ++s) kraw[u][s] = make_uint4(0u, 0u, 0u, 0u);
                    if (j < n_tok) {
                        const size_t idx = row_of(d.n_k, kg, j);
                        if (kScaled) row_scale[u] *= k_scale[idx];
#pragma unroll
                        for (int s = 0; s < kSlots; ++s)
                            if (sl + s * lpr < vecs_per_row)
                                kraw[u][s] = cache_load<kAppend>(reinterpret_cast<const uint4*>(k_cache + idx * d.d_h + (sl + s * lpr) * VEC));
                    }
                }
#pragma unroll 1
                for (int g = kg * q_per_k; g < (kg + 1) * q_per_k; ++g) {
                    float dot[kScoreRows];
#pragma unroll
                    for (int u = 0; u < kScoreRows; ++u) dot[u] = 0.f;
#pragma unroll
                    for (int s = 0; s < kSlots; ++s) {
                        if (sl + s * lpr < vecs_per_row) {
                            float qv[VEC];
#pragma unroll
                            for (int e = 0; e < VEC; e += 4) {
                                const float4 q4 = *reinterpret_cast<const float4*>(q_s + g * d.d_h + (sl + s * lpr) * VEC + e);
                                qv[e] = q4.x; qv[e + 1] = q4.y; qv[e + 2] = q4.z; qv[e + 3] = q4.w;
                            }
#pragma unroll
                            for (int u = 0; u < kScoreRows; ++u) {
                                float kv[VEC];
                                Vec16<CT>::widen(kraw[u][s], kv);
#pragma unroll
                                for (int e = 0; e < VEC; ++e) dot[u] = fmaf(qv[e], kv[e], dot[u]);
                            }
                        }
                    }
                    for (int o = lpr >> 1; o > 0; o >>= 1) {
#pragma unroll
                        for (int u = 0; u < kScoreRows; ++u) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], o);
                    }
                    if (sl == 0) {
#pragma unroll
                        for (int u = 0; u < kScoreRows; ++u)
                            if (j0 + u * step < n_tok) p_s[(j0 + u * step) * d.n_q + g] = dot[u] * row_scale[u];
                    }
                }
            }
        }
    }
    __syncthreads();

    // ---- chunk-local softmax per map: m = max, p = exp(s - m), l = sum p ----
    for (int g = warp; g < d.n_q; g += kWarps) {
        float m = -INFINITY;
        for (int j = lane; j < n_tok; j += 32) m = fmaxf(m, p_s[j * d.n_q + g]);
        m = warp_max(m);
        float l = 0.f;
        for (int j = lane; j < n_tok; j += 32) {
            const float p = exp_fn<T>(p_s[j * d.n_q + g] - m);
            p_s[j * d.n_q + g] = p;
            l += p;
        }
        l = warp_sum(l);
        if (lane == 0) {
            float* ml = part_ml + (((size_t)b * n_chunks + ck) * d.n_q + g) * 2;
            ml[0] = m;
            ml[1] = l;
        }
    }
    __syncthreads();

    // ---- latent sums
    const int maps_per_c = d.n_q / d.n_c;
    for (int cg = 0; cg < d.n_c; ++cg) {
        const int g_end = (cg + 1) * maps_per_c;
        for (int g0 = cg * maps_per_c; g0 < g_end; g0 += CM) {
            float acc[CM][CV];
#pragma unroll
            for (int gi = 0; gi < CM; ++gi)
#pragma unroll
                for (int e = 0; e < CV; ++e) acc[gi][e] = 0.f;
            for (int j0 = 0; j0 < n_tok; j0 += U * R) {
                if (g0 > 0 || j0 > 0) fetch(cg, j0);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int j = j0 + r + u * R;
                    if (!active || j >= n_tok) break;
                    float cv[CV];
                    widen_latent((const CT*)nullptr, raw[u], cv);
                    const float* pj = p_s + j * d.n_q + g0;
#pragma unroll
                    for (int gi = 0; gi < CM; ++gi) {
                        if (g0 + gi >= g_end) break;
                        const float p = pj[gi] * cs[u];          // the row's scale folded into its probability
#pragma unroll
                        for (int e = 0; e < CV; ++e) acc[gi][e] = fmaf(p, cv[e], acc[gi][e]);
                    }
                }
            }
            // add up the R row slots through shared memory
            const int maps = min(CM, g_end - g0);
            if (g0 > 0) __syncthreads();
            if (active) {
#pragma unroll
                for (int gi = 0; gi < CM; ++gi) {
                    if (gi >= maps) break;
#pragma unroll
                    for (int e = 0; e < CV; e += 4)
                        *reinterpret_cast<float4*>(red + ((size_t)gi * R + r) * d.d_l + v * CV + e) =
                            make_float4(acc[gi][e], acc[gi][e + 1], acc[gi][e + 2], acc[gi][e + 3]);
                }
            }
            __syncthreads();
            float* dst = part_o + (((size_t)b * n_chunks + ck) * d.n_q + g0) * d.d_l;
            for (int idx = tid * 4; idx < maps * d.d_l; idx += kDecodeThreads * 4) {
                const int gi = idx / d.d_l;
                const float* src = red + (size_t)gi * R * d.d_l + (idx - gi * d.d_l);
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
                for (int rr = 0; rr < R; ++rr) {
                    const float4 x = *reinterpret_cast<const float4*>(src + rr * d.d_l);
                    s.x += x.x; s.y += x.y; s.z += x.z; s.w += x.w;
                }
                *reinterpret_cast<float4*>(dst + idx) = s;
            }
        }
    }
}

// What a fused step appends, and where: rows [B, groups, width], the caches they go to, the lengths that advance.
struct StepAppend {
    const void *k_new, *c_new;
    void *k_cache, *c_cache;
    int32_t* seq_lens;
};

// Log-sum-exp merge of the chunk partials of one (map, sequence), in place: the normalised latent L takes the room of the
// sequence's first chunk, whose weight becomes one and that of the others nothing, so that a second merge finds L again
// (gta_decode_stages).  The threads form groups that cover a
// pass of the d_l columns, four each; group i takes the chunks i, i + groups, ..., and the groups' results meet in
// shared memory: a chain of rounds of loads over all chunks would be what the kernel waits for.
__global__ void __launch_bounds__(kDecodeThreads)
decode_chunk_merge_kernel(Dims d, int chunk, int n_chunks, int S_cap, const int32_t* __restrict__ seq_lens,
                          float* part_o, float* part_ml, bool append) {
    __shared__ float4 acc_s[kDecodeThreads];
    __shared__ float2 ml_s[kDecodeThreads];
    ptx::grid_launch_dependents();
    const int g = blockIdx.x, b = blockIdx.y, tid = threadIdx.x;
    const int width = min(d.d_l >> 2, kDecodeThreads), groups = kDecodeThreads / width;
    const int grp = tid / width, v = tid - grp * width;
    const int len = step_len(seq_lens[b], S_cap, append);  // (older than the partial kernel, which was released after its own wait)
    const int live = (len + chunk - 1) / chunk;
    ptx::grid_dependency_wait();
    float2* ml = reinterpret_cast<float2*>(part_ml) + (size_t)b * n_chunks * d.n_q + g;
    float* po = part_o + ((size_t)b * n_chunks * d.n_q + g) * d.d_l;
    for (int col0 = 0; col0 < d.d_l; col0 += 4 * kDecodeThreads) {
        const int col = col0 + 4 * v;
        float m = -INFINITY, l = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (grp < groups && col < d.d_l) {
            constexpr int U = 8;                             // chunks whose loads are issued together
            for (int c0 = grp; c0 < live; c0 += U * groups) {
                float2 x[U];
                float4 p[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int c = c0 + u * groups;
                    x[u] = make_float2(-INFINITY, 0.f);
                    p[u] = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (c < live) {
                        x[u] = ml[(size_t)c * d.n_q];
                        p[u] = *reinterpret_cast<const float4*>(po + (size_t)c * d.n_q * d.d_l + col);
                    }
                }
                float mn = m;
#pragma unroll
                for (int u = 0; u < U; ++u) mn = fmaxf(mn, x[u].x);
                const float old = expf(m - mn);              // 0 on the first round
                l *= old;
                acc.x *= old; acc.y *= old; acc.z *= old; acc.w *= old;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float w = expf(x[u].x - mn);
                    l = fmaf(x[u].y, w, l);
                    acc.x = fmaf(p[u].x, w, acc.x); acc.y = fmaf(p[u].y, w, acc.y);
                    acc.z = fmaf(p[u].z, w, acc.z); acc.w = fmaf(p[u].w, w, acc.w);
                }
                m = mn;
            }
        }
        acc_s[tid] = acc;
        ml_s[tid] = make_float2(m, l);
        __syncthreads();
        if (grp == 0 && col < d.d_l) {
            float mn = m;
            for (int i = 1; i < groups; ++i) mn = fmaxf(mn, ml_s[i * width + v].x);
            float ls = 0.f;
            float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int i = 0; i < groups; ++i) {
                const float2 x = ml_s[i * width + v];
                const float w = x.x == -INFINITY ? 0.f : expf(x.x - mn);
                const float4 p = acc_s[i * width + v];
                ls = fmaf(x.y, w, ls);
                o.x = fmaf(p.x, w, o.x); o.y = fmaf(p.y, w, o.y); o.z = fmaf(p.z, w, o.z); o.w = fmaf(p.w, w, o.w);
            }
            const float inv = live > 0 ? 1.f / ls : 0.f;     // an empty sequence gives zeros
            *reinterpret_cast<float4*>(po + col) =     // (these columns of every chunk have been read)
                make_float4(o.x * inv, o.y * inv, o.z * inv, o.w * inv);
        }
        __syncthreads();
    }
    for (int c = tid; c < live; c += kDecodeThreads)
        ml[(size_t)c * d.n_q] = c == 0 ? make_float2(0.f, 1.f) : make_float2(-FLT_MAX, 0.f);
}

// Four neighbouring elements as floats.
__device__ __forceinline__ float4 ldg4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 widen4(const uint2 r) {
    return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                       __uint_as_float(r.y & 0xffff0000u));
}
__device__ __forceinline__ float4 ldg4(const __nv_bfloat16* p) { return widen4(__ldg(reinterpret_cast<const uint2*>(p))); }

// Four neighbouring weights as they are stored, on their way to shared memory by cp.async and from there.
template <typename T> struct Weights4;
template <> struct Weights4<float> {
    using Raw = float4;
    static __device__ __forceinline__ void copy(Raw* dst, const float* src) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ptx::smem_addr(dst)), "l"(src) : "memory");
    }
    static __device__ __forceinline__ float4 widen(const Raw& r) { return r; }
};
template <> struct Weights4<__nv_bfloat16> {
    using Raw = uint2;
    static __device__ __forceinline__ void copy(Raw* dst, const __nv_bfloat16* src) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(ptx::smem_addr(dst)), "l"(src) : "memory");
    }
    static __device__ __forceinline__ float4 widen(const Raw& r) { return widen4(r); }
};

// The finish kernel's contractions in slabs of at most `size` elements: those of X W_G, then those of L W_P.  The weights
// of a slab and of the one behind it are on their way at once: buffers of even and odd slabs in turn, every thread the
// pieces that it uses itself.  1280 elements where every CTA has an SM to itself and the gate's weights are one such slab, 640
// otherwise: a CTA then leaves room for another, and for the partial kernel's CTAs, beside which it fetches its weights (the whole
// fp32 step, us, 1280 / 640: 1B layer, four sequences of about 1100 tokens 16.4 / 17.9, 8 of 500 15.9 / 19.0, 16 of 500 23.1 / 20.0;
// 2048 wide, 16 heads of 128: 4 of 100 22.7 / 19.0, 8 of 100 26.7 / 21.5, 4 of 2000 24.8 / 28.2).
struct FinishSlabs {
    int size;                      // a multiple of 64
    int gate, all;                 // slabs of the gate; of both
    int even_pieces, odd_pieces;   // of a thread, in the two buffers
};
static FinishSlabs finish_slabs(const Dims& d, long long ctas) {
    FinishSlabs f;
    f.size = ctas <= 148 && d.H <= 1280 ? 1280 : 640;
    f.gate = (d.H + f.size - 1) / f.size;
    f.all = f.gate + (d.d_l + f.size - 1) / f.size;
    f.even_pieces = f.odd_pieces = 0;
    for (int i = 0; i < f.all; ++i) {
        const int left = i < f.gate ? d.H - i * f.size : d.d_l - (i - f.gate) * f.size;
        const int pieces = ((left < f.size ? left : f.size) + 63) / 64;
        int& most = i & 1 ? f.odd_pieces : f.even_pieces;
        if (pieces > most) most = pieces;
    }
    return f;
}
// Adds acc up over the 64 k-slices of the CTA; the sum of (row, column) ends in thread row 16 + column (tid < 128).
__device__ __forceinline__ float finish_reduce(float (&acc)[8][4], float* red) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the lanes of a warp that share columns halve the rows among them: 8 -> 4 -> 2 -> 1 row per lane
#pragma unroll
    for (int h = 4; h >= 1; h >>= 1) {
        const bool up = (lane & (4 * h)) != 0;
#pragma unroll
        for (int i = 0; i < h; ++i)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float give = up ? acc[i][c] : acc[i + h][c], keep = up ? acc[i + h][c] : acc[i][c];
                acc[i][c] = keep + __shfl_xor_sync(0xffffffffu, give, 4 * h);
            }
    }
    // the row this lane ended with: bits 16, 8, 4 of the lane are bits 4, 2, 1 of the row
    const int row = lane >> 2;
    *reinterpret_cast<float4*>(red + (warp * 8 + row) * kFinishCols + 4 * (lane & 3)) =
        make_float4(acc[0][0], acc[0][1], acc[0][2], acc[0][3]);
    __syncthreads();
    float s = 0.f;
    if (tid < 128) {
#pragma unroll
        for (int w = 0; w < 8; ++w) s += red[w * 128 + tid];
    }
    return s;
}

// Gate, decoder and store of 8 sequences x 16 columns of one head.  The gate's half needs only x_t and W_G and runs
// before the dependency wait, under the kernels ahead; after it come one pass over W_P's columns and the store.
// Narrow tiles, because at small batches the weights' way through few SMs sets the time (1280 columns: 80 CTAs; the
// former pair of kernels, a head and a 128-column block per CTA, took 18.6 + 19.6 us for four fp32 sequences), and all of a
// CTA's weights asked for at once (four fp32 sequences of about 1100 tokens, the whole step: 16.4 us; with eight
// pieces a thread in registers 20.5).
// Dynamic shared memory: weights [even pieces][256], [odd pieces][256] | xs [2][slab][4] | red [2][8 warps][8][16]
template <typename T>
__global__ void __launch_bounds__(kDecodeThreads)
decode_finish_kernel(Dims d, int tiles_per_head, FinishSlabs slabs, const T* __restrict__ x_t, const float* l_in, size_t seq_stride,
                     const T* __restrict__ w_p, const T* __restrict__ w_g, T* __restrict__ out, int32_t* step_lens, int S_cap) {
    using W = Weights4<T>;
    extern __shared__ __align__(16) float smem[];
    typename W::Raw* w_s = reinterpret_cast<typename W::Raw*>(smem);
    float* xs = reinterpret_cast<float*>(w_s + (slabs.even_pieces + slabs.odd_pieces) * kDecodeThreads);
    float* red = xs + 2 * slabs.size * 4;
    ptx::grid_launch_dependents();
    const int tid = threadIdx.x, ks = tid >> 2;
    const int i = blockIdx.x / tiles_per_head, e0 = (blockIdx.x % tiles_per_head) * kFinishCols, b0 = blockIdx.y * kFinishSeqs;
    const int nb = min(kFinishSeqs, d.B - b0), col = e0 + 4 * (tid & 3);
    const bool live = col < d.d_h;                          // (d_h is a multiple of 8)
    const T* wg_col = w_g + (size_t)i * d.d_h + col;
    const T* wp_col = w_p + (size_t)i * d.d_l * d.d_h + col;
    const size_t ldw_g = (size_t)d.n_h * d.d_h;

    // this thread's weights of a slab: k = ks + 64 u
    const auto fetch = [&](int s) {
        if (s < slabs.all && live) {
            const bool gate = s < slabs.gate;
            const int k0 = (gate ? s : s - slabs.gate) * slabs.size, n = min(slabs.size, (gate ? d.H : d.d_l) - k0);
            const T* src = (gate ? wg_col : wp_col) + (size_t)(k0 + ks) * (gate ? ldw_g : (size_t)d.d_h);
            typename W::Raw* dst = w_s + (s & 1 ? slabs.even_pieces * kDecodeThreads : 0) + tid;
            for (int k = ks; k < n; k += 64, src += 64 * (gate ? ldw_g : (size_t)d.d_h), dst += kDecodeThreads) W::copy(dst, src);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(0);
    fetch(1);

    float acc[8][4], z = 0.f;
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0.f;
    for (int s = 0; s < slabs.all; ++s) {
        const bool gate = s < slabs.gate;
        if (s == slabs.gate) {
            z = finish_reduce(acc, red);
#pragma unroll
            for (int r = 0; r < 8; ++r) acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0.f;
            ptx::grid_dependency_wait();
        }
        const int k0 = (gate ? s : s - slabs.gate) * slabs.size, n = min(slabs.size, (gate ? d.H : d.d_l) - k0);
        if (s > 0) __syncthreads();                          // the slab before has been read
        // its rows lie in shared memory four by four ([2][slab][4]), so that the eight k of a warp are 128 contiguous bytes
        for (int idx = tid; idx < 2 * n; idx += kDecodeThreads) {
            const int r = idx & 7, k = (idx >> 3) * 4;
            if (r < nb) {
                float4 x;
                if (gate) x = ldg4(x_t + (size_t)(b0 + r) * d.H + k0 + k);
                else x = *reinterpret_cast<const float4*>(l_in + (size_t)(b0 + r) * seq_stride + (size_t)d.head_to_q(i) * d.d_l + k0 + k);
                float* dst = xs + ((r >> 2) * slabs.size + k) * 4 + (r & 3);
                dst[0] = x.x; dst[4] = x.y; dst[8] = x.z; dst[12] = x.w;
            }
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        if (live) {
            const typename W::Raw* wv = w_s + (s & 1 ? slabs.even_pieces * kDecodeThreads : 0) + tid;
            const auto rows = [&](int k, const float4 w, int h) {
                const float4 a = *reinterpret_cast<const float4*>(xs + (h * slabs.size + k) * 4);
                const float xr[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    acc[4 * h + r][0] = fmaf(xr[r], w.x, acc[4 * h + r][0]);
                    acc[4 * h + r][1] = fmaf(xr[r], w.y, acc[4 * h + r][1]);
                    acc[4 * h + r][2] = fmaf(xr[r], w.z, acc[4 * h + r][2]);
                    acc[4 * h + r][3] = fmaf(xr[r], w.w, acc[4 * h + r][3]);
                }
            };
            if (nb > 4) {
#pragma unroll 4
                for (int k = ks; k < n; k += 64, wv += kDecodeThreads) {
                    const float4 w = W::widen(*wv);
                    rows(k, w, 0);
                    rows(k, w, 1);
                }
            } else {
#pragma unroll 4
                for (int k = ks; k < n; k += 64, wv += kDecodeThreads) rows(k, W::widen(*wv), 0);
            }
        }
        fetch(s + 2);                                        // into the pieces that this thread has just used
    }
    const float y = finish_reduce(acc, red + 8 * 128);
    // a fused step: the kernels that read the lengths are complete
    if (step_lens != nullptr && blockIdx.x == 0 && blockIdx.y == 0)
        for (int b = tid; b < d.B; b += kDecodeThreads) {
            const int len = step_lens[b];
            if (len >= 0 && len < S_cap) step_lens[b] = len + 1;
        }
    const int r = tid >> 4, c = e0 + (tid & 15);
    if (tid < 128 && r < nb && c < d.d_h)
        out[((size_t)(b0 + r) * d.n_h + i) * d.d_h + c] = from_f32<T>(y * (1.f / (1.f + expf(-z))));
}

// behind: programmatic stream serialisation.  The first kernel of a call is launched so only if it waits before it touches
// anything; the merge and the finish kernel do not (they rely on the kernel ahead for that), so where a stage mask begins with
// one of them, it is launched the ordinary way.
template <typename Kern, typename... Args>
static cudaError_t launch_chained(bool behind, Kern kern, dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
    if (smem > 48 * 1024) {
        const cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (err != cudaSuccess) return err;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = behind ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <typename T, typename CT>
static cudaError_t launch_decode_typed(const Dims& d, const void* q, const void* k_cache, const void* c_cache,
                                       const int32_t* seq_lens, int S_cap, const void* x_t, const void* w_p,
                                       const void* w_g, void* out, void* workspace, size_t room, int32_t* status_word,
                                       cudaStream_t stream, int stages, int* launches, const PageMap& pm,
                                       const float* k_scale = nullptr, const float* c_scale = nullptr,
                                       const StepAppend* append = nullptr) {
    const DecodePlan p = make_plan(d, S_cap, room);
    float* part_o = reinterpret_cast<float*>(workspace);
    float* part_ml = reinterpret_cast<float*>(static_cast<char*>(workspace) + p.off_ml);
    cudaError_t err;

    if ((stages & 2) && S_cap > 0) {
        const int maps = d.n_q / d.n_c;
        const auto go = [&](auto cm) {
            constexpr int CM = decltype(cm)::value;
            const size_t smem = partial_smem(d, p.chunk, CM, LatentVec<CT>::N);
            if constexpr (std::is_same<CT, T>::value) {
                if (append != nullptr)
                    return launch_chained(true, decode_partial_kernel<T, CT, CM, true>, dim3(p.n_chunks, d.B), kDecodeThreads, smem, stream, d,
                                         p.chunk, p.n_chunks, S_cap, (const T*)q, (CT*)append->k_cache, (CT*)append->c_cache, seq_lens,
                                         part_o, part_ml, pm, status_word, k_scale, c_scale, (const CT*)append->k_new,
                                         (const CT*)append->c_new);
            }
            return launch_chained(true, decode_partial_kernel<T, CT, CM, false>, dim3(p.n_chunks, d.B), kDecodeThreads, smem, stream, d, p.chunk,
                                 p.n_chunks, S_cap, (const T*)q, (const CT*)k_cache, (const CT*)c_cache, seq_lens, part_o, part_ml, pm,
                                 status_word, k_scale, c_scale, (const CT*)nullptr, (const CT*)nullptr);
        };
        // as few passes over the latent rows as the accumulators allow (and as shared memory does, with very many maps)
        const auto fits = [&](int cm) { return partial_smem(d, p.chunk, cm, LatentVec<CT>::N) <= 227 * 1024; };
        err = maps >= 5 && fits(8)   ? go(std::integral_constant<int, 8>{})
              : maps >= 3 && fits(4) ? go(std::integral_constant<int, 4>{})
              : maps >= 2 && fits(2) ? go(std::integral_constant<int, 2>{})
                                     : go(std::integral_constant<int, 1>{});
        if (err != cudaSuccess) return err;
        *launches += 1;
    }
    if (stages & 4) {
        err = launch_chained((stages & 2) && S_cap > 0, decode_chunk_merge_kernel, dim3(d.n_q, d.B), kDecodeThreads, 0, stream, d,
                             p.chunk, p.n_chunks, S_cap, seq_lens, part_o, part_ml, append != nullptr);
        if (err != cudaSuccess) return err;
        const int tiles = (d.d_h + kFinishCols - 1) / kFinishCols;
        const dim3 grid(d.n_h * tiles, (d.B + kFinishSeqs - 1) / kFinishSeqs);
        const FinishSlabs slabs = finish_slabs(d, (long long)grid.x * grid.y);
        const size_t smem = (size_t)(slabs.even_pieces + slabs.odd_pieces) * kDecodeThreads * sizeof(typename Weights4<T>::Raw) +
                            (2 * slabs.size * 4 + 2 * 8 * 128) * sizeof(float);
        err = launch_chained(true, decode_finish_kernel<T>, grid, kDecodeThreads, smem,
                            stream, d, tiles, slabs, (const T*)x_t, (const float*)part_o, (size_t)p.n_chunks * d.n_q * d.d_l, (const T*)w_p,
                            (const T*)w_g, (T*)out, append != nullptr ? append->seq_lens : nullptr, S_cap);
        if (err != cudaSuccess) return err;
        *launches += 2;
    }
    return cudaSuccess;
}

// ---- 8-bit caches: e4m3 codes with one fp32 scale per cached row (token and group).  Reading (the paper
//      fixes none; its Sec. 5.3 / App. C.2 only observe that decode is bound by the bytes of the cache):
//      scale = max|row| / 448 (1 for an all-zero row), code = round-to-nearest-even(x / scale), both
//      divisions in fp32; the operator runs on code * scale.
cudaError_t launch_decode_fp8(const Dims& d, int dtype, const void* q, const void* k_codes, const void* c_codes,
                              const float* k_scale, const float* c_scale, const int32_t* seq_lens, int S_cap,
                              const void* x_t, const void* w_p, const void* w_g, void* out, void* workspace, size_t room,
                              int32_t* status_word, cudaStream_t stream, int* launches) {
    if (dtype == GTA_F32)
        return launch_decode_typed<float, Fp8>(d, q, k_codes, c_codes, seq_lens, S_cap, x_t, w_p, w_g, out, workspace,
                                               room, status_word, stream, 7, launches, PageMap(), k_scale, c_scale);
    return launch_decode_typed<__nv_bfloat16, Fp8>(d, q, k_codes, c_codes, seq_lens, S_cap, x_t, w_p, w_g, out, workspace,
                                                   room, status_word, stream, 7, launches, PageMap(), k_scale, c_scale);
}

// Quantising append.  A new row (token and group) is handled by a group of lanes of one warp, eight elements per lane
// and piece: the row stays in registers between its two uses (largest magnitude, codes), is read with 16-byte loads
// and written as 8-byte pieces of codes.
//
// code = e4m3(y), y = fl(x / scale): the quotient comes from the correctly rounded reciprocal of the row's scale and
// two of Markstein's corrections (P. Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990: q' = fl(q + fl(x - q s) r) is the correctly rounded quotient when q is within one unit in the last
// place of it and r = fl(1 / s); the first correction brings fl(x r), which is within 1.5 units, there), two elements
// per instruction.  Rows whose scale is far from 1, where a residual could leave the normal numbers, divide.
// What bounds the kernel: issue slots (about 175 instructions per piece where a lane has one of a row, fewer with four), and the
// latency of a CTA's length and rows; 4 prompts of 2048 tokens (25 MB): 9.1 us.  (One or two pieces per lane 11.1, a division per
// element 13.3; one CTA per sequence with 2-byte loads, the first form, left the chip idle: 1318 us.  CTAs that stay, behind a ring
// of bulk copies: 14.7.)
__device__ __forceinline__ uint32_t f32_to_e4m3x2(float lo, float hi) {
    uint16_t r;   // the low byte of the pair is the second source operand
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
__device__ __forceinline__ uint2 f32_to_e4m3x8(const float (&y)[8]) {
    return make_uint2(f32_to_e4m3x2(y[0], y[1]) | (f32_to_e4m3x2(y[2], y[3]) << 16),
                      f32_to_e4m3x2(y[4], y[5]) | (f32_to_e4m3x2(y[6], y[7]) << 16));
}
// Eight elements as they are stored, their largest magnitude (not a number if one of them is none; of the numbers among
// them), their values, their signs.
template <typename T> struct Piece;
template <> struct Piece<float> {
    float4 a, b;
    __device__ __forceinline__ void zero() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
    __device__ __forceinline__ void load(const float* p) {
        a = __ldg(reinterpret_cast<const float4*>(p));
        b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    }
    __device__ __forceinline__ float amax() const {
        using ptx::max_nan;
        return max_nan(max_nan(max_nan(fabsf(a.x), fabsf(a.y)), max_nan(fabsf(a.z), fabsf(a.w))),
                       max_nan(max_nan(fabsf(b.x), fabsf(b.y)), max_nan(fabsf(b.z), fabsf(b.w))));
    }
    __device__ __forceinline__ float amax_of_numbers() const {
        return fmaxf(fmaxf(fmaxf(fabsf(a.x), fabsf(a.y)), fmaxf(fabsf(a.z), fabsf(a.w))),
                     fmaxf(fmaxf(fabsf(b.x), fabsf(b.y)), fmaxf(fabsf(b.z), fabsf(b.w))));
    }
    __device__ __forceinline__ void widen(float (&v)[8]) const {
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
    __device__ __forceinline__ uint2 signs() const {       // bit 7 of byte j of the pair: the sign of element j
        const auto pack = [](const float4& f) {
            const uint32_t lo = ptx::byte_perm(__float_as_uint(f.x), __float_as_uint(f.y), 0x0073u);
            const uint32_t hi = ptx::byte_perm(__float_as_uint(f.z), __float_as_uint(f.w), 0x7300u);
            return ptx::byte_perm(lo, hi, 0x7610u) & 0x80808080u;
        };
        return make_uint2(pack(a), pack(b));
    }
};
template <> struct Piece<__nv_bfloat16> {
    uint4 a;
    __device__ __forceinline__ void zero() { a = make_uint4(0u, 0u, 0u, 0u); }
    __device__ __forceinline__ void load(const __nv_bfloat16* p) { a = __ldg(reinterpret_cast<const uint4*>(p)); }
    __device__ __forceinline__ float amax() const {        // two magnitudes per instruction
        const auto h = [](uint32_t w) { return __habs2(*reinterpret_cast<const __nv_bfloat162*>(&w)); };
        const __nv_bfloat162 m = __hmax2_nan(__hmax2_nan(h(a.x), h(a.y)), __hmax2_nan(h(a.z), h(a.w)));
        return ptx::max_nan(__low2float(m), __high2float(m));
    }
    __device__ __forceinline__ float amax_of_numbers() const {
        float v[8], m = 0.f;
        widen(v);
#pragma unroll
        for (int j = 0; j < 8; ++j) m = fmaxf(m, fabsf(v[j]));
        return m;
    }
    __device__ __forceinline__ void widen(float (&v)[8]) const { Vec16<__nv_bfloat16>::widen(a, v); }
    __device__ __forceinline__ uint2 signs() const {
        return make_uint2(ptx::byte_perm(a.x, a.y, 0x7531u) & 0x80808080u, ptx::byte_perm(a.z, a.w, 0x7531u) & 0x80808080u);
    }
};

// The codes of a piece by division (out of line: the rare rows).
template <typename T>
__device__ __noinline__ uint2 codes_by_division(Piece<T> p, float scale) {
    float v[8];
    p.widen(v);
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = __fdiv_rn(v[j], scale);
    return f32_to_e4m3x8(v);
}

// The largest magnitude of the numbers of a row.
template <typename T, int NV>
__device__ __forceinline__ float largest_number(const Piece<T> (&p)[NV], int lpr) {
    float amax = p[0].amax_of_numbers();
#pragma unroll
    for (int i = 1; i < NV; ++i) amax = fmaxf(amax, p[i].amax_of_numbers());
    for (int o = lpr >> 1; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    return amax;
}

// Row of `width` (a multiple of 8, at most 8 lpr NV) elements on `lpr` lanes (a power of two; `sl` is this lane's
// place among them, `live` false on the lanes of a row that is not there).
template <typename T, int NV>
__device__ __forceinline__ void load_row(Piece<T> (&p)[NV], const T* __restrict__ src, int width, int lpr, int sl, bool live) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int e = (sl + i * lpr) * 8;
        p[i].zero();
        if (live && e < width) p[i].load(src + e);
    }
}
template <typename T, int NV>
__device__ __forceinline__ void quantise_row(const Piece<T> (&p)[NV], uint8_t* __restrict__ dst,
                                             float* __restrict__ scale_out, int width, int lpr, int sl, bool live) {
    float amax = p[0].amax();
#pragma unroll
    for (int i = 1; i < NV; ++i) amax = ptx::max_nan(amax, p[i].amax());
    for (int o = lpr >> 1; o > 0; o >>= 1) amax = ptx::max_nan(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    // a row with elements that are no numbers: its scale is that of the others, and it is divided (the code of such an element
    // has no sign)
    const bool numbers = amax == amax;
    if (__any_sync(0xffffffffu, !numbers)) amax = largest_number<T, NV>(p, lpr);
    const float scale = amax > 0.f ? __fdiv_rn(amax, 448.f) : 1.f;
    if (!live) return;
    const bool plain = numbers && scale > 8.7e-19f && scale < 1.2e18f;      // 2^-60, 2^60
    const float inv = __frcp_rn(scale);
    const uint64_t inv2 = ptx::f32x2(inv, inv), neg2 = ptx::f32x2(-scale, -scale);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int e = (sl + i * lpr) * 8;
        if (e < width) {
            uint2 w;
            if (plain) {
                float v[8], y[8];
                p[i].widen(v);
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    const uint64_t x = ptx::f32x2(v[j], v[j + 1]);
                    uint64_t y2 = ptx::mul2(x, inv2);
                    y2 = ptx::fma2(ptx::fma2(y2, neg2, x), inv2, y2);
                    y2 = ptx::fma2(ptx::fma2(y2, neg2, x), inv2, y2);
                    ptx::f32x2_split(y2, y[j], y[j + 1]);
                }
                w = f32_to_e4m3x8(y);
                const uint2 sign = p[i].signs();        // (the corrections turn -0 into +0)
                w = make_uint2(w.x | sign.x, w.y | sign.y);
            } else {
                w = codes_by_division(p[i], scale);
            }
            *reinterpret_cast<uint2*>(dst + e) = w;
        }
    }
    if (sl == 0) *scale_out = scale;
}

struct AppendFp8Args {
    uint8_t *k_codes, *c_codes;
    float *k_scale, *c_scale;
    const void *k_new, *c_new;    // [B][groups][n_new][width]
    int n_k, n_c, d_h, d_l, S_cap, n_new;
    int k_lpr, c_lpr;             // lanes per key / latent row (powers of two)
};

// Warps `first`, `first + step`, ... of the work of sequence b: 32 / lpr neighbouring rows each, keys then latents.
template <typename T, int NV>
__device__ __forceinline__ void append_fp8_rows(const AppendFp8Args& a, int b, int len, int first, int step) {
    const int lane = threadIdx.x & 31;
    const int k_per = 32 / a.k_lpr, c_per = 32 / a.c_lpr;
    const int k_rows = a.n_k * a.n_new, c_rows = a.n_c * a.n_new;
    const int k_units = (k_rows + k_per - 1) / k_per, units = k_units + (c_rows + c_per - 1) / c_per;
    for (int u = first; u < units; u += step) {
        if (u < k_units) {
            const int r = u * k_per + lane / a.k_lpr, g = r / a.n_new, n = r - g * a.n_new, sl = lane & (a.k_lpr - 1);
            const size_t row = ((size_t)b * a.n_k + g) * a.S_cap + len + n;
            Piece<T> p[1];
            load_row<T, 1>(p, static_cast<const T*>(a.k_new) + ((size_t)b * k_rows + r) * a.d_h, a.d_h, a.k_lpr, sl, r < k_rows);
            quantise_row<T, 1>(p, a.k_codes + row * a.d_h, a.k_scale + row, a.d_h, a.k_lpr, sl, r < k_rows);
        } else {
            const int r = (u - k_units) * c_per + lane / a.c_lpr, g = r / a.n_new, n = r - g * a.n_new, sl = lane & (a.c_lpr - 1);
            const size_t row = ((size_t)b * a.n_c + g) * a.S_cap + len + n;
            Piece<T> p[NV];
            load_row<T, NV>(p, static_cast<const T*>(a.c_new) + ((size_t)b * c_rows + r) * a.d_l, a.d_l, a.c_lpr, sl, r < c_rows);
            quantise_row<T, NV>(p, a.c_codes + row * a.d_l, a.c_scale + row, a.d_l, a.c_lpr, sl, r < c_rows);
        }
    }
}

// One CTA per sequence (few new rows, e.g. one decode step): quantise, then advance the length.
template <typename T, int NV>
__global__ void __launch_bounds__(256)
append_fp8_small_kernel(AppendFp8Args a, int32_t* __restrict__ seq_lens, int32_t* status_word) {
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int b = blockIdx.x;
    const int len = seq_lens[b];
    __syncthreads();   // every thread has read the old length before thread 0 rewrites it
    if (len < 0 || (long long)len + a.n_new > a.S_cap) {
        if (threadIdx.x == 0) raise_status(status_word, GTA_ERR_CACHE_FULL);
        return;
    }
    if (threadIdx.x == 0) seq_lens[b] = len + a.n_new;
    append_fp8_rows<T, NV>(a, b, len, threadIdx.x >> 5, 8);
}

// Rows [n0, n0 + U 32 / lpr) of one group of one sequence, the loads of all of them ahead of the first use.
template <typename T, int NV, int U>
__device__ __forceinline__ void append_fp8_plane(const T* __restrict__ src, uint8_t* __restrict__ dst,
                                                 float* __restrict__ scales, int n_new, int width, int lpr, int n0) {
    const int lane = threadIdx.x & 31, per = 32 / lpr, sl = lane & (lpr - 1);
    Piece<T> p[U][NV];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int n = n0 + u * per + lane / lpr;
        load_row<T, NV>(p[u], src + (size_t)n * width, width, lpr, sl, n < n_new);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int n = n0 + u * per + lane / lpr;
        if (n0 + u * per < n_new)
            quantise_row<T, NV>(p[u], dst + (size_t)n * width, scales + n, width, lpr, sl, n < n_new);
    }
}

// Many new rows (a prompt): grid (n_k k_parts + n_c c_parts, B) quantises, the lengths advance in the launch behind it.
// A warp takes two key rows (times 32 / lpr) or one latent row at once: with more in flight the registers cost CTAs.
__host__ __device__ constexpr int append_fp8_rows_at_once(int nv) { return nv < 2 ? 2 : 1; }
template <typename T, int NK, int NV>
__global__ void __launch_bounds__(256)
append_fp8_bulk_kernel(AppendFp8Args a, const int32_t* __restrict__ seq_lens, int k_parts, int c_parts) {
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int b = blockIdx.y, warp = threadIdx.x >> 5;
    const int len = seq_lens[b];
    if (len < 0 || (long long)len + a.n_new > a.S_cap) return;
    const int k_blocks = a.n_k * k_parts;
    if ((int)blockIdx.x < k_blocks) {
        constexpr int U = append_fp8_rows_at_once(NK);
        const int g = blockIdx.x / k_parts, part = blockIdx.x - g * k_parts;
        const size_t plane = (size_t)b * a.n_k + g, row = plane * a.S_cap + len;
        append_fp8_plane<T, NK, U>(static_cast<const T*>(a.k_new) + plane * a.n_new * a.d_h, a.k_codes + row * a.d_h,
                                  a.k_scale + row, a.n_new, a.d_h, a.k_lpr, (part * 8 + warp) * U * (32 / a.k_lpr));
    } else {
        constexpr int U = append_fp8_rows_at_once(NV);
        const int g = (blockIdx.x - k_blocks) / c_parts, part = blockIdx.x - k_blocks - g * c_parts;
        const size_t plane = (size_t)b * a.n_c + g, row = plane * a.S_cap + len;
        append_fp8_plane<T, NV, U>(static_cast<const T*>(a.c_new) + plane * a.n_new * a.d_l, a.c_codes + row * a.d_l,
                                   a.c_scale + row, a.n_new, a.d_l, a.c_lpr, (part * 8 + warp) * U * (32 / a.c_lpr));
    }
}

// Turns of a warp over the new rows of a sequence, with the lanes that `a` gives a row.  One CTA per sequence takes up to four turns
// per warp (its 2 - 3 us are launch and latency); beyond that the launch behind, about 2 us, is the smaller part.
static bool append_fp8_one_cta(const AppendFp8Args& a) {
    const int k_per = 32 / a.k_lpr, c_per = 32 / a.c_lpr;
    return ((long long)a.n_k * a.n_new + k_per - 1) / k_per + ((long long)a.n_c * a.n_new + c_per - 1) / c_per <= 32;
}

template <typename T, int NK, int NV>
static cudaError_t launch_append_fp8(const AppendFp8Args& a, int B, int32_t* seq_lens, int32_t* status_word,
                                     cudaStream_t stream, int* launches) {
    const int k_per = 32 / a.k_lpr, c_per = 32 / a.c_lpr;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (NK == 1 && append_fp8_one_cta(a)) {
        cfg.gridDim = dim3(B);
        *launches += 1;
        return cudaLaunchKernelEx(&cfg, append_fp8_small_kernel<T, NV>, a, seq_lens, status_word);
    }
    const auto parts = [&](int per, int nv) {
        const int rows = 8 * per * append_fp8_rows_at_once(nv);
        return (a.n_new + rows - 1) / rows;
    };
    const int k_parts = parts(k_per, NK), c_parts = parts(c_per, NV);
    cfg.gridDim = dim3(a.n_k * k_parts + a.n_c * c_parts, B);
    cudaError_t err = cudaLaunchKernelEx(&cfg, append_fp8_bulk_kernel<T, NK, NV>, a, (const int32_t*)seq_lens, k_parts, c_parts);
    if (err != cudaSuccess) return err;
    *launches += 2;
    return launch_append_advance(B, a.S_cap, a.n_new, seq_lens, status_word, stream);
}

// Lanes of a row of `width` elements with up to `pieces` pieces each (d_h <= 256; latent rows up to 8 pieces a lane).
static int append_fp8_lanes(int width, int pieces) {
    int n = 1;
    while (n < 32 && n * 8 * pieces < width) n *= 2;
    return n;
}

template <typename T>
static cudaError_t launch_append_fp8_typed(AppendFp8Args a, int B, int32_t* seq_lens, int32_t* status_word,
                                           cudaStream_t stream, int* launches) {
    // Long prompts: four pieces per lane, so that what a row costs whatever its width -- its largest element among the lanes, its
    // scale, the reciprocal, addresses -- is spent on fewer lanes of more elements (us, one piece of a key row and up to four of a
    // latent row per lane / four of both: 25 MB 11.1 / 9.1, 101 MB 33.0 / 24.4, 202 MB with rows of 1024 53.5 / 43.9, 10 MB of the 1B
    // layer 6.7 / 5.5; 6 MB 5.3 / 5.3, 2 MB 4.6 / 4.8).  Few rows of many sequences leave such lanes idle: they stay as they are (1000
    // sequences, 10 rows of 2048 elements: 28.3 / 30.4), or with one CTA each where that takes them (4096 sequences, a token of
    // 2048 elements: 18.0 / 103.5).
    const long long elements = (long long)B * a.n_new * (a.n_k * a.d_h + a.n_c * a.d_l);
    if (elements >= 3 << 20 && a.d_l <= 1024 && a.n_new >= 16 && !append_fp8_one_cta(a)) {
        a.k_lpr = append_fp8_lanes(a.d_h, 4);
        a.c_lpr = append_fp8_lanes(a.d_l, 4);
        return launch_append_fp8<T, 4, 4>(a, B, seq_lens, status_word, stream, launches);
    }
    const int nv = (a.d_l / 8 + a.c_lpr - 1) / a.c_lpr;     // 8-element pieces per lane of a latent row
    if (nv <= 1) return launch_append_fp8<T, 1, 1>(a, B, seq_lens, status_word, stream, launches);
    if (nv <= 2) return launch_append_fp8<T, 1, 2>(a, B, seq_lens, status_word, stream, launches);
    if (nv <= 4) return launch_append_fp8<T, 1, 4>(a, B, seq_lens, status_word, stream, launches);
    return launch_append_fp8<T, 1, 8>(a, B, seq_lens, status_word, stream, launches);
}

cudaError_t launch_cache_append_fp8(const Dims& d, int dtype, void* k_codes, void* c_codes, float* k_scale,
                                    float* c_scale, int S_cap, const void* k_new, const void* c_new, int n_new,
                                    int32_t* seq_lens, int32_t* status_word, cudaStream_t stream, int* launches) {
    AppendFp8Args a;
    a.k_codes = (uint8_t*)k_codes; a.c_codes = (uint8_t*)c_codes;
    a.k_scale = k_scale; a.c_scale = c_scale;
    a.k_new = k_new; a.c_new = c_new;
    a.n_k = d.n_k; a.n_c = d.n_c; a.d_h = d.d_h; a.d_l = d.d_l; a.S_cap = S_cap; a.n_new = n_new;
    a.k_lpr = append_fp8_lanes(d.d_h, 1);
    a.c_lpr = append_fp8_lanes(d.d_l, 1);
    if (dtype == GTA_F32) return launch_append_fp8_typed<float>(a, d.B, seq_lens, status_word, stream, launches);
    return launch_append_fp8_typed<__nv_bfloat16>(a, d.B, seq_lens, status_word, stream, launches);
}

size_t decode_plain_workspace_bytes(const Dims& d, int S_cap) { return plan_bound(d, S_cap); }
size_t decode_plain_least_workspace(const Dims& d, int S_cap) { return least_plan(d, S_cap).total; }

// The plain-ALU kernels whatever the shape: they read the caches with ordinary 16-byte loads, which is what a cache
// in page-locked host memory (reached over the host link) needs; the TMA path is kept to device memory.
cudaError_t launch_decode_plain(const Dims& d, int dtype, const void* q, const void* k_cache, const void* c_cache,
                                const int32_t* seq_lens, int S_cap, const void* x_t, const void* w_p,
                                const void* w_g, void* out, void* workspace, size_t room, int32_t* status_word,
                                cudaStream_t stream, int* launches) {
    if (dtype == GTA_F32)
        return launch_decode_typed<float, float>(d, q, k_cache, c_cache, seq_lens, S_cap, x_t, w_p, w_g, out,
                                                workspace, room, status_word, stream, 7, launches, PageMap());
    return launch_decode_typed<__nv_bfloat16, __nv_bfloat16>(d, q, k_cache, c_cache, seq_lens, S_cap, x_t, w_p, w_g, out,
                                                    workspace, room, status_word, stream, 7, launches, PageMap());
}

cudaError_t launch_decode(const Dims& d, int dtype, const void* q, const void* k_cache, const void* c_cache,
                          const int32_t* seq_lens, int S_cap, const void* x_t, const void* w_p,
                          const void* w_g, void* out, void* workspace, size_t room, int32_t* status_word,
                          cudaStream_t stream, int stages, int* launches, const PageMap& pm) {
    const int page_size = pm.table ? pm.page_size : 0;
    if (decode_fast_supported(d, dtype, page_size) && S_cap > 0 && room >= decode_fast_workspace_bytes(d, page_size))
        return launch_decode_fast(d, q, k_cache, c_cache, seq_lens, S_cap, x_t, w_p, w_g, out, workspace,
                                  status_word, stream, stages, launches, pm);
    if (dtype == GTA_F32)
        return launch_decode_typed<float, float>(d, q, k_cache, c_cache, seq_lens, S_cap, x_t, w_p, w_g, out,
                                          workspace, room, status_word, stream, stages, launches, pm);
    return launch_decode_typed<__nv_bfloat16, __nv_bfloat16>(d, q, k_cache, c_cache, seq_lens, S_cap, x_t, w_p, w_g, out,
                                              workspace, room, status_word, stream, stages, launches, pm);
}

// The step with the append of its token folded in (contiguous caches): no kernel of its own in front.
cudaError_t launch_decode_plain_append(const Dims& d, int dtype, const void* q, void* k_cache, void* c_cache, const void* k_new,
                                       const void* c_new, int32_t* seq_lens, int S_cap, const void* x_t, const void* w_p,
                                       const void* w_g, void* out, void* workspace, size_t room, int32_t* status_word,
                                       cudaStream_t stream, int* launches) {
    const StepAppend append = {k_new, c_new, k_cache, c_cache, seq_lens};
    if (dtype == GTA_F32)
        return launch_decode_typed<float, float>(d, q, k_cache, c_cache, seq_lens, S_cap, x_t, w_p, w_g, out, workspace, room,
                                                 status_word, stream, 7, launches, PageMap(), nullptr, nullptr, &append);
    return launch_decode_typed<__nv_bfloat16, __nv_bfloat16>(d, q, k_cache, c_cache, seq_lens, S_cap, x_t, w_p, w_g, out, workspace,
                                                             room, status_word, stream, 7, launches, PageMap(), nullptr, nullptr,
                                                             &append);
}

}  // namespace gta
