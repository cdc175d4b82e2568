// Plain-ALU (fp32 FMA) prefill kernels: any supported shape, fp32 or bf16 storage.
// They carry small fp32 calls (larger ones run on the tensor cores in bf16 pieces, f32_plan below) and every shape
// the tcgen05 kernels do not cover.  Two kernels, and one (short_prefill_f32_kernel) that does the work of both for a short
// fp32 prompt:
//   generic_attention_kernel : shared attention map per query group, online softmax, latent
//                              P·C  ->  normalised L[n_q, B, N, d_l] (fp32, workspace)
//   generic_decoder_kernel   : out_i = (L_{q(i)} W_P,i) (.) sigmoid(X W_G,i)
// (Sec. 3.3 reformulated equation; causal sum of App. B.1.1.)
//
// Both are bound by the fp32 FMA pipe (72 TFLOP/s over 148 SMs at 1.9 GHz) where there is enough work, by latency
// where there is not.  All products are two-wide fp32 instructions (one issue slot for two results; the pipe's rate
// is the same), operands come from shared memory in 16-byte pieces that several lanes share, and tiles are brought
// in by cp.async while the tiles before them are multiplied.
#include <type_traits>

#include "gta_common.cuh"
#include "gta_sm100.cuh"
#include "sm100_ptx.cuh"

namespace gta {

__device__ __forceinline__ void cp_async_16(void* dst, const void* src, bool live) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_addr(dst)), "l"(src), "r"(live ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Four elements of storage type T at `src` -> four floats at `dst` in shared memory; zeros where !live (src is then
// not read).  fp32 travels asynchronously, bf16 is widened on the way.
__device__ __forceinline__ void stage4(float* dst, const float* src, bool live) { cp_async_16(dst, src, live); }
__device__ __forceinline__ void stage4(float* dst, const __nv_bfloat16* src, bool live) {
    uint2 r = make_uint2(0u, 0u);
    if (live) r = __ldg(reinterpret_cast<const uint2*>(src));
    *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u),
                                                  __uint_as_float(r.y << 16), __uint_as_float(r.y & 0xffff0000u));
}

__device__ __forceinline__ void store4(float* dst, const float (&v)[4]) {
    *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(__nv_bfloat16* dst, const float (&v)[4]) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b = __floats2bfloat162_rn(v[2], v[3]);
    *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

// 16 bytes of shared memory as two pairs of floats
struct Pair2 { uint64_t lo, hi; };
__device__ __forceinline__ Pair2 lds_pair2(const float* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ float pair_sum(uint64_t v) {
    float a, b;
    ptx::f32x2_split(v, a, b);
    return a + b;
}

// ---------------------------------------------------------------------------------------------
// Attention.  A warp owns 16 query rows and works on tiles of 32 keys, by itself between the CTA's tile barriers:
//   scores  4 rows x 4 keys per lane; rows and keys lie d-contiguous in shared memory (rows padded by 4 floats), so a
//           pair is two neighbouring elements of the contraction and its halves are added at the end;
//   P^T     goes to a buffer of the warp's own ([key][16 rows]), from where
//   sums    8 rows x 4 NC columns per lane take it (a pair is two neighbouring latent columns).
// QW warps of the CTA share a key tile on rows of their own; SW groups of them take every SW-th key tile and are merged
// by log-sum-exp at the end: more key groups shorten the longest rows' chain, for calls whose CTAs would leave SMs idle.
// CTAs take d_l in slices of 64 NC columns (the scores are recomputed per slice).  One buffer per operand: the key tile is
// fetched while the sums of the tile before are taken, the latent tile under the scores; with two buffers of each, one
// CTA of four warps filled an SM's shared memory and a scheduler had a single warp (2 x 1500 tokens of the 1B layer: 282
// us; 212 with three CTAs per SM).
constexpr int kAttnKeys = 32, kPStride = 20;

struct AttnSmem {
    int q_stride, k_floats, c_floats, total_floats;
};
__host__ __device__ inline AttnSmem attn_smem(int d_h, int rows, int tile_keys, int cols, int warps) {
    AttnSmem s;
    s.q_stride = d_h + 4;
    s.k_floats = tile_keys * s.q_stride;
    s.c_floats = tile_keys * cols;
    s.total_floats = rows * s.q_stride + s.k_floats + s.c_floats + tile_keys + warps * (kAttnKeys * kPStride + 32);
    return s;
}

// DH: the head width where it is a compile-time constant, 0 otherwise.  Rows t0 .. of map g of sequence b, latent columns col0 ..;
// `tid` of the 32 QW SW threads, which `sync` brings together; put(row, float4 column, v) takes the normalised sums.
// bulk != nullptr (fp32, contiguous caches, d_l = 64 NC): a latent tile is one bulk copy, counted on the barrier there.  `armed`: how
// many copies thread 0 has asked for; none once a wait has given up, behind which the copy before may still be on its way.
struct BulkLatents { uint64_t* bar; volatile int* abort_flag; int armed; };
// Test hook of the bounded waits of short_prefill_f32_kernel (gta_debug_attention_wait): their time limit, and a switch that keeps
// the first latents back.
struct ShortWait { unsigned long long limit_ns; int withhold; };
static __constant__ ShortWait c_short_wait = {ptx::kWaitLimitNs, 0};
template <typename T, int QW, int SW, int NC, int DH, typename Sync, typename Put>
__device__ __forceinline__ void attention_tile(BulkLatents* bulk, const Dims& d, const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ c,
                                               const PageMap& pm, int32_t* status_word, float* smem, int tid, int t0, int col0, int g,
                                               int b, Sync sync, Put put) {
    constexpr int kWarps = QW * SW, kThreads = 32 * kWarps;
    constexpr int kRows = 16 * QW, kTile = kAttnKeys * SW, kCols = 64 * NC;
    const int d_h = DH > 0 ? DH : d.d_h;
    const AttnSmem L = attn_smem(d_h, kRows, kTile, kCols, kWarps);
    const int ld = d_h + 4;
    float* q_s = smem;                                          // [kRows][ld]
    float* k_s = q_s + kRows * ld;                              // [kTile][ld]
    float* c_s = k_s + L.k_floats;                              // [kTile][kCols]
    int* bad_s = reinterpret_cast<int*>(c_s + L.c_floats);      // [kTile]: key on a page outside the pool
    const int warp = tid >> 5, lane = tid & 31;
    float* p_s = reinterpret_cast<float*>(bad_s + kTile) + warp * kAttnKeys * kPStride;   // [32][kPStride]
    float* row_s = reinterpret_cast<float*>(bad_s + kTile) + kWarps * kAttnKeys * kPStride + warp * 32;   // [2][16]
    const int qw = warp % QW, sw = warp / QW;

    const int kg = d.q_to_k(g), cg = d.q_to_c(g);
    const int n_cols = min(kCols, d.d_l - col0);
    const int off = d.causal ? d.Nk - d.N : 0;                  // causal: row t attends keys 0 .. t + off
    const int rows = min(kRows, d.N - t0);
    const int n_keys = d.causal ? min(t0 + rows + off, d.Nk) : d.Nk;
    const int n_iter = (n_keys + kTile - 1) / kTile;

    // lanes that share a row when a tile is brought in (powers of two)
    const int h_vecs = d_h >> 2, c_vecs = n_cols >> 2;
    int h_sh = 1, c_sh = 1;
    while (h_sh < 5 && (1 << h_sh) < h_vecs) ++h_sh;
    while (c_sh < 5 && (1 << c_sh) < c_vecs) ++c_sh;

    const int h_row = tid >> h_sh, h_vec = tid & ((1 << h_sh) - 1), h_step = kThreads >> h_sh;
    const int c_row = tid >> c_sh, c_vec = tid & ((1 << c_sh) - 1), c_step = kThreads >> c_sh;
    const T* k_plane = k + ((size_t)b * d.n_k + kg) * d.S * d_h;            // (contiguous caches)
    const T* c_plane = c + ((size_t)b * d.n_c + cg) * d.S * d.d_l + col0;

    auto load_keys = [&](int it) {
        const int j0 = it * kTile;
        if (pm.table == nullptr) {
            const T* src = k_plane + (size_t)(j0 + h_row) * d_h;
            for (int r = h_row; r < kTile; r += h_step, src += (size_t)h_step * d_h)
                if (j0 + r < n_keys)
                    for (int v = h_vec; v < h_vecs; v += 1 << h_sh) stage4(k_s + r * ld + 4 * v, src + 4 * v, true);
            return;
        }
        for (int r = h_row; r < kTile; r += h_step) {
            const long long idx = j0 + r < n_keys ? cache_row(pm, b, d.n_k, kg, d.S, j0 + r, status_word) : -1;
            if (h_vec == 0) bad_s[r] = idx < 0;
            if (idx >= 0)
                for (int v = h_vec; v < h_vecs; v += 1 << h_sh)
                    stage4(k_s + r * ld + 4 * v, k + (size_t)idx * d_h + 4 * v, true);
        }
    };
    auto load_latents = [&](int it) {       // (a row that does not exist meets zero probabilities: it is cleared)
        const int j0 = it * kTile;
        if (bulk != nullptr) {
            const int n = min(kTile, n_keys - j0);
            if (tid == 0 && *bulk->abort_flag == 0 && !(it == 0 && c_short_wait.withhold != 0)) {
                ++bulk->armed;
                ptx::fence_proxy_async_smem();           // (the memory has been read by ordinary loads)
                ptx::mbar_arrive_expect_tx(bulk->bar, (uint32_t)(n * kCols * 4));
                ptx::bulk_load_1d(c_s, c_plane + (size_t)j0 * kCols, (uint32_t)(n * kCols * 4), bulk->bar);
            }
            for (int i = tid; i < (kTile - n) * kCols / 4; i += kThreads)
                reinterpret_cast<float4*>(c_s + n * kCols)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            return;
        }
        if (pm.table == nullptr) {
            const T* src = c_plane + (size_t)(j0 + c_row) * d.d_l;
            for (int r = c_row; r < kTile; r += c_step, src += (size_t)c_step * d.d_l) {
                const bool live = j0 + r < n_keys;
                for (int v = c_vec; v < c_vecs; v += 1 << c_sh) stage4(c_s + r * kCols + 4 * v, live ? src + 4 * v : c_plane, live);
            }
            return;
        }
        for (int r = c_row; r < kTile; r += c_step) {
            const long long idx = j0 + r < n_keys ? cache_row(pm, b, d.n_c, cg, d.S, j0 + r, status_word) : -1;
            const T* src = c + (size_t)(idx < 0 ? 0 : idx) * d.d_l + col0;
            for (int v = c_vec; v < c_vecs; v += 1 << c_sh) stage4(c_s + r * kCols + 4 * v, src + 4 * v, idx >= 0);
        }
    };

    if (bulk != nullptr && n_iter > 0) load_latents(0);
    {
        const T* q_rows = q + (((size_t)b * d.n_q + g) * d.N + t0) * d_h;
        for (int r = h_row; r < kRows; r += h_step)
            for (int v = h_vec; v < h_vecs; v += 1 << h_sh)
                stage4(q_s + r * ld + 4 * v, q_rows + (size_t)(r < rows ? r : 0) * d_h + 4 * v, r < rows);
    }
    if (n_iter > 0) load_keys(0);
    cp_async_commit();

    const int rg = lane >> 3, kc = lane & 7;       // scores: rows 4 rg + i, keys kc + 8 j
    const int rh = lane >> 4, cc = lane & 15;      // sums: rows 8 rh + i, columns 4 cc + 64 n
    const float scale2 = d.scale * 1.4426950408889634f;      // scores, maxima in powers of two
    float m[4], l[4];
    uint64_t o[8][NC][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) { m[i] = -INFINITY; l[i] = 0.f; }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int n = 0; n < NC; ++n) o[i][n][0] = o[i][n][1] = 0ull;
    const int row0 = t0 + 16 * qw;                 // first row of this warp
    const int warp_keys = row0 >= d.N ? 0 : (d.causal ? min(min(row0 + 16, d.N) + off, d.Nk) : d.Nk);

    for (int it = 0; it < n_iter; ++it) {
        cp_async_wait<0>();
        sync();                 // the key tile is there, the latent tile before has been used
        if (bulk == nullptr || it > 0) load_latents(it);
        cp_async_commit();
        const int j0 = it * kTile + sw * kAttnKeys;
        const bool mine = j0 < warp_keys;
        if (mine) {
            const float* ks = k_s + sw * kAttnKeys * ld;
            const int* bad = bad_s + sw * kAttnKeys;
            uint64_t s2[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) s2[i][j] = 0ull;
            const float* qa = q_s + (16 * qw + 4 * rg) * ld;
            const float* kb = ks + kc * ld;
#pragma unroll(DH > 0 ? DH / 4 : 2)
            for (int e = 0; e < d_h; e += 4) {
                Pair2 a[4], bb[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i] = lds_pair2(qa + i * ld + e);
#pragma unroll
                for (int j = 0; j < 4; ++j) bb[j] = lds_pair2(kb + 8 * j * ld + e);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        s2[i][j] = ptx::fma2(a[i].lo, bb[j].lo, s2[i][j]);
                        s2[i][j] = ptx::fma2(a[i].hi, bb[j].hi, s2[i][j]);
                    }
            }
            const bool edge = j0 + kAttnKeys > (d.causal ? row0 + off + 1 : d.Nk) || pm.table != nullptr;
            float p[4][4], alpha[4];
            bool raised = false;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int live = d.causal ? min(row0 + 4 * rg + i + off + 1, d.Nk) : d.Nk;     // keys of this row
                float mt = -INFINITY;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    p[i][j] = pair_sum(s2[i][j]) * scale2;
                    if (edge && (j0 + kc + 8 * j >= live || (pm.table != nullptr && bad[kc + 8 * j]))) p[i][j] = -INFINITY;
                    mt = fmaxf(mt, p[i][j]);
                }
#pragma unroll
                for (int x = 1; x < 8; x <<= 1) mt = fmaxf(mt, __shfl_xor_sync(0xffffffffu, mt, x));
                const float m_new = fmaxf(m[i], mt);
                const float ref = m_new == -INFINITY ? 0.f : m_new;       // (nothing but masked keys so far)
                alpha[i] = m_new == m[i] ? 1.f : exp2f(m[i] - ref);       // 2^-inf = 0 on the first tile
                raised |= m_new != m[i];
                m[i] = m_new;
                float sum = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    p[i][j] = exp2f(p[i][j] - ref);
                    sum += p[i][j];
                }
                l[i] = l[i] * alpha[i] + sum;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                *reinterpret_cast<float4*>(p_s + (kc + 8 * j) * kPStride + 4 * rg) = make_float4(p[0][j], p[1][j], p[2][j], p[3][j]);
            if (kc == 0) *reinterpret_cast<float4*>(row_s + 4 * rg) = make_float4(alpha[0], alpha[1], alpha[2], alpha[3]);
            const bool rescale = __any_sync(0xffffffffu, raised);
            __syncwarp();
            if (rescale) {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float al = row_s[8 * rh + i];
                    const uint64_t al2 = ptx::f32x2(al, al);
#pragma unroll
                    for (int n = 0; n < NC; ++n) {
                        o[i][n][0] = ptx::mul2(o[i][n][0], al2);
                        o[i][n][1] = ptx::mul2(o[i][n][1], al2);
                    }
                }
            }
        }
        if (bulk != nullptr) ptx::mbar_wait_sleep(bulk->bar, it & 1, bulk->abort_flag, 0, c_short_wait.limit_ns);
        cp_async_wait<0>();
        sync();                 // the latent tile is there, the key tile has been used
        if (it + 1 < n_iter) load_keys(it + 1);
        cp_async_commit();
        if (mine) {
            const float* cs = c_s + sw * kAttnKeys * kCols;
            // The probabilities of keys past the end are zero and their latent rows cleared.  On the diagonal some rows do not see
            // some keys, whose latents may be infinite or not a number (0 x NaN): where the tile holds such a one, the rows leave
            // the keys out that they do not see.  (Leaving them out always cost 128 tokens of the tiny layer 1.8 us of 16.5.)
            const auto add_key = [&](int j, int first_row) {
                const float4 pa = *reinterpret_cast<const float4*>(p_s + j * kPStride + 8 * rh);
                const float4 pb = *reinterpret_cast<const float4*>(p_s + j * kPStride + 8 * rh + 4);
                const float pr[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
                Pair2 cv[NC];
#pragma unroll
                for (int n = 0; n < NC; ++n) cv[n] = lds_pair2(cs + j * kCols + 4 * cc + 64 * n);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (i < first_row) continue;
                    const uint64_t pp = ptx::f32x2(pr[i], pr[i]);
#pragma unroll
                    for (int n = 0; n < NC; ++n) {
                        o[i][n][0] = ptx::fma2(pp, cv[n].lo, o[i][n][0]);
                        o[i][n][1] = ptx::fma2(pp, cv[n].hi, o[i][n][1]);
                    }
                }
            };
            const int seen = d.causal ? row0 + off + 1 - j0 : kAttnKeys;      // keys of the tile that all rows see
            float odd = 0.f;
#pragma unroll 2
            for (int j = max(seen, 0) + rh; j < kAttnKeys; j += 2)
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    const float4 v = *reinterpret_cast<const float4*>(cs + j * kCols + 4 * cc + 64 * n);
                    odd = fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, fmaf(v.w, 0.f, odd))));
                }
            if (__any_sync(0xffffffffu, odd != 0.f)) {
#pragma unroll 1
                for (int j = 0; j < kAttnKeys; ++j) add_key(j, j + 1 - seen - 8 * rh);
            } else {
#pragma unroll 4
                for (int j = 0; j < kAttnKeys; ++j) add_key(j, 0);
            }
            __syncwarp();
        }
    }
    sync();                     // (the tiles' memory is used again below)

    // ---- row sums over the lanes of a row, then (maximum, row sum) in the lanes that hold the row's sums
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int x = 1; x < 8; x <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], x);
    if (kc == 0) {
        *reinterpret_cast<float4*>(row_s + 4 * rg) = make_float4(m[0], m[1], m[2], m[3]);
        *reinterpret_cast<float4*>(row_s + 16 + 4 * rg) = make_float4(l[0], l[1], l[2], l[3]);
    }
    // log-sum-exp merge of the SW key splits of every row: the key tiles' memory takes the sums
    float* o_s = k_s;                                                   // [SW][kRows][kCols]
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int n = 0; n < NC; ++n) {
            float4 v;
            ptx::f32x2_split(o[i][n][0], v.x, v.y);
            ptx::f32x2_split(o[i][n][1], v.z, v.w);
            *reinterpret_cast<float4*>(o_s + ((size_t)sw * kRows + 16 * qw + 8 * rh + i) * kCols + 4 * cc + 64 * n) = v;
        }
    sync();
    const float* all_rows = row_s - warp * 32;                          // [warp][2][16]
    for (int idx = tid; idx < rows * 16 * NC; idx += kThreads) {
        const int r = idx / (16 * NC), v4 = idx % (16 * NC);
        if (4 * v4 >= n_cols) continue;
        float mx = -INFINITY;
#pragma unroll
        for (int s = 0; s < SW; ++s) mx = fmaxf(mx, all_rows[(s * QW + (r >> 4)) * 32 + (r & 15)]);
        float ls = 0.f;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < SW; ++s) {
            const float* rs = all_rows + (s * QW + (r >> 4)) * 32 + (r & 15);
            const float w = rs[0] == -INFINITY ? 0.f : exp2f(rs[0] - mx);
            ls = fmaf(rs[16], w, ls);
            const float4 v = *reinterpret_cast<const float4*>(o_s + ((size_t)s * kRows + r) * kCols + 4 * v4);
            a.x = fmaf(v.x, w, a.x); a.y = fmaf(v.y, w, a.y); a.z = fmaf(v.z, w, a.z); a.w = fmaf(v.w, w, a.w);
        }
        const float inv = ls > 0.f ? 1.f / ls : 0.f;
        put(r, v4, make_float4(a.x * inv, a.y * inv, a.z * inv, a.w * inv));
    }
}

template <typename T, int QW, int SW, int NC, int DH>
__global__ void __launch_bounds__(32 * QW * SW)
generic_attention_kernel(Dims d, const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ c,
                         float* __restrict__ o_lat, const PageMap pm, int32_t* status_word, int tiles) {
    extern __shared__ __align__(16) float smem[];
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();       // (the decoder kernel's gate phase may start as SMs free up)
    // (row tiles and slices of d_l share x, heads and maps have y to themselves: 65535 of them)
    const int slice = (int)blockIdx.x / tiles, t0 = (tiles - 1 - ((int)blockIdx.x - slice * tiles)) * 16 * QW;   // the longest rows first
    const int g = blockIdx.y, b = blockIdx.z, col0 = slice * 64 * NC;
    attention_tile<T, QW, SW, NC, DH>(
        nullptr, d, q, k, c, pm, status_word, smem, threadIdx.x, t0, col0, g, b, [] { __syncthreads(); },
        // (the address is made here: held in registers from the start it costs some of these kernels a CTA of an SM)
        [&](int r, int v4, const float4 v) {
            *reinterpret_cast<float4*>(o_lat + (((size_t)blockIdx.y * d.B + blockIdx.z) * d.N + t0 + r) * d.d_l + col0 + 4 * v4) = v;
        });
}

// ---------------------------------------------------------------------------------------------
// Decoder + gate.  CTA tile: 16 RW token rows x 64 columns of one attention map's heads; 4 rows x 8 columns per lane
// and accumulator (gate pre-activation and decoded value); KW warps share a tile and each contract a KW-th of every
// k-block (added through shared memory at the end).  The gate's k-blocks (X, W_G) come first: they do not need the
// attention kernel's result, behind which this kernel is programmatically launched.
constexpr int kDecStages = 3;
__host__ __device__ constexpr int dec_bk(int KW) { return KW == 1 ? 32 : 16 * KW; }
constexpr size_t dec_smem_bytes(int RW, int KW) {
    return (size_t)kDecStages * (16 * RW * (dec_bk(KW) + 4) + dec_bk(KW) * 64) * sizeof(float);
}

template <typename T, int RW, int KW>
__global__ void __launch_bounds__(32 * RW * KW)
generic_decoder_kernel(Dims d, const float* __restrict__ o_lat, const T* __restrict__ x, const T* __restrict__ w_p,
                       const T* __restrict__ w_g, T* __restrict__ out, int tile0) {
    constexpr int kThreads = 32 * RW * KW, BM = 16 * RW, BN = 64, BK = dec_bk(KW), KPW = BK / KW;
    constexpr int kLdA = BK + 4, kStage = BM * kLdA + BK * BN;
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rw = warp % RW, kw = warp / RW;
    const int rg = lane >> 3, cg = lane & 7;                 // rows rg + 4 i; columns 4 cg + {0..3}, 32 + 4 cg + {0..3}

    const long long M = (long long)d.B * d.N;
    const int map_cols = d.n_h / d.n_q * d.d_h;
    const int g = blockIdx.z, c0 = (tile0 + (int)blockIdx.y) * BN;     // columns c0 .. of map g
    const int n_cols = min(BN, map_cols - c0);
    const long long m0 = (long long)blockIdx.x * BM;
    const int rows = (int)(M - m0 < BM ? M - m0 : BM);

    // A loader: BK / 4 vectors per row
    constexpr int kAVecs = BK / 4, kARows = kThreads / kAVecs, kAIter = BM / kARows;
    static_assert(kThreads % kAVecs == 0 && BM % kARows == 0, "A tile is dealt out evenly");
    const int a_row = tid / kAVecs, a_vec = tid % kAVecs;
    // B loader: BN / 4 vectors per k
    constexpr int kBVecs = BN / 4, kBRows = kThreads / kBVecs, kBIter = BK / kBRows;
    static_assert(kThreads % kBVecs == 0 && BK % kBRows == 0, "B tile is dealt out evenly");
    const int b_k = tid / kBVecs, b_col = 4 * (tid % kBVecs);
    const bool b_live = b_col < n_cols;
    const int head = g * (d.n_h / d.n_q) + (c0 + b_col) / d.d_h, elem = (c0 + b_col) % d.d_h;   // (d_h is a multiple of 8)
    const T* wg_col = w_g + (size_t)(b_live ? head : 0) * d.d_h + elem;
    const T* wp_col = w_p + (size_t)(b_live ? head : 0) * d.d_l * d.d_h + elem;
    const int n_g = (d.H + BK - 1) / BK, n_p = (d.d_l + BK - 1) / BK, n_it = n_g + n_p;

    auto load_block = [&](int it) {
        float* as = smem + (it % kDecStages) * kStage;
        float* bs = as + BM * kLdA;
        const bool gate = it < n_g;
        const int k0 = (gate ? it : it - n_g) * BK, K = gate ? d.H : d.d_l;
#pragma unroll
        for (int i = 0; i < kAIter; ++i) {
            const int r = a_row + i * kARows, kk = k0 + 4 * a_vec;
            const bool live = r < rows && kk < K;
            const long long m = live ? m0 + r : 0;
            float* dst = as + r * kLdA + 4 * a_vec;
            if (gate) {
                stage4(dst, x + (size_t)m * d.H + (live ? kk : 0), live);
            } else {
                stage4(dst, o_lat + ((size_t)g * M + m) * d.d_l + (live ? kk : 0), live);
            }
        }
        const T* w = gate ? wg_col : wp_col;
        const size_t ldw = gate ? (size_t)d.n_h * d.d_h : (size_t)d.d_h;
#pragma unroll
        for (int i = 0; i < kBIter; ++i) {
            const int kk = b_k + i * kBRows;
            const bool live = b_live && k0 + kk < K;
            stage4(bs + kk * BN + b_col, w + (size_t)(live ? k0 + kk : 0) * ldw, live);
        }
    };

    uint64_t acc_g[4][4], acc_p[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc_g[i][j] = acc_p[i][j] = 0ull;

    auto multiply = [&](int it, uint64_t (&acc)[4][4]) {
        const float* as = smem + (it % kDecStages) * kStage + (16 * rw + rg) * kLdA + kw * KPW;
        const float* bs = smem + (it % kDecStages) * kStage + BM * kLdA + kw * KPW * BN + 4 * cg;
#pragma unroll 2
        for (int k = 0; k < KPW; k += 4) {
            float4 a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(as + 4 * i * kLdA + k);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Pair2 b0 = lds_pair2(bs + (k + u) * BN), b1 = lds_pair2(bs + (k + u) * BN + 32);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float av = u == 0 ? a[i].x : u == 1 ? a[i].y : u == 2 ? a[i].z : a[i].w;
                    const uint64_t aa = ptx::f32x2(av, av);
                    acc[i][0] = ptx::fma2(aa, b0.lo, acc[i][0]);
                    acc[i][1] = ptx::fma2(aa, b0.hi, acc[i][1]);
                    acc[i][2] = ptx::fma2(aa, b1.lo, acc[i][2]);
                    acc[i][3] = ptx::fma2(aa, b1.hi, acc[i][3]);
                }
            }
        }
    };
    auto issue = [&](int it) {
        if (it < n_it) {
            if (it == n_g) ptx::grid_dependency_wait();     // L is the attention kernel's; X and the weights are older
            load_block(it);
        }
        cp_async_commit();
    };

#pragma unroll
    for (int s = 0; s < kDecStages - 1; ++s) issue(s);
    auto step = [&](int it, uint64_t (&acc)[4][4]) {
        cp_async_wait<kDecStages - 2>();
        __syncthreads();
        issue(it + kDecStages - 1);          // into the stage that everybody has left
        multiply(it, acc);
    };
    for (int it = 0; it < n_g; ++it) step(it, acc_g);
    for (int it = n_g; it < n_it; ++it) step(it, acc_p);

    if constexpr (KW > 1) {
        // the k-warps' partial sums meet in shared memory: [KW - 1][16][64] per accumulator, lane-contiguous
        cp_async_wait<0>();
        __syncthreads();
        uint64_t* part = reinterpret_cast<uint64_t*>(smem);
        static_assert(RW == 1, "one tile");
        static_assert((size_t)(KW - 1) * 32 * 32 * 8 <= dec_smem_bytes(1, KW), "the partial sums fit");
        if (kw > 0) {
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    part[((size_t)(kw - 1) * 32 + i * 4 + j) * 32 + lane] = acc_g[i][j];
                    part[((size_t)(kw - 1) * 32 + 16 + i * 4 + j) * 32 + lane] = acc_p[i][j];
                }
        }
        __syncthreads();
        if (kw > 0) return;
        for (int s = 0; s < KW - 1; ++s)
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc_g[i][j] = ptx::add2(acc_g[i][j], part[((size_t)s * 32 + i * 4 + j) * 32 + lane]);
                    acc_p[i][j] = ptx::add2(acc_p[i][j], part[((size_t)s * 32 + 16 + i * 4 + j) * 32 + lane]);
                }
    }

#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = 16 * rw + rg + 4 * i;
        if (r >= rows) continue;
        T* o_row = out + (size_t)(m0 + r) * d.n_h * d.d_h + (size_t)g * map_cols + c0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int cc = 32 * h + 4 * cg;
            if (cc >= n_cols) continue;
            float z[4], y[4];
            ptx::f32x2_split(acc_g[i][2 * h], z[0], z[1]);
            ptx::f32x2_split(acc_g[i][2 * h + 1], z[2], z[3]);
            ptx::f32x2_split(acc_p[i][2 * h], y[0], y[1]);
            ptx::f32x2_split(acc_p[i][2 * h + 1], y[2], y[3]);
#pragma unroll
            for (int u = 0; u < 4; ++u) y[u] *= 1.f / (1.f + expf(-z[u]));
            store4(o_row + cc, y);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// A short fp32 prompt in one kernel (d_h = 64, d_l = 128): 16 rows x 64 output columns of one map per CTA.  Warps 0-3 do the rows'
// attention (once more for every column block: it is latency, not work), warps 4-7 the gates meanwhile, with the first weights and
// W_P on their way from the start; then all eight contract L, which never leaves shared memory, with W_P.
// What bounds it is one chain of latencies and the way of 210 KB into an SM; two kernels have two chains, and a result through L2
// between them (128 tokens of the tiny layer 16.9 us, 11.7 in one; 100 tokens of the 1B layer 31.2, 18.3).  The latents and W_P, one
// piece each, travel by bulk copies beside the others' cp.async: 9.9 us.  (Keys and W_G by TMA too: 11.3; rows of 256 bytes by
// bulk copies: 15.5.)
constexpr int kShortBk = 64, kShortStages = 3, kShortLdA = kShortBk + 4, kShortLdL = 132;
constexpr int kShortStage = 16 * kShortLdA + kShortBk * 64;
__host__ __device__ inline int short_attn_floats() { return attn_smem(64, 16, 4 * kAttnKeys, 128, 4).total_floats; }
static size_t short_smem_bytes() {
    return (size_t)(short_attn_floats() + kShortStages * kShortStage + 128 * 64 + 16 * kShortLdL) * sizeof(float);
}

__global__ void __launch_bounds__(256)
short_prefill_f32_kernel(Dims d, const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ c,
                         const float* __restrict__ x, const float* __restrict__ w_p, const float* __restrict__ w_g,
                         float* __restrict__ out, int tiles, int32_t* status_word) {
    extern __shared__ __align__(16) float smem[];
    __shared__ uint64_t latent_bar, wp_bar;
    __shared__ int abort_word;
    volatile int* abort_flag = &abort_word;
    float* ring = smem + short_attn_floats();
    float* wp_s = ring + kShortStages * kShortStage;             // [128][64]
    float* l_s = wp_s + 128 * 64;                                // [16][kShortLdL]
    if (threadIdx.x == 0) {
        ptx::mbar_init(&latent_bar, 1);
        ptx::mbar_init(&wp_bar, 1);
        *abort_flag = 0;
        ptx::fence_mbar_init();
    }
    __syncthreads();
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ct = (int)blockIdx.x / tiles, t0 = (tiles - 1 - ((int)blockIdx.x - ct * tiles)) * 16;
    const int g = blockIdx.y, b = blockIdx.z, rows = min(16, d.N - t0);
    const int map_cols = d.n_h / d.n_q * d.d_h, c0 = ct * 64;    // (a multiple of 64)
    const int rg = lane >> 3, cg = lane & 7;                     // rows rg + 4 i; columns 4 cg + {0..3}, 32 + 4 cg + {0..3}
    const int head = g * (d.n_h / d.n_q) + ct;                   // (64 columns are a head)

    // 16 rows x 64 columns: a (rows apart by lda) times w [k][64], k = 0 .. 15
    const auto multiply16 = [&](const float* a_s, int lda, const float* w_s, uint64_t (&acc)[4][4]) {
        const float* as = a_s + rg * lda;
        const float* bs = w_s + 4 * cg;
#pragma unroll
        for (int kk = 0; kk < 16; kk += 4) {
            float4 a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(as + 4 * i * lda + kk);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const Pair2 b0 = lds_pair2(bs + (kk + u) * 64), b1 = lds_pair2(bs + (kk + u) * 64 + 32);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float av = u == 0 ? a[i].x : u == 1 ? a[i].y : u == 2 ? a[i].z : a[i].w;
                    const uint64_t aa = ptx::f32x2(av, av);
                    acc[i][0] = ptx::fma2(aa, b0.lo, acc[i][0]);
                    acc[i][1] = ptx::fma2(aa, b0.hi, acc[i][1]);
                    acc[i][2] = ptx::fma2(aa, b1.lo, acc[i][2]);
                    acc[i][3] = ptx::fma2(aa, b1.hi, acc[i][3]);
                }
            }
        }
    };
    uint64_t acc_g[4][4], acc_p[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc_g[i][j] = acc_p[i][j] = 0ull;

    BulkLatents bars{&latent_bar, abort_flag, 0};
    if (warp < 4) {
        attention_tile<float, 1, 4, 2, 64>(
            &bars, d, q, k, c, PageMap(), nullptr, smem, tid, t0, 0, g, b, [] { ptx::named_sync(1, 128); },
            [&](int r, int v4, const float4 v) { *reinterpret_cast<float4*>(l_s + r * kShortLdL + 4 * v4) = v; });
        // (rows past the last meet W_P too; their results go nowhere)
        for (int idx = tid; idx < (16 - rows) * 32; idx += 128)
            *reinterpret_cast<float4*>(l_s + (rows + idx / 32) * kShortLdL + 4 * (idx % 32)) = make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
        const int tg = tid - 128, n_blocks = (d.H + kShortBk - 1) / kShortBk;
        const float* x_rows = x + ((size_t)b * d.N + t0) * d.H;
        const float* wg = w_g + (size_t)head * d.d_h;
        const size_t ldw = (size_t)d.n_h * d.d_h;
        if (tg == 0) {
            ptx::mbar_arrive_expect_tx(&wp_bar, 128 * 64 * 4);
            ptx::bulk_load_1d(wp_s, w_p + (size_t)head * 128 * 64, 128 * 64 * 4, &wp_bar);
        }
        const auto load = [&](int it) {
            if (it < n_blocks) {
                float* as = ring + it % kShortStages * kShortStage;
                float* ws = as + 16 * kShortLdA;
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int r = (tg >> 4) + 8 * i, kk = it * kShortBk + 4 * (tg & 15);
                    const bool live = r < rows && kk < d.H;
                    cp_async_16(as + r * kShortLdA + 4 * (tg & 15), x_rows + (live ? (size_t)r * d.H + kk : 0), live);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int kl = (tg >> 4) + 8 * i, kk = it * kShortBk + kl;
                    cp_async_16(ws + kl * 64 + 4 * (tg & 15), wg + (kk < d.H ? kk * ldw : 0) + 4 * (tg & 15), kk < d.H);
                }
            }
        };
#pragma unroll
        for (int it = 0; it < kShortStages - 1; ++it) {
            load(it);
            cp_async_commit();
        }
        for (int it = 0; it < n_blocks; ++it) {
            cp_async_wait<kShortStages - 2>();
            ptx::named_sync(2, 128);
            load(it + kShortStages - 1);         // into the stage that everybody has left
            cp_async_commit();
            const float* as = ring + it % kShortStages * kShortStage;
            multiply16(as + 16 * (warp - 4), kShortLdA, as + 16 * kShortLdA + 16 * (warp - 4) * 64, acc_g);
        }
        cp_async_wait<0>();
        ptx::mbar_wait_sleep(&wp_bar, 0, abort_flag, 0, c_short_wait.limit_ns);
    }
    __syncthreads();
    multiply16(l_s + 16 * warp, kShortLdL, wp_s + 16 * warp * 64, acc_p);
    // the warps' partial sums meet where the latents were: [warp][pair of accumulators][lane], values, then gates
    uint64_t* part = reinterpret_cast<uint64_t*>(smem);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            part[(warp * 16 + 4 * i + j) * 32 + lane] = acc_p[i][j];
            if (warp >= 4) part[((warp + 4) * 16 + 4 * i + j) * 32 + lane] = acc_g[i][j];
        }
    __syncthreads();
    const int i = warp >> 1, j = 2 * (warp & 1), r = rg + 4 * i;     // this thread's four outputs
    float y[4], z[4];
    uint64_t s0 = 0ull, s1 = 0ull;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        s0 = ptx::add2(s0, part[(w * 16 + 4 * i + j) * 32 + lane]);
        s1 = ptx::add2(s1, part[(w * 16 + 4 * i + j + 1) * 32 + lane]);
    }
    ptx::f32x2_split(s0, y[0], y[1]);
    ptx::f32x2_split(s1, y[2], y[3]);
    s0 = s1 = 0ull;
#pragma unroll
    for (int w = 8; w < 12; ++w) {
        s0 = ptx::add2(s0, part[(w * 16 + 4 * i + j) * 32 + lane]);
        s1 = ptx::add2(s1, part[(w * 16 + 4 * i + j + 1) * 32 + lane]);
    }
    ptx::f32x2_split(s0, z[0], z[1]);
    ptx::f32x2_split(s1, z[2], z[3]);
    if (tid == 0 && *abort_flag) {           // a wait gave up: whatever is still on its way lands before the CTA leaves
        int gave_up = 0;
        if (bars.armed > 0) ptx::mbar_wait_drain(&latent_bar, (bars.armed - 1) & 1, &gave_up);
        ptx::mbar_wait_drain(&wp_bar, 0, &gave_up);
        raise_status(status_word, GTA_ERR_TIMEOUT);
    }
    if (r >= rows) return;
#pragma unroll
    for (int u = 0; u < 4; ++u) y[u] *= 1.f / (1.f + expf(-z[u]));
    store4(out + ((size_t)b * d.N + t0 + r) * d.n_h * d.d_h + (size_t)g * map_cols + c0 + 16 * j + 4 * cg, y);
}

// ---------------------------------------------------------------------------------------------
// Launch with programmatic stream serialisation (the kernel waits for the one before it by itself), or without.
template <typename Kern, typename... Args>
static cudaError_t launch_chained(bool behind, Kern kern, dim3 grid, int threads, size_t smem, cudaStream_t stream, Args... args) {
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

template <typename T, int QW, int SW, int NC, int DH>
static cudaError_t launch_attention(const Dims& d, const T* q, const T* k, const T* c, float* o_lat, cudaStream_t stream,
                                    const PageMap& pm, int32_t* status_word) {
    const AttnSmem L = attn_smem(d.d_h, 16 * QW, kAttnKeys * SW, 64 * NC, QW * SW);
    const size_t smem = (size_t)L.total_floats * sizeof(float);
    const int tiles = (d.N + 16 * QW - 1) / (16 * QW), n_slices = (d.d_l + 64 * NC - 1) / (64 * NC);
    auto kern = generic_attention_kernel<T, QW, SW, NC, DH>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    return launch_chained(true, kern, dim3(tiles * n_slices, d.n_q, d.B), 32 * QW * SW, smem, stream, d, q, k, c, o_lat, pm, status_word,
                          tiles);
}

template <typename T, int RW, int KW>
static cudaError_t launch_decoder(const Dims& d, const float* o_lat, const T* x, const T* w_p, const T* w_g, T* out,
                                  cudaStream_t stream, bool behind, int* launches) {
    auto kern = generic_decoder_kernel<T, RW, KW>;
    constexpr size_t smem = dec_smem_bytes(RW, KW);
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (err != cudaSuccess) return err;
    const int map_cols = d.n_h / d.n_q * d.d_h;
    const long long M = (long long)d.B * d.N;
    // a map of more than 65535 column tiles takes several launches (the tiles in x next to the rows' cost 3.5 % of 2 x 1500
    // tokens of the 1B layer)
    const int tiles = (map_cols + 63) / 64;
    for (int tile0 = 0; tile0 < tiles && err == cudaSuccess; tile0 += 65535, ++*launches)
        err = launch_chained(behind, kern, dim3((unsigned)((M + 16 * RW - 1) / (16 * RW)), min(tiles - tile0, 65535), d.n_q),
                             32 * RW * KW, smem, stream, d, o_lat, x, w_p, w_g, out, tile0);
    return err;
}

// Which kernels serve an fp32 call.  Measured, us, plain-ALU / tensor cores.  Attention: 1B layer, 64 tokens 18.5 / 21.2, 128
// 29.6 / 32.4, 2 x 100 47.4 / 32.3, 200 47.4 / 32.7; tiny layer, 4 x 128 17.3 / 20.1, 8 x 128 23.0 / 20.8, 333 28.5 / 23.3, 8 x 2048
// 527 / 160: from 192 keys, or more than 64 plain CTAs of 16 rows, on; but a tile of 128 rows that is half empty loses (64 tokens of 64
// sequences, w512 (16 heads, 8 maps, latents of 512) 222 / 236, 1B 131 / 128; 16 of 256 270 / 549, 135 / 176; 96 of 64 369 / 308,
// 150 / 137), and so do few rows behind short caches once there is more than a wave of them (64 sequences, a row behind 300 keys:
// w512 192 / 235, tiny 28 / 28; behind 1000 503 / 533, 69 / 62), the longer the more elements a token has, whose pieces are made for so
// few rows: all of these stay on the FMA pipe.  Decoder: 1B 200 tokens (80 tiles of 64 x 64) 32.7 / 42.7, 333
// (120) 54.4 / 42.6; tiny 700 (44) 28.4 / 30.3, 2048 (128) 45.3 / 38.7: from 100 tiles on; in blocks of 128 columns while those of
// 256 are few (us, 128 / 256: 1B, 1000 tokens, 20 blocks of 256, 44.1 / 56.7; 1100, 25, 46.5 / 56.6; 1200, 25, 60.5 / 56.9; 1400, 30,
// 65.7 / 58.3; 16 heads of 128, 4 maps, 700, 24, 162 / 174; 1000, 32, 251 / 244).  The line of 100 tiles, plain / 128: 1B 80 33.8 / 42.8, 100
// 44.1 / 42.9; 16 heads of 128, 64 77.8 / 78.6, 128 88.7 / 70.1; w512 96 61.1 / 50.1, 112 64.4 / 62.3; one map of 8 heads 88 38.9 / 30.4.
//
// CTAs that share the keys of a row tile (a model fitted to the tiny and the 1B layer, with 148 places for clusters too): a key tile
// takes 1.25 us, a CTA 6 us more and 1 for every one that it merges with, a stage of the decoder 0.9 or 1.05 us.  The decoder's gates run beside the attention kernel where both fit the chip at once (1B, 1000
// tokens: 47.1 with one, 54.6 with two; tiny, 2048: 75.5 / 48.8 / 38.7 with one / two / four); a plain decoder wants the SMs that a
// split takes (1B, 200 tokens: 32.7 / 43.3; tiny, 333: 26.0 / 23.3).
//
// Below both lines, d_h = 64 and d_l = 128 run in one kernel while its CTAs are one wave (tiny, 4 x 128, 128 CTAs: 17.8 us in two, 12.8;
// a second wave would bring every column block's attention once more).
struct F32Plan { int split = 0, cols = 0; bool one = false; };       // 0: the plain-ALU kernel; one: both in one kernel
static size_t l_bytes(const Dims& d) { return ((size_t)d.B * d.n_q * d.N * d.d_l * sizeof(float) + 255) & ~(size_t)255; }
static F32Plan f32_plan(const Dims& d, const PageMap& pm, size_t room) {
    F32Plan plan;
    const long long M = (long long)d.B * d.N;
    const int map_cols = d.n_h / d.n_q * d.d_h;
    if (M > (1 << 30) || (long long)d.n_h * d.d_h > (1 << 30)) return plan;       // (the kernels count rows and columns in 32 bits)
    const long long tiles64 = ((M + 63) / 64) * d.n_q * ((map_cols + 63) / 64);
    if (d.d_h % 64 == 0 && tiles64 >= 100) plan.cols = map_cols > 128 && sm100_decoder_f32_units(d, 256) > 28 ? 256 : 128;
    const long long plain = (long long)d.B * d.n_q * ((d.N + 15) / 16);
    const long long items = (long long)((d.N + 127) / 128) * (d.d_l / 128) * d.n_q * d.B;
    const int token = d.n_k * d.d_h + d.n_c * d.d_l;             // cached elements of a token
    const bool few_rows = d.Nk < 192 ? plain <= 64 || d.N < 96 : d.N < 64 && (token < 512 ? items > 296 && d.Nk < 640 : items > 148 && d.Nk < 1536);
    if (pm.table != nullptr || !sm100_attention_f32_supported(d) || few_rows ||
        room < l_bytes(d) + sm100_attention_f32_scratch(d)) {
        plan.one = pm.table == nullptr && plan.cols == 0 && d.d_h == 64 && d.d_l == 128 && d.Nk < 192 &&
                   plain * (d.n_h / d.n_q) <= 148;
        return plan;
    }
    const long long dec_ctas = plan.cols ? 2 * sm100_decoder_f32_units(d, plan.cols) : 0;
    const float stage = plan.cols == 256 ? 1.05f : 0.9f, dec_waves = (float)((dec_ctas + 147) / 148);
    const float gates = dec_waves * stage * ((d.H + 31) / 32), values = dec_waves * stage * ((d.d_l + 31) / 32);
    const float most = (float)((d.Nk + 63) / 64), mean = d.causal ? most - 0.5f * d.N / 64.f + 0.5f : most;       // key tiles of an item
    float best = 0.f;
    for (int split = 1; split <= 4; split *= 2) {
        const float fixed = 6.f + split;
        const float waves = (float)((items * split + 147) / 148);
        const float att = fmaxf(1.25f * most / split + fixed, waves * (1.25f * mean / split + fixed));
        const float total = plan.cols == 0                        ? att + (split > 1 ? 2.f : 0.f)
                            : items * split + dec_ctas <= 148 ? fmaxf(att, gates) + values
                                                              : att + gates + values;
        if (plan.split == 0 || total < best) { best = total; plan.split = split; }
    }
    return plan;
}

gta_status_t short_prefill_debug_wait(unsigned long long limit_ns, int withhold_first_arrive) {
    const ShortWait w = {limit_ns ? limit_ns : ptx::kWaitLimitNs, withhold_first_arrive ? 1 : 0};
    if (cudaMemcpyToSymbol(c_short_wait, &w, sizeof(w)) == cudaSuccess) return GTA_OK;
    cudaGetLastError();
    return GTA_ERR_CUDA;
}

template <typename T>
static cudaError_t launch_typed(const Dims& d, const void* q, const void* k, const void* c, const void* x,
                                const void* w_p, const void* w_g, void* out, float* o_lat_ws, size_t room,
                                cudaStream_t stream, int stages, int* launches, const PageMap& pm,
                                int32_t* status_word) {
    cudaError_t err;
    const F32Plan plan = std::is_same_v<T, float> ? f32_plan(d, pm, room) : F32Plan{};
    if constexpr (std::is_same_v<T, float>) {
        if (plan.one && (stages & 3) == 3) {
            const size_t smem = short_smem_bytes();
            const int tiles = (d.N + 15) / 16;
            err = cudaFuncSetAttribute(short_prefill_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (err != cudaSuccess) return err;
            *launches += 1;
            return launch_chained(true, short_prefill_f32_kernel, dim3(tiles * (d.n_h / d.n_q), d.n_q, d.B), 256, smem, stream, d, (const float*)q,
                                  (const float*)k, (const float*)c, (const float*)x, (const float*)w_p, (const float*)w_g, (float*)out, tiles, status_word);
        }
    }
    if constexpr (std::is_same_v<T, float>) {
        if ((stages & 1) && plan.split) {
            err = launch_sm100_attention_f32(d, (const float*)q, (const float*)k, (const float*)c, o_lat_ws,
                                             reinterpret_cast<uint8_t*>(o_lat_ws) + l_bytes(d), status_word, stream, plan.split, launches);
            if (err != cudaSuccess) return err;
        }
    }
    if ((stages & 1) && !plan.split) {
        // Which split: the CTAs of 64 rows that the call would have.  Measured (us; (1,4) / (2,4) / (2,2) warps over rows and
        // keys; four warps on 64 rows were never the best): 20 (1B layer, 256 tokens) 16 / 20 / 24; 56 (tiny layer, 1767)
        // 86 / 112 / 162; 80 (1B, 1000) 84 / 67 / 101; 128 (tiny, 8 x 512) 72 / 59 / 72; 160 (1B, 2048) 268 / 209 / 269;
        // 240 (1B, 2 x 1500) 276 / 214 / 212; 375 (1B, 5 x 900) 273 / 197 / 177; 512 (tiny, 8 x 2048) 731 / 523 / 462.
        // Wide heads have no room for the larger key tiles.
        const long long ctas64 = (long long)d.B * d.n_q * ((d.N + 63) / 64) * ((d.d_l + 127) / 128);
        const auto fits = [&](int qw, int sw) {
            return (size_t)attn_smem(d.d_h, 16 * qw, sw * kAttnKeys, 128, qw * sw).total_floats * sizeof(float) <= 227 * 1024;
        };
        const auto go = [&](auto nc, auto dh) {
            constexpr int NC = decltype(nc)::value, DH = decltype(dh)::value;
            const T *qt = (const T*)q, *kt = (const T*)k, *ct = (const T*)c;
            if (ctas64 <= 60 && fits(1, 4)) return launch_attention<T, 1, 4, NC, DH>(d, qt, kt, ct, o_lat_ws, stream, pm, status_word);
            if (ctas64 <= 200 && fits(2, 4)) return launch_attention<T, 2, 4, NC, DH>(d, qt, kt, ct, o_lat_ws, stream, pm, status_word);
            return launch_attention<T, 2, 2, NC, DH>(d, qt, kt, ct, o_lat_ws, stream, pm, status_word);
        };
        const auto go_dh = [&](auto nc) {
            if (d.d_h == 64) return go(nc, std::integral_constant<int, 64>{});
            if (d.d_h == 128) return go(nc, std::integral_constant<int, 128>{});
            return go(nc, std::integral_constant<int, 0>{});
        };
        err = d.d_l <= 64 ? go_dh(std::integral_constant<int, 1>{}) : go_dh(std::integral_constant<int, 2>{});
        if (err != cudaSuccess) return err;
        *launches += 1;
    }
    if (stages & 2) {
        // 64 x 64 tiles, or 16 x 64 tiles with the contraction split over four or eight warps where those would not fill
        // the chip.  Measured (us; 8 / 4 warps / 64 rows): 20 tiles of 64 x 64 (64 rows, 1280 columns) 19 / 22 / 59; 60:
        // 36 / 32 / 59; 112 (1767 rows, 256 columns) 26 / 16 / 21; 200 (600 rows) 105 / 78 / 91; 256 (4096 rows, 256
        // columns) 58 / 34 / 30; 640 (2048 rows) 315 / 220 / 200.
        const long long tiles64 = (((long long)d.B * d.N + 63) / 64) * d.n_q * ((d.n_h / d.n_q * d.d_h + 63) / 64);
        const float* l = o_lat_ws;
        if constexpr (std::is_same_v<T, float>) {
            if (plan.cols) {
                err = launch_sm100_decoder_f32(d, l, (const float*)x, (const float*)w_p, (const float*)w_g, (float*)out, status_word,
                                               stream, stages & 1, plan.cols);
                if (err != cudaSuccess) return err;
                *launches += 1;
                return cudaSuccess;
            }
        }
        const bool behind = stages & 1;      // X and W_G are read ahead of the wait: they are older than the attention kernel only
        err = tiles64 < 40    ? launch_decoder<T, 1, 8>(d, l, (const T*)x, (const T*)w_p, (const T*)w_g, (T*)out, stream, behind, launches)
              : tiles64 < 256 ? launch_decoder<T, 1, 4>(d, l, (const T*)x, (const T*)w_p, (const T*)w_g, (T*)out, stream, behind, launches)
                              : launch_decoder<T, 4, 1>(d, l, (const T*)x, (const T*)w_p, (const T*)w_g, (T*)out, stream, behind, launches);
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

cudaError_t launch_generic_prefill(const Dims& d, int dtype, const void* q, const void* k, const void* c,
                                   const void* x, const void* w_p, const void* w_g, void* out,
                                   float* o_lat_ws, size_t room, cudaStream_t stream, int stages, int* launches,
                                   const PageMap& pm, int32_t* status_word) {
    if (dtype == GTA_F32)
        return launch_typed<float>(d, q, k, c, x, w_p, w_g, out, o_lat_ws, room, stream, stages, launches, pm, status_word);
    return launch_typed<__nv_bfloat16>(d, q, k, c, x, w_p, w_g, out, o_lat_ws, room, stream, stages, launches, pm,
                                       status_word);
}

}  // namespace gta
