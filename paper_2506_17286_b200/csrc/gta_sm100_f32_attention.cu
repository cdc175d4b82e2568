// fp32 attention on the tensor cores (head width 64): L = Softmax(scale Q K^T) C per attention map.
//
// Operands are sums of three bf16 pieces, exactly from 2^-110 on, and six of the nine products of pieces are taken (what is left
// out is below 2^-24 of a product, 2^-26.5 rms); see gta_sm100_f32_decoder.cu.  A sum stays in tensor memory for 64 elements of
// its contraction (the head width; the keys of a tile), small products first, and is added up in registers (rounded) from there.
//   split_rows_kernel        writes the pieces of K and C once ([piece][row], bf16, workspace), and per tile of 64
//                            rows the first that holds an element without pieces: every map and row tile reads them.
//   sm100_attention_f32_kernel  a CTA (or a cluster of two or four that take the key tiles in turn and merge at the end through
//                            distributed shared memory) owns 128 query rows x 128 latent columns of a map:
//     warp 0       brings the pieces of key tiles in by TMA (64 keys x (64 + 128) columns x 3 = 72 KB a stage, 3 stages).
//     warp 1       issues the MMAs: S = Q K^T (pieces of Q in tensor memory), two tiles ahead of O = P C (pieces of P in tensor
//                  memory, the first two where the scores were), 64 latent columns after 64.
//     warps 4-11   softmax, two warpgroups on alternating tiles with a running maximum and row sum each: a thread is a row.
//     warps 12-19  add the O of a tile to their registers, in the scale of the largest maximum so far.
// Per key tile: 72 MMAs of N = 64, 2304 cycles of the tensor pipe, which the rest is to hide under: measured 2850.  (With one
// buffer of P, written between two products, and O in one piece: 3060.)
//
// An element that is infinite, not a number or rounds to infinity in bf16 has no pieces.  In K and C zeros stand in for it, so
// that rows which do not see it keep their bits (0 x infinity); the rows that do, and the rows of Q that hold one, are done
// again with plain FMAs.  So are those that see, or are, a row of elements too small for pieces (kPiecesFloor).  A probability
// is taken against the largest of its row so far: one below 2^-110 of it loses at most 2^-134 of it.
#include "gta_sm100.cuh"

#include <cuda.h>

#include <type_traits>

#include "sm100_ptx.cuh"
#include "tma_host.cuh"

namespace gta {

namespace {

constexpr int kDh = 64, kRows = 128, kKeys = 64, kCols = 128;        // head width; rows, keys of a tile, latent columns of a CTA
constexpr int kStages = 3;
constexpr uint32_t kKPlane = kKeys * kDh * 2, kCPlane = kKeys * kCols * 2, kCBlock = kKeys * 128;
constexpr uint32_t kStageBytes = 3 * (kKPlane + kCPlane);            // 72 KB
constexpr uint32_t kBarOffset = kStages * kStageBytes;
constexpr uint32_t kSmem = kBarOffset + 512 + 8 * kRows * 4 + 1024;  // barriers; maxima and sums of rows; alignment
static_assert(kSmem <= 227 * 1024, "shared memory of a CTA");
constexpr int kSoftWarp0 = 4, kAddWarp0 = 12, kThreads = 640;
// registers: 640 threads start with 96 each (61440): 128 x 48 + 256 x 104 + 256 x 112
constexpr int kIssueRegs = 48, kSoftRegs = 104, kAddRegs = 112;
// tensor memory columns
constexpr uint32_t kTmS = 0, kTmSP = 96, kTmQ = 192, kTmO = 320;      // [2] 64 columns of scores or 96 of P; Q 96; O 128

// ---------------------------------------------------------------------------------------------
// Pieces of four floats.  What two pieces leave of a number has eight bits, which are the upper half of its word; the lower half
// of `rest` (an OR over the four) is not zero where one leaves more: it ends below bf16's range, or has no pieces.
struct Pieces { uint2 p[3]; uint32_t rest; };
__device__ __forceinline__ Pieces split4(uint64_t r0, uint64_t r1) {
    Pieces o;
    float a, b, e, f;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        ptx::f32x2_split(r0, a, b);
        ptx::f32x2_split(r1, e, f);
        o.p[p] = make_uint2(ptx::cvt_bf16x2(a, b), ptx::cvt_bf16x2(e, f));
        r0 = ptx::sub2(r0, ptx::f32x2(__uint_as_float(o.p[p].x << 16), __uint_as_float(o.p[p].x & 0xffff0000u)));
        r1 = ptx::sub2(r1, ptx::f32x2(__uint_as_float(o.p[p].y << 16), __uint_as_float(o.p[p].y & 0xffff0000u)));
    }
    ptx::f32x2_split(r0, a, b);
    ptx::f32x2_split(r1, e, f);
    o.p[2] = make_uint2(ptx::upper_halves(__float_as_uint(a), __float_as_uint(b)), ptx::upper_halves(__float_as_uint(e), __float_as_uint(f)));
    o.rest = __float_as_uint(a) | __float_as_uint(b) | __float_as_uint(e) | __float_as_uint(f);
    return o;
}
// Does what its pieces do not add up to matter to a row: has it an element without pieces, or small ones alone?
__device__ __noinline__ bool is_odd_row(const float* row, int width) {
    float mx = 0.f;
    for (int e = 0; e < width; ++e) {
        if (!(fabsf(row[e]) < 3.3895e38f)) return true;
        mx = fmaxf(mx, fabsf(row[e]));
    }
    return mx < kPiecesFloor;
}

// The pair with zeros for what has no pieces (3.3895e38 is bf16's largest).
__device__ __forceinline__ uint64_t whole2(uint64_t v) {
    float a, b;
    ptx::f32x2_split(v, a, b);
    return ptx::f32x2(fabsf(a) < 3.3895e38f ? a : 0.f, fabsf(b) < 3.3895e38f ? b : 0.f);
}

// One CTA per tile of 64 rows of one (sequence, group) of K (the first B n_k of them) or C, tiles of a group next to one another.
__global__ void __launch_bounds__(256)
split_rows_kernel(Dims d, const float* __restrict__ k, const float* __restrict__ c, uint8_t* __restrict__ k_planes,
                  uint8_t* __restrict__ c_planes, int32_t* __restrict__ first_odd, int tiles) {
    ptx::grid_dependency_wait();
    ptx::grid_launch_dependents();
    const int n_kp = d.B * d.n_k, tile = (int)blockIdx.x % tiles, which = (int)blockIdx.x / tiles;
    const bool latent = which >= n_kp;
    const int plane = latent ? which - n_kp : which;
    const int width = latent ? d.d_l : kDh, vecs = width / 4;
    const float* src = (latent ? c : k) + ((size_t)plane * d.S + (size_t)tile * kKeys) * width;
    const size_t n_rows = (size_t)d.B * (latent ? d.n_c : d.n_k) * d.Nk;
    uint8_t* dst = (latent ? c_planes : k_planes) + ((size_t)plane * d.Nk + (size_t)tile * kKeys) * width * 2;
    const int live = min(kKeys, d.Nk - tile * kKeys) * vecs;
    __shared__ int first;
    if (threadIdx.x == 0) first = INT32_MAX;
    __syncthreads();
    // (four loads ahead of the stores, which the compiler cannot move them across)
    for (int i0 = threadIdx.x; i0 < live; i0 += 4 * 256) {
        ulonglong2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + 256 * u < live) v[u] = __ldg(reinterpret_cast<const ulonglong2*>(src) + i0 + 256 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + 256 * u;
            if (i >= live) break;
            Pieces s = split4(v[u].x, v[u].y);
            if ((s.rest & 0xffffu) != 0u) {
                if (is_odd_row(src + (size_t)(i / vecs) * width, width)) atomicMin(&first, tile * kKeys + i / vecs);
                s = split4(whole2(v[u].x), whole2(v[u].y));
            }
#pragma unroll
            for (int p = 0; p < 3; ++p) *reinterpret_cast<uint2*>(dst + (size_t)p * n_rows * width * 2 + (size_t)i * 8) = s.p[p];
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) first_odd[blockIdx.x] = first;
}

// ---------------------------------------------------------------------------------------------
// 32 neighbouring query rows with plain FMAs by eight warps (`tid` of 256, barrier 2), four rows each, 32 keys at a time: a lane has a
// key's scores, then four columns of the sums.  Row r has live0 + r live_step keys, live_max at most, and none of the others is
// looked at (0 x infinity).  odd(r): is the row to be stored?
// (A warp per row and a key at a time, the lanes sharing the head width, took 12 ms where an infinity in the first key or latent made
// all rows of 2 x 1500 tokens of the 1B layer odd; four rows a warp with keys from L1 1.4 ms, 0.65 now; the plain-ALU kernel takes 0.21 for all.)
constexpr int kOddRows = 32, kOddLd = kDh + 4;
constexpr uint32_t kOddSmem = (32 * kOddLd + 32 * kCols + kOddRows * kDh + kOddRows * 32) * 4;
static_assert(kOddSmem <= kBarOffset, "in the ring's memory");
template <typename Odd>
__device__ __forceinline__ void plain_rows(const Dims& d, const float* __restrict__ q_rows, const float* __restrict__ k_rows,
                                           const float* __restrict__ c_rows, float* __restrict__ out, int live0, int live_step, int live_max,
                                           int n_rows, float* smem, int tid, Odd odd) {
    const float scale2 = d.scale * 1.4426950408889634f;
    float* k_s = smem;                                         // [32][kOddLd]
    float* c_s = k_s + 32 * kOddLd;                            // [32][kCols]
    float* q_s = c_s + 32 * kCols;                             // [row][kDh]
    float* p_s = q_s + kOddRows * kDh;                         // [row][32]
    const int warp = tid >> 5, lane = tid & 31, r0 = 4 * warp;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = tid; i < kOddRows * kDh / 4; i += 256)
        reinterpret_cast<float4*>(q_s)[i] = i < n_rows * kDh / 4 ? reinterpret_cast<const float4*>(q_rows)[i] : zero;
    float m[4], l[4];
    float4 o[4];
    int live[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        m[r] = -INFINITY;
        l[r] = 0.f;
        o[r] = zero;
        live[r] = r0 + r < n_rows ? min(live0 + (r0 + r) * live_step, live_max) : 0;
    }
    const int most = min(live0 + (n_rows - 1) * live_step, live_max);
#pragma unroll 1
    for (int j0 = 0; j0 < most; j0 += 32) {
        const int n = min(32, most - j0);
        // (what a thread stages is asked for at once)
        float4 kv[2], cv[4];
#pragma unroll
        for (int u = 0; u < 2; ++u)
            kv[u] = reinterpret_cast<const float4*>(k_rows + (size_t)(j0 + min((tid >> 4) + 16 * u, n - 1)) * kDh)[tid & 15];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            cv[u] = reinterpret_cast<const float4*>(c_rows + (size_t)(j0 + min((tid >> 5) + 8 * u, n - 1)) * d.d_l)[tid & 31];
        ptx::named_sync(2, 256);                               // (the keys before have been used; q is there)
#pragma unroll
        for (int u = 0; u < 2; ++u) *reinterpret_cast<float4*>(k_s + ((tid >> 4) + 16 * u) * kOddLd + 4 * (tid & 15)) = kv[u];
#pragma unroll
        for (int u = 0; u < 4; ++u) reinterpret_cast<float4*>(c_s)[tid + 256 * u] = cv[u];
        ptx::named_sync(2, 256);
        float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
        for (int e = 0; e < kDh; e += 4) {
            const float4 kv = *reinterpret_cast<const float4*>(k_s + lane * kOddLd + e);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const float4 qv = *reinterpret_cast<const float4*>(q_s + (r0 + r) * kDh + e);
                s[r] = fmaf(qv.x, kv.x, fmaf(qv.y, kv.y, fmaf(qv.z, kv.z, fmaf(qv.w, kv.w, s[r]))));
            }
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float v = j0 + lane < live[r] ? s[r] * scale2 : -INFINITY;
            const float m_new = fmaxf(m[r], warp_max(v)), ref = m_new == -INFINITY ? 0.f : m_new;
            const float al = m_new == m[r] ? 1.f : exp2f(m[r] - ref), pr = exp2f(v - ref);
            m[r] = m_new;
            l[r] = fmaf(l[r], al, pr);
            o[r].x *= al; o[r].y *= al; o[r].z *= al; o[r].w *= al;
            p_s[(r0 + r) * 32 + lane] = pr;
        }
        __syncwarp();
#pragma unroll 4
        for (int jj = 0; jj < n; ++jj) {
            const float4 cv = *reinterpret_cast<const float4*>(c_s + jj * kCols + 4 * lane);
#pragma unroll
            for (int r = 0; r < 4; ++r)
                if (j0 + jj < live[r]) {
                    const float pr = p_s[(r0 + r) * 32 + jj];
                    o[r].x = fmaf(pr, cv.x, o[r].x); o[r].y = fmaf(pr, cv.y, o[r].y);
                    o[r].z = fmaf(pr, cv.z, o[r].z); o[r].w = fmaf(pr, cv.w, o[r].w);
                }
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const float sum = warp_sum(l[r]), inv = sum > 0.f ? 1.f / sum : 0.f;
        if (r0 + r < n_rows && odd(r0 + r))
            reinterpret_cast<float4*>(out + (size_t)(r0 + r) * d.d_l)[lane] = make_float4(o[r].x * inv, o[r].y * inv, o[r].z * inv, o[r].w * inv);
    }
    ptx::named_sync(2, 256);
}

// The rows of an item that see, or are, odd elements (see the top), by the adding warps.
__device__ __forceinline__ void redo_rows(const Dims& d, const float* q, const float* k, const float* c, float* o_lat, int t0, int slice, int g, int b,
                                       int first, const uint32_t* odd_rows, float* smem, int tid) {
    const int off = d.causal ? d.Nk - d.N : 0, rows = min(kRows, d.N - t0);
    for (int r = 0; r < rows; r += kOddRows) {
        const int n = min(kOddRows, rows - r), live0 = d.causal ? t0 + r + off + 1 : d.Nk, step = d.causal ? 1 : 0;
        const uint32_t bits = odd_rows[r >> 5];
        if (bits == 0 && min(live0 + (n - 1) * step, d.Nk) <= first) continue;
        plain_rows(d, q + (((size_t)b * d.n_q + g) * d.N + t0 + r) * kDh, k + ((size_t)b * d.n_k + d.q_to_k(g)) * d.S * kDh,
                   c + ((size_t)b * d.n_c + d.q_to_c(g)) * d.S * d.d_l + slice * kCols,
                   o_lat + (((size_t)g * d.B + b) * d.N + t0 + r) * d.d_l + slice * kCols, live0, step, d.Nk, n, smem, tid,
                   [&](int i) { return (bits >> i & 1) != 0 || min(live0 + i * step, d.Nk) > first; });
    }
}

// Test hook of the bounded waits (gta_debug_attention_wait): their time limit, and a switch that makes one softmax warp keep its first
// arrival to itself.
struct WaitHook { unsigned long long limit_ns; int withhold; };
static __constant__ WaitHook c_wait = {ptx::kWaitLimitNs, 0};

template <int SW>
__global__ void __launch_bounds__(kThreads, 1)
sm100_attention_f32_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_c,
                           const __grid_constant__ CUtensorMap tm_l, Dims d, const float* __restrict__ q, const float* __restrict__ k,
                           const float* __restrict__ c, float* o_lat, const int32_t* __restrict__ first_odd, int row_tiles, int slices,
                           int32_t* status_word) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* k_full = reinterpret_cast<uint64_t*>(smem + kBarOffset);
    uint64_t* c_full = k_full + kStages;
    uint64_t* k_empty = c_full + kStages;        // 4 warps: the softmax warpgroup that has seen the scores complete ...
    uint64_t* c_empty = k_empty + kStages;       // ... and the adding one that has seen the last sums complete (a commit more
                                                 // by the issuing thread takes it some 200 cycles)
    uint64_t* s_full = c_empty + kStages;        // [2]
    uint64_t* p_full = s_full + 2;               // [2]: 4 warps
    uint64_t* o_full = p_full + 2;               // [2] halves of the columns
    uint64_t* o_free = o_full + 2;               // [2]: 4 warps
    uint64_t* q_full = o_free + 2;               // 8 warps
    uint64_t* drain_bar = q_full + 1;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* drain_flag = abort_flag + 1;
    int* odd_key = reinterpret_cast<int*>(tmem_slot + 3);                     // first key of the item that is done again
    uint32_t* odd_rows = tmem_slot + 4;                                       // [4]: query rows, a bit each
    float* ref_s = reinterpret_cast<float*>(smem + kBarOffset + 512);        // [4][128]: the scale of a tile's P
    float* fin_m = ref_s + 4 * kRows;                                         // [2][128]
    float* fin_l = fin_m + 2 * kRows;                                         // [2][128]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = SW > 1 ? (int)ptx::cluster_ctarank() : 0;
    // the longest rows first
    const int u = blockIdx.x / SW, per_tile = slices * d.n_q * d.B;
    const int t0 = (row_tiles - 1 - u / per_tile) * kRows;
    const int slice = u % slices, g = u / slices % d.n_q, b = u / (slices * d.n_q) % d.B;
    const int kg = d.q_to_k(g), cg = d.q_to_c(g);
    const int off = d.causal ? d.Nk - d.N : 0;                                // causal: row t attends keys 0 .. t + off
    const int rows = min(kRows, d.N - t0);
    const int n_keys = d.causal ? min(t0 + rows + off, d.Nk) : d.Nk;
    const int n_tiles = (n_keys + kKeys - 1) / kKeys;
    const int n_my = n_tiles > rank ? (n_tiles - rank + SW - 1) / SW : 0;     // tiles rank, rank + SW, ...

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) { ptx::mbar_init(&k_full[s], 1); ptx::mbar_init(&c_full[s], 1); ptx::mbar_init(&k_empty[s], 4); ptx::mbar_init(&c_empty[s], 4); }
        for (int s = 0; s < 2; ++s) { ptx::mbar_init(&s_full[s], 1); ptx::mbar_init(&p_full[s], 4); ptx::mbar_init(&o_full[s], 1); ptx::mbar_init(&o_free[s], 4); }
        ptx::mbar_init(q_full, 8);
        ptx::mbar_init(drain_bar, 1);
        *abort_flag = 0;
        *drain_flag = 0;
        *odd_key = INT32_MAX;
        for (int i = 0; i < 4; ++i) odd_rows[i] = 0;
        ptx::fence_mbar_init();
    }
    if (warp == 0) ptx::tmem_alloc(tmem_slot, 512);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::tc_fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    ptx::grid_launch_dependents();       // (the decoder kernel's gates may start as SMs free up)

    const auto wait = [&](uint64_t* bar, uint32_t parity) { return ptx::mbar_wait_sleep(bar, parity, abort_flag, 0, c_wait.limit_ns); };

    if (warp < kSoftWarp0) {
        ptx::set_max_regs_dec<kIssueRegs>();
        if (warp == 0 && ptx::elect_one()) {
            ptx::prefetch_tensormap(&tm_k); ptx::prefetch_tensormap(&tm_c); ptx::prefetch_tensormap(&tm_l);
            ptx::grid_dependency_wait();
            const int k_plane = b * d.n_k + kg, c_plane = b * d.n_c + cg;
            bool ok = true, c_last = true;       // (whether the last tile's latents were asked for too)
            int i = 0, s = 0;
            uint32_t ph = 1;
            for (; i < n_my; ++i) {
                ok = wait(&k_empty[s], ph);
                if (!ok) break;
                const int j0 = (rank + SW * i) * kKeys;
                uint8_t* st = smem + s * kStageBytes;
                ptx::mbar_arrive_expect_tx(&k_full[s], 3 * kKPlane);
                for (int p = 0; p < 3; ++p) ptx::tma_load_3d(st + p * kKPlane, &tm_k, &k_full[s], 0, j0, p * d.B * d.n_k + k_plane);
                ok = wait(&c_empty[s], ph);
                if (!ok) { ++i; c_last = false; break; }
                ptx::mbar_arrive_expect_tx(&c_full[s], 3 * kCPlane);
                for (int p = 0; p < 3; ++p)
                    for (int v = 0; v < kCols / 64; ++v)
                        ptx::tma_load_3d(st + 3 * kKPlane + p * kCPlane + v * kCBlock, &tm_c, &c_full[s], slice * kCols + 64 * v, j0,
                                         p * d.B * d.n_c + c_plane);
                s = s + 1 == kStages ? 0 : s + 1;
                ph ^= s == 0;
            }
            // every armed tile lands (or the wait gives up) before this thread is done: others may give up behind its last wait
            for (int back = 1; back <= kStages && i - back >= 0; ++back) {
                ptx::mbar_wait_drain(&k_full[(i - back) % kStages], ((i - back) / kStages) & 1, drain_flag);
                if (back > 1 || c_last) ptx::mbar_wait_drain(&c_full[(i - back) % kStages], ((i - back) / kStages) & 1, drain_flag);
            }
        } else if (warp == 1 && ptx::elect_one()) {
            const uint32_t idesc_s = ptx::make_idesc_bf16(kRows, kKeys, 0, 0), idesc_o = ptx::make_idesc_bf16(kRows, 64, 0, 1);
            const uint64_t k_desc = ptx::make_smem_desc(ptx::smem_addr(smem), 16, 1024);
            const uint64_t c_desc = ptx::make_smem_desc(ptx::smem_addr(smem) + 3 * kKPlane, kCBlock, 1024);
            const uint32_t k_lo0 = (uint32_t)k_desc, k_hi = (uint32_t)(k_desc >> 32), c_lo0 = (uint32_t)c_desc, c_hi = (uint32_t)(c_desc >> 32);
            constexpr int kPa[6] = {2, 1, 0, 1, 0, 0}, kPb[6] = {0, 1, 2, 0, 1, 0};       // products of pieces, the smallest first
            bool ok = true;
            int ss = 0, so = 0;          // stages of the next scores and sums
            uint32_t phs = 0;
            // (the scores of i - 2 have been read and their P used: both by MMAs and waits before)
            auto scores = [&](int i) {
                ok = wait(&k_full[ss], phs);
                if (!ok) return;
                ptx::tc_fence_after_sync();
                const uint32_t lo = k_lo0 + ss * (kStageBytes >> 4);
#pragma unroll
                for (int v = 0; v < 6; ++v)
#pragma unroll
                    for (int k4 = 0; k4 < kDh / 16; ++k4)
                        ptx::mma_ts(tmem + kTmS + (i & 1) * kTmSP, tmem + kTmQ + kPa[v] * 32 + k4 * 8,
                                    ptx::desc_of(lo + ((kPb[v] * kKPlane + k4 * 32) >> 4), k_hi), idesc_s, (v | k4) ? 1u : 0u);
                ptx::tc_commit(&s_full[i & 1]);
                ss = ss + 1 == kStages ? 0 : ss + 1;
                phs ^= ss == 0;
            };
            if (n_my > 0) {
                ok = wait(q_full, 0);
                if (ok) scores(0);
                if (ok && n_my > 1) scores(1);
            }
            for (int i = 0; i < n_my && ok; ++i) {
                ok = wait(&p_full[i & 1], (i >> 1) & 1);      // (and the latents are there)
                if (!ok) break;
                const uint32_t lo = c_lo0 + so * (kStageBytes >> 4);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    ok = wait(&o_free[h], (i & 1) ^ 1);
                    if (!ok) break;
                    ptx::tc_fence_after_sync();
#pragma unroll
                    for (int v = 0; v < 6; ++v)
#pragma unroll
                        for (int k4 = 0; k4 < kKeys / 16; ++k4)
                            ptx::mma_ts(tmem + kTmO + 64 * h, tmem + kTmS + (i & 1) * kTmSP + kPa[v] * 32 + k4 * 8,
                                        ptx::desc_of(lo + ((kPb[v] * kCPlane + h * kCBlock + k4 * 16 * 128) >> 4), c_hi), idesc_o,
                                        (v | k4) ? 1u : 0u);
                    ptx::tc_commit(&o_full[h]);
                }
                if (!ok) break;
                so = so + 1 == kStages ? 0 : so + 1;
                if (i + 2 < n_my) scores(i + 2);
            }
            // tensor memory is freed below: nothing may be on its way there, also where others give up behind this thread's last wait
            ptx::tc_commit(drain_bar);
            ptx::mbar_wait_drain(drain_bar, 0, drain_flag);
        }
        __syncwarp();
        if constexpr (SW > 1) {
            ptx::cluster_arrive(); ptx::cluster_wait();
            ptx::cluster_arrive(); ptx::cluster_wait();
        }
    } else if (warp < kAddWarp0) {
        ptx::set_max_regs_inc<kSoftRegs>();
        const int quarter = warp & 3, w = (warp - kSoftWarp0) >> 2;          // TMEM lanes; this warpgroup's tiles
        const int row = quarter * 32 + lane;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        {   // pieces of Q: this warpgroup's 32 elements of the row
            const ulonglong2* src = reinterpret_cast<const ulonglong2*>(q + (((size_t)b * d.n_q + g) * d.N + t0 + (row < rows ? row : 0)) * kDh + 32 * w);
            uint32_t pc[3][16];
            uint32_t rest = 0u;
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                ulonglong2 e = __ldg(src + v);
                if (row >= rows) e = make_ulonglong2(0ull, 0ull);
                const Pieces s = split4(e.x, e.y);
                rest |= s.rest;
#pragma unroll
                for (int p = 0; p < 3; ++p) { pc[p][2 * v] = s.p[p].x; pc[p][2 * v + 1] = s.p[p].y; }
            }
#pragma unroll
            for (int p = 0; p < 3; ++p) ptx::tmem_st16(tmem + kTmQ + lane_base + p * 32 + 16 * w, pc[p]);
            ptx::tmem_wait_st();
            if ((rest & 0xffffu) != 0u && is_odd_row(reinterpret_cast<const float*>(src) - 32 * w, kDh)) atomicOr(&odd_rows[quarter], 1u << lane);
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(q_full);
        }
        {   // (all tiles of the item, also those of the cluster's other CTAs)
            ptx::grid_dependency_wait();
            const int all_tiles = (d.Nk + kKeys - 1) / kKeys;
            const int32_t* fk = first_odd + (size_t)(b * d.n_k + kg) * all_tiles;
            const int32_t* fc = first_odd + (size_t)(d.B * d.n_k + b * d.n_c + cg) * all_tiles;
            int first = INT32_MAX;
            for (int i = threadIdx.x - 32 * kSoftWarp0; i < n_tiles; i += 256) first = min(first, min(__ldcg(fk + i), __ldcg(fc + i)));
            if (first != INT32_MAX) atomicMin(odd_key, first);
        }
        const float scale2 = d.scale * 1.4426950408889634f;                  // scores, maxima in powers of two
        const int live = d.causal ? min(t0 + row + off + 1, d.Nk) : d.Nk;    // keys of this row
        float m = -INFINITY, l = 0.f;
        // (a wait that has given up makes every later one return at once: the loops run to their end on meaningless data)
        for (int i = w; i < n_my; i += 2) {
            const int j0 = (rank + SW * i) * kKeys;
            wait(&s_full[w], (i >> 1) & 1);
            __syncwarp();
            ptx::tc_fence_after_sync();
            const int st = i % kStages;
            const uint32_t st_ph = (i / kStages) & 1;
            if (lane == 0) ptx::mbar_arrive(&k_empty[st]);
            uint32_t sv[2][32];
            ptx::tmem_ld32(tmem + kTmS + lane_base + w * kTmSP, sv[0]);
            ptx::tmem_ld32(tmem + kTmS + lane_base + w * kTmSP + 32, sv[1]);
            ptx::tmem_wait_ld();
            if (__any_sync(0xffffffffu, j0 + kKeys > live)) {
#pragma unroll
                for (int e = 0; e < kKeys; ++e)
                    if (j0 + e >= live) sv[e >> 5][e & 31] = 0xff800000u;
            }
            float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
            for (int e = 0; e < kKeys; e += 8)
#pragma unroll
                for (int x = 0; x < 4; ++x)
                    mx[x] = ptx::max3(mx[x], __uint_as_float(sv[e >> 5][(e & 31) + 2 * x]), __uint_as_float(sv[e >> 5][(e & 31) + 2 * x + 1]));
            const float m_new = fmaxf(m, fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * scale2);
            const float ref = m_new == -INFINITY ? 0.f : m_new;              // (nothing but masked keys so far)
            const float alpha = m_new == m ? 1.f : exp2f(m - ref);
            m = m_new;
            float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int e = 0; e < kKeys; ++e) {
                const float p = exp2f(fmaf(__uint_as_float(sv[e >> 5][e & 31]), scale2, -ref));
                sv[e >> 5][e & 31] = __float_as_uint(p);
                sum[e & 3] += p;
            }
            l = fmaf(l, alpha, (sum[0] + sum[1]) + (sum[2] + sum[3]));
            // (P of i - 2 was read before the scores of i came; the adding warps are through with the scale of i - 4)
            ref_s[(i & 3) * kRows + row] = m_new;
#pragma unroll
            for (int p = 0; p < 3; ++p) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint32_t pc[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const float a = __uint_as_float(sv[h][2 * e]), bb = __uint_as_float(sv[h][2 * e + 1]);
                        pc[e] = ptx::cvt_bf16x2(a, bb);
                        if (p < 2) {
                            float x, y;
                            ptx::f32x2_split(ptx::sub2(ptx::f32x2(a, bb), ptx::f32x2(__uint_as_float(pc[e] << 16), __uint_as_float(pc[e] & 0xffff0000u))), x, y);
                            sv[h][2 * e] = __float_as_uint(x);
                            sv[h][2 * e + 1] = __float_as_uint(y);
                        }
                    }
                    ptx::tmem_st16(tmem + kTmS + lane_base + w * kTmSP + p * 32 + h * 16, pc);
                }
            }
            ptx::tmem_wait_st();
            ptx::tc_fence_before_sync();
            wait(&c_full[st], st_ph);
            __syncwarp();
            if (lane == 0 && !(i == 0 && quarter == 0 && rank == 0 && c_wait.withhold != 0)) ptx::mbar_arrive(&p_full[w]);
        }
        fin_m[w * kRows + row] = m;
        fin_l[w * kRows + row] = l;
        ptx::named_sync(1, 512);         // maxima and row sums are there
        if constexpr (SW > 1) {
            ptx::cluster_arrive(); ptx::cluster_wait();
            ptx::cluster_arrive(); ptx::cluster_wait();
        }
    } else {
        ptx::set_max_regs_inc<kAddRegs>();
        uint64_t acc[kCols / 4];
        float R = -INFINITY, lsum;
        const int quarter = warp & 3, half = (warp - kAddWarp0) >> 2, row = quarter * 32 + lane;
        const uint32_t o_tmem = tmem + kTmO + ((uint32_t)(quarter * 32) << 16) + half * (kCols / 2);
#pragma unroll
        for (int e = 0; e < kCols / 4; ++e) acc[e] = 0ull;
        for (int i = 0; i < n_my; ++i) {
            wait(&o_full[half], i & 1);
            __syncwarp();
            if (half == 1 && lane == 0) ptx::mbar_arrive(&c_empty[i % kStages]);
            ptx::tc_fence_after_sync();
            const float r = ref_s[(i & 3) * kRows + row];
            const float R_new = fmaxf(R, r);
            const float fa = R == R_new || R == -INFINITY ? 1.f : exp2f(R - R_new);
            const float fb = r == R_new ? 1.f : r == -INFINITY ? 0.f : exp2f(r - R_new);
            R = R_new;
            if (__any_sync(0xffffffffu, fa != 1.f)) {
                const uint64_t fa2 = ptx::f32x2(fa, fa);
#pragma unroll
                for (int e = 0; e < kCols / 4; ++e) acc[e] = ptx::mul2(acc[e], fa2);
            }
            const uint64_t fb2 = ptx::f32x2(fb, fb);
#pragma unroll
            for (int ch = 0; ch < kCols / 2 / 16; ++ch) {
                uint32_t v[16];
                ptx::tmem_ld16(o_tmem + ch * 16, v);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    acc[ch * 8 + e] = ptx::fma2(ptx::f32x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])), fb2, acc[ch * 8 + e]);
            }
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&o_free[half]);
        }
        ptx::named_sync(1, 512);         // maxima and row sums are there
        {
            const float m0 = fin_m[row], m1 = fin_m[kRows + row];
            lsum = (m0 == -INFINITY ? 0.f : fin_l[row] * exp2f(m0 - R)) + (m1 == -INFINITY ? 0.f : fin_l[kRows + row] * exp2f(m1 - R));
        }
        if constexpr (SW > 1) {
            // the other CTAs' sums, maxima and row sums go to CTA 0, into the ring's memory
            constexpr uint32_t kPart = kRows * kCols * 4, kStats = 3 * kPart;
            ptx::cluster_arrive();       // nobody uses the ring any more
            ptx::cluster_wait();
            if (rank > 0) {
                const uint32_t dst = ptx::map_to_cta(ptx::smem_addr(smem), 0) + (rank - 1) * kPart + (half * 16 * kRows + row) * 16;
#pragma unroll
                for (int v = 0; v < 16; ++v) ptx::st_cluster_v2_b64(dst + v * kRows * 16, acc[2 * v], acc[2 * v + 1]);
                if (half == 0) {
                    const uint32_t st = ptx::map_to_cta(ptx::smem_addr(smem), 0) + kStats + ((rank - 1) * 2 * kRows + row) * 4;
                    ptx::st_cluster_u32(st, __float_as_uint(R));
                    ptx::st_cluster_u32(st + kRows * 4, __float_as_uint(lsum));
                }
            }
            ptx::cluster_arrive();
            ptx::cluster_wait();
            if (rank == 0) {
                const float* stats = reinterpret_cast<const float*>(smem + kStats);
                float R_new = R;
#pragma unroll
                for (int r = 0; r < SW - 1; ++r) R_new = fmaxf(R_new, stats[r * 2 * kRows + row]);
                const float f0 = R == -INFINITY ? 0.f : exp2f(R - R_new);
                lsum *= f0;
                const uint64_t f02 = ptx::f32x2(f0, f0);
#pragma unroll
                for (int e = 0; e < kCols / 4; ++e) acc[e] = ptx::mul2(acc[e], f02);
#pragma unroll
                for (int r = 0; r < SW - 1; ++r) {
                    const float mr = stats[r * 2 * kRows + row];
                    const float f = mr == -INFINITY ? 0.f : exp2f(mr - R_new);
                    lsum = fmaf(stats[(2 * r + 1) * kRows + row], f, lsum);
                    const uint64_t f2 = ptx::f32x2(f, f);
                    const uint8_t* src = smem + r * kPart + (half * 16 * kRows + row) * 16;
#pragma unroll
                    for (int v = 0; v < 16; ++v) {
                        const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(src + v * kRows * 16);
                        acc[2 * v] = ptx::fma2(e.x, f2, acc[2 * v]);
                        acc[2 * v + 1] = ptx::fma2(e.y, f2, acc[2 * v + 1]);
                    }
                }
            }
        }
        if (rank == 0) {
            ptx::named_sync(2, 256);     // the parts have been read: the output passes through the same memory
            const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
            uint8_t* stage = smem + (warp - kAddWarp0) * (kCols / 2 * 32 * 4);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint8_t* box = stage + h * 4096 + lane * 128;
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    float y[4];
                    ptx::f32x2_split(acc[h * 16 + 2 * v], y[0], y[1]);
                    ptx::f32x2_split(acc[h * 16 + 2 * v + 1], y[2], y[3]);
                    *reinterpret_cast<float4*>(box + ((v ^ (lane & 7)) << 4)) = make_float4(y[0] * inv, y[1] * inv, y[2] * inv, y[3] * inv);
                }
                ptx::fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && quarter * 32 < rows) {
                    ptx::tma_store_3d(&tm_l, stage + h * 4096, slice * kCols + half * (kCols / 2) + 32 * h, t0 + quarter * 32, g * d.B + b);
                    ptx::bulk_commit_group();
                }
            }
            ptx::bulk_wait_group_read_all();
            const int first = *odd_key;
            if (first < n_keys || (odd_rows[0] | odd_rows[1] | odd_rows[2] | odd_rows[3]) != 0) {
                ptx::bulk_wait_group_all();
                ptx::named_sync(2, 256);
                redo_rows(d, q, k, c, o_lat, t0, slice, g, b, first, odd_rows, reinterpret_cast<float*>(smem), threadIdx.x - 32 * kAddWarp0);
            }
        }
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem, 512);
    if (threadIdx.x == 0 && *abort_flag) raise_status(status_word, GTA_ERR_TIMEOUT);
}

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

gta_status_t sm100_attention_f32_debug_wait(unsigned long long limit_ns, int withhold_first_arrive) {
    const WaitHook w = {limit_ns ? limit_ns : ptx::kWaitLimitNs, withhold_first_arrive ? 1 : 0};
    if (cudaMemcpyToSymbol(c_wait, &w, sizeof(w)) == cudaSuccess) return GTA_OK;
    cudaGetLastError();
    return GTA_ERR_CUDA;
}

bool sm100_attention_f32_supported(const Dims& d) {
    const long long ctas = 4ll * ((d.N + kRows - 1) / kRows) * (d.d_l / kCols) * d.n_q * d.B;
    const long long tiles = (long long)((d.Nk + kKeys - 1) / kKeys) * d.B * (d.n_k + d.n_c);
    return sm100_attention_f32_shape(d) && ctas <= INT32_MAX && tiles <= INT32_MAX;
}

bool sm100_attention_f32_shape(const Dims& d) { return d.d_h == kDh && d.d_l % kCols == 0; }


size_t sm100_attention_f32_scratch(const Dims& d) {
    const size_t rows = (size_t)d.B * d.Nk, tiles = ((size_t)d.Nk + kKeys - 1) / kKeys;
    return align256(6 * rows * d.n_k * d.d_h) + align256(6 * rows * d.n_c * d.d_l) + align256(4 * tiles * d.B * (d.n_k + d.n_c));
}

cudaError_t launch_sm100_attention_f32(const Dims& d, const float* q, const float* k, const float* c, float* o_lat, void* scratch,
                                       int32_t* status_word, cudaStream_t stream, int split, int* launches) {
    uint8_t* k_planes = static_cast<uint8_t*>(scratch);
    uint8_t* c_planes = k_planes + align256(6 * (size_t)d.B * d.Nk * d.n_k * d.d_h);
    int32_t* first_odd = reinterpret_cast<int32_t*>(c_planes + align256(6 * (size_t)d.B * d.Nk * d.n_c * d.d_l));
    CUtensorMap tm_k, tm_c, tm_l;
    {
        const uint64_t dk[3] = {(uint64_t)kDh, (uint64_t)d.Nk, 3ull * d.B * d.n_k}, dc[3] = {(uint64_t)d.d_l, (uint64_t)d.Nk, 3ull * d.B * d.n_c};
        const uint64_t dl[3] = {(uint64_t)d.d_l, (uint64_t)d.N, (uint64_t)d.n_q * d.B};
        const uint32_t tile[3] = {64, kKeys, 1}, box[3] = {32, 32, 1};
        if (!make_bf16_map(&tm_k, k_planes, 3, dk, tile) || !make_bf16_map(&tm_c, c_planes, 3, dc, tile) ||
            !make_f32_map(&tm_l, o_lat, 3, dl, box, true))
            return cudaErrorInvalidValue;
    }
    const int key_tiles = (d.Nk + kKeys - 1) / kKeys, row_tiles = (d.N + kRows - 1) / kRows, slices = d.d_l / kCols;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3((unsigned)key_tiles * d.B * (d.n_k + d.n_c));
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t err = cudaLaunchKernelEx(&cfg, split_rows_kernel, d, k, c, k_planes, c_planes, first_odd, key_tiles);
    if (err != cudaSuccess) return err;
    const auto go = [&](auto sw) {
        constexpr int SW = decltype(sw)::value;
        auto kern = sm100_attention_f32_kernel<SW>;
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        if (e != cudaSuccess) return e;
        cfg.gridDim = dim3((unsigned)SW * row_tiles * slices * d.n_q * d.B);
        cfg.blockDim = dim3(kThreads);
        cfg.dynamicSmemBytes = kSmem;
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = SW;
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = SW > 1 ? 2 : 1;
        return cudaLaunchKernelEx(&cfg, kern, tm_k, tm_c, tm_l, d, q, k, c, o_lat, (const int32_t*)first_odd, row_tiles, slices, status_word);
    };
    err = split == 4 ? go(std::integral_constant<int, 4>{}) : split == 2 ? go(std::integral_constant<int, 2>{}) : go(std::integral_constant<int, 1>{});
    if (err == cudaSuccess) *launches += 2;
    return err;
}

}  // namespace gta
