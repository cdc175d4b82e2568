// fp32 decoder + gate on the tensor cores:
//     out_i = (L_{q(i)} W_P,i) (.) Sigmoid(X W_G,i)          (Sec. 3.3, reformulated equation)
//
// Every fp32 operand is the sum of three bf16 pieces, exactly from 2^-110 on (8 significant bits each, rounded to nearest, the
// rest handed on); six of the nine products of pieces are taken (what is left out, of which two can reach 2^-25 of a product
// each, is below 2^-24 of it, 2^-26.5 rms), each exact in the tensor core, which adds them in fp32 but cuts where fp32
// arithmetic rounds.  So a sum stays in tensor memory for 32 elements of the contraction only, small products first, and is
// added up in registers (rounded) from there: against 64 bits the result is closer than the FMA chain of the plain-ALU kernel.
//
// CTA pairs, one item of 256 token rows x NT output columns of one attention map per pair.
//   warp 0       (leader CTA) issues the MMAs: twelve per stage, two accumulators in tensor memory in turn.
//   warp 1       brings the fp32 operands in by TMA, two or three blocks of 32 k ahead of the
//   warps 4-11   that split them and store the pieces into a ring of swizzled stages.
//   warps 12-19  add finished accumulators to their registers: a lane is a token row, a warp has half of the item's columns.
// The gates come first (they need nothing of the attention kernel, behind which this kernel is launched) and then wait in one
// of the two accumulators, while the decoded values take the other.
//
// What bounds it: a stage of 256 x 256 x 32 takes 1536 cycles of MMAs and 208 KB of shared-memory traffic (raw blocks in and
// out, pieces in, operands read once per product: 1664 cycles); measured 1800.
//
// An element that is infinite, not a number or rounds to infinity in bf16 makes its row or column of the item not a number
// (0 x infinity); the splitting threads see it, and where it is an infinity or a large number those rows and columns are done again
// with plain FMAs.  So are rows and columns whose elements are all too small for pieces (kPiecesFloor).
#include "gta_sm100.cuh"

#include <cuda.h>

#include "sm100_ptx.cuh"
#include "tma_host.cuh"

namespace gta {

namespace {

constexpr int kSplitWarp0 = 4, kSplitThreads = 256, kAddWarp0 = 12, kAddWarps = 8, kThreads = 640;
constexpr int kBoth = kSplitThreads + 32 * kAddWarps;
// registers: 640 threads start with 96 each (61440), which the warpgroups share out anew: 128 x 48 + 256 x 64 + 256 x 152
constexpr int kIssueRegs = 48, kSplitRegs = 64, kAddRegs = 152;
constexpr int kTileM = 128, kBlockK = 32;      // token rows of a CTA; elements of the contraction per stage
constexpr uint32_t kRawBlock = kBlockK * 64 * 4;         // 64 columns of a block of the weights, in fp32
constexpr uint32_t kAPlane = kTileM * kBlockK * 2;      // one piece of the A tile: rows of 64 bytes

template <int NT> struct Cfg {
    static constexpr int kCols = NT / 2;                         // columns that a CTA stages
    static constexpr uint32_t kBPlane = kBlockK * kCols * 2;     // blocks of 64 columns, [k][128 bytes]
    static constexpr uint32_t kStageBytes = 3 * (kAPlane + kBPlane);
    // 16-byte pieces of a block, per splitting thread: rows of the A tile, then k-rows of the weight tile
    static constexpr int kAPieces = kTileM * kBlockK / 4 / kSplitThreads, kBPieces = kBlockK * kCols / 4 / kSplitThreads;
    static constexpr uint32_t kRawBytes = (kAPieces + kBPieces) * kSplitThreads * 16;
    static constexpr int kStages = NT == 256 ? 3 : 4, kRaw = NT == 256 ? 2 : 3;
    static constexpr uint32_t kBarOffset = kStages * kStageBytes + kRaw * kRawBytes;
    static constexpr uint32_t kSmem = kBarOffset + 1024 /* barriers, flags */ + 1024 /* alignment */;
    static_assert(kSmem <= 227 * 1024, "shared memory of a CTA");
};

// Sigmoid to an ulp or two: an exponential, a reciprocal of 1 ulp and a Newton step (a denominator near the end of the range
// stays without it: 1 - d r would not be a number).
__device__ __forceinline__ float sigmoid(float z) {
    const float den = 1.f + expf(-z), r = ptx::rcp_approx(den);
    return den < 1e37f ? fmaf(r, fmaf(-den, r, 1.f), r) : r;
}

// What a CTA works on
struct Block {
    int g, n0, n_cols, map_cols, rows;     // map, first column inside it, columns, columns of the map, token rows
    long long m0;                          // first token row
};
template <int NT> __device__ __forceinline__ Block block_of(const Dims& d, int row_tiles, int col_tiles, uint32_t block) {
    // items of one column block and map follow one another: their CTAs read the same weights
    const int pr = block >> 1, rt = pr % row_tiles, ct = pr / row_tiles % col_tiles;
    const long long M = (long long)d.B * d.N;
    Block w;
    w.g = pr / (row_tiles * col_tiles);
    w.map_cols = d.n_h / d.n_q * d.d_h;
    w.m0 = (long long)rt * 2 * kTileM + (block & 1) * kTileM;
    w.rows = (int)(M - w.m0 < 0 ? 0 : M - w.m0 < kTileM ? M - w.m0 : kTileM);
    w.n0 = ct * NT;
    w.n_cols = min(NT, w.map_cols - w.n0);
    return w;
}

// What the splitting threads found: rows and groups of four columns to be done again (`bad`), and those that hold an element which
// its pieces do not add up to (`small`).
template <int NT> struct Marks {
    uint8_t row_bad[kTileM], col_bad[NT / 4], row_small[kTileM], col_small[NT / 4];
};

// The rows and columns that hold an element which the pieces cannot: plain FMAs, by the adding warps.
template <int NT>
__device__ __forceinline__ void redo(const Dims& d, const float* o_lat, const float* x, const float* w_p, const float* w_g, float* out,
                                     int row_tiles, int col_tiles, uint32_t block, Marks<NT>* marks, float* smem) {
    const Block w = block_of<NT>(d, row_tiles, col_tiles, block);
    const size_t ldw = (size_t)d.n_h * d.d_h;
    const int tid = threadIdx.x - 32 * kAddWarp0, warp = tid >> 5, lane = tid & 31;
    uint8_t *row_bad = marks->row_bad, *col_bad = marks->col_bad;
    for (int r = warp; r < w.rows; r += kAddWarps)
        if (marks->row_small[r] && !row_bad[r]) {
            const float* xr = x + (w.m0 + r) * d.H;
            const float* lr = o_lat + ((size_t)w.g * d.B * d.N + w.m0 + r) * d.d_l;
            float mx = 0.f, ml = 0.f;
            for (int k = lane; k < d.H; k += 32) mx = fmaxf(mx, fabsf(xr[k]));
            for (int k = lane; k < d.d_l; k += 32) ml = fmaxf(ml, fabsf(lr[k]));
            if (fminf(warp_max(mx), warp_max(ml)) < kPiecesFloor) row_bad[r] = 1;
        }
    for (int c4 = warp; 4 * c4 < w.n_cols; c4 += kAddWarps)
        if (marks->col_small[c4] && !col_bad[c4]) {
            const int f = w.n0 + 4 * c4, head = w.g * (d.n_h / d.n_q) + f / d.d_h;       // (four columns of one head)
            const float* wg = w_g + (size_t)w.g * w.map_cols + f;
            const float* wp = w_p + (size_t)head * d.d_l * d.d_h + f % d.d_h;
            float4 mg = make_float4(0.f, 0.f, 0.f, 0.f), mp = mg;
            const auto larger = [](float4& m, const float4 v) {
                m.x = fmaxf(m.x, fabsf(v.x)); m.y = fmaxf(m.y, fabsf(v.y)); m.z = fmaxf(m.z, fabsf(v.z)); m.w = fmaxf(m.w, fabsf(v.w));
            };
            for (int k = lane; k < d.H; k += 32) larger(mg, *reinterpret_cast<const float4*>(wg + k * ldw));
            for (int k = lane; k < d.d_l; k += 32) larger(mp, *reinterpret_cast<const float4*>(wp + (size_t)k * d.d_h));
            const float least = fminf(fminf(fminf(warp_max(mg.x), warp_max(mg.y)), fminf(warp_max(mg.z), warp_max(mg.w))),
                                      fminf(fminf(warp_max(mp.x), warp_max(mp.y)), fminf(warp_max(mp.z), warp_max(mp.w))));
            if (least < kPiecesFloor) col_bad[c4] = 1;
        }
    ptx::named_sync(3, 32 * kAddWarps);
    // kPass rows after kPass rows, where one of them or one of the columns is to be done again: 32 elements of the contraction at a time
    // through the ring's memory, two slabs in turn, four rows x four columns to a thread.  (Few registers: all roles come here, so the
    // compiler has the 48 of the smallest.  A row and a column at a time, with strided loads, an infinity in all rows of X took 9.5 ms
    // for 2 x 1500 tokens of the 1B layer, 0.9 now, 0.42 where the plain-ALU kernels take the whole call; eight rows a thread, mostly in
    // local memory, 2.1.)
    constexpr int kThr = 32 * kAddWarps, kGroups = kThr / (NT / 4), kPass = 4 * kGroups, kSlab = 32, kLd = kSlab + 4;
    constexpr int kSlabFloats = kSlab * NT + kPass * kLd;
    float* z_s = smem + 2 * kSlabFloats;        // [kPass][NT]; slabs: weights [kSlab][NT], rows [kPass][kLd]
    static_assert((2 * kSlabFloats + kPass * NT) * 4 <= Cfg<NT>::kBarOffset, "in the ring's memory");
    int n_col = 0;
    for (int c4 = 0; 4 * c4 < w.n_cols; ++c4) n_col += col_bad[c4];
    const bool any_col = n_col > 4;             // (fewer columns one by one, below)
    const int cg = tid % (NT / 4), rg = tid / (NT / 4), f = w.n0 + min(4 * cg, w.n_cols - 4), head = w.g * (d.n_h / d.n_q) + f / d.d_h;
    const auto copy16 = [](float* dst, const float* src, bool there) {      // zeros where there is nothing
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ptx::smem_addr(dst)), "l"(src), "r"(there ? 16 : 0) : "memory");
    };
    for (int r0 = 0; r0 < w.rows; r0 += kPass) {
        bool any = any_col;
        for (int r = r0; r < min(r0 + kPass, w.rows); ++r) any |= row_bad[r] != 0;
        if (!any) continue;
        float acc[4][4];
        // col: this thread's four columns
        const auto contract = [&](const float* rows, int K, const float* col, size_t ld) {
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
            const auto fetch = [&](int k0) {
                float* w_s = smem + (k0 / kSlab & 1) * kSlabFloats;
                for (int k = rg; k < kSlab; k += kGroups) copy16(w_s + k * NT + 4 * cg, col + (k0 + k < K ? (size_t)(k0 + k) * ld : 0), k0 + k < K);
                for (int i = tid; i < kPass * (kSlab / 4); i += kThr) {
                    const int r = i / (kSlab / 4), e = k0 + 4 * (i % (kSlab / 4));
                    copy16(w_s + kSlab * NT + r * kLd + e - k0, rows + (size_t)min(r0 + r, w.rows - 1) * K + (e < K ? e : 0), e < K);
                }
                asm volatile("cp.async.commit_group;" ::: "memory");
            };
            ptx::named_sync(3, kThr);                               // (the slabs before have been used)
            fetch(0);
            for (int k0 = 0; k0 < K; k0 += kSlab) {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
                ptx::named_sync(3, kThr);
                if (k0 + kSlab < K) fetch(k0 + kSlab);
                const float* w_s = smem + (k0 / kSlab & 1) * kSlabFloats + 4 * cg;
                const float* a_s = smem + (k0 / kSlab & 1) * kSlabFloats + kSlab * NT + 4 * rg * kLd;
#pragma unroll 1
                for (int k = 0; k < kSlab; k += 2) {
                    float2 x2[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) x2[i] = *reinterpret_cast<const float2*>(a_s + i * kLd + k);
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const float4 v = *reinterpret_cast<const float4*>(w_s + (k + u) * NT);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float xi = u == 0 ? x2[i].x : x2[i].y;
                            acc[i][0] = fmaf(xi, v.x, acc[i][0]);
                            acc[i][1] = fmaf(xi, v.y, acc[i][1]);
                            acc[i][2] = fmaf(xi, v.z, acc[i][2]);
                            acc[i][3] = fmaf(xi, v.w, acc[i][3]);
                        }
                    }
                }
            }
        };
        contract(x + w.m0 * d.H, d.H, w_g + (size_t)w.g * w.map_cols + f, ldw);
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(z_s + (4 * rg + i) * NT + 4 * cg) = make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]);
        contract(o_lat + ((size_t)w.g * d.B * d.N + w.m0) * d.d_l, d.d_l, w_p + (size_t)head * d.d_l * d.d_h + f % d.d_h, d.d_h);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = r0 + 4 * rg + i;
            if (r < w.rows && 4 * cg < w.n_cols && (row_bad[r] | col_bad[cg]) != 0) {
                const float4 z = *reinterpret_cast<const float4*>(z_s + (4 * rg + i) * NT + 4 * cg);
                *reinterpret_cast<float4*>(out + (w.m0 + r) * ldw + (size_t)w.g * w.map_cols + w.n0 + 4 * cg) =
                    make_float4(acc[i][0] * (1.f / (1.f + expf(-z.x))), acc[i][1] * (1.f / (1.f + expf(-z.y))),
                                acc[i][2] * (1.f / (1.f + expf(-z.z))), acc[i][3] * (1.f / (1.f + expf(-z.w))));
            }
        }
    }
    if (any_col || n_col == 0) return;
    const auto again = [&](int r, int c) {
        const long long m = w.m0 + r;
        const int fc = w.n0 + c, hd = w.g * (d.n_h / d.n_q) + fc / d.d_h;
        const float* xr = x + m * d.H;
        const float* wg = w_g + (size_t)w.g * w.map_cols + fc;
        float z = 0.f, y = 0.f;
        for (int k = 0; k < d.H; ++k) z = fmaf(xr[k], wg[k * ldw], z);
        const float* lr = o_lat + ((size_t)w.g * d.B * d.N + m) * d.d_l;
        const float* wp = w_p + (size_t)hd * d.d_l * d.d_h + fc % d.d_h;
        for (int k = 0; k < d.d_l; ++k) y = fmaf(lr[k], wp[(size_t)k * d.d_h], y);
        out[m * ldw + (size_t)w.g * w.map_cols + fc] = y * (1.f / (1.f + expf(-z)));
    };
    for (int c4 = 0; 4 * c4 < w.n_cols; ++c4)
        if (col_bad[c4])
            for (int e = tid; e < 4 * w.rows; e += kThr) again(e >> 2, 4 * c4 + (e & 3));
}

// Test hook of the bounded waits (gta_debug_attention_wait): their time limit, and a switch that keeps the first accumulator's
// completion from the adding warps.
struct WaitHook { unsigned long long limit_ns; int withhold; };
static __constant__ WaitHook c_wait = {ptx::kWaitLimitNs, 0};

template <int NT>
__global__ void __launch_bounds__(kThreads, 1)
sm100_decoder_f32_kernel(const __grid_constant__ CUtensorMap tm_l, const __grid_constant__ CUtensorMap tm_x,
                         const __grid_constant__ CUtensorMap tm_wp, const __grid_constant__ CUtensorMap tm_wg,
                         const __grid_constant__ CUtensorMap tm_out, Dims d, const float* __restrict__ o_lat,
                         const float* __restrict__ x, const float* __restrict__ w_p, const float* __restrict__ w_g, float* out,
                         int row_tiles, int col_tiles, int32_t* status_word) {
    using C = Cfg<NT>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* raw = smem + C::kStages * C::kStageBytes;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + C::kBarOffset);     // leader CTA: 16 warps arrive
    uint64_t* empty_bar = full_bar + C::kStages;                                 // both CTAs
    uint64_t* raw_full = empty_bar + C::kStages;                                 // own CTA
    uint64_t* raw_empty = raw_full + C::kRaw;                                    // own CTA: 8 warps arrive
    uint64_t* acc_full = raw_empty + C::kRaw;                                    // both CTAs, [2]
    uint64_t* acc_free = acc_full + 2;                                           // leader CTA, [2]: 16 warps arrive
    uint64_t* drain_bar = acc_free + 2;                                          // leader CTA: an unwinding issuer's
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* drain_flag = abort_flag + 1;
    uint32_t* any_bad = tmem_slot + 3;
    int* armed = reinterpret_cast<int*>(tmem_slot + 4);                          // blocks that were asked for
    Marks<NT>* marks = reinterpret_cast<Marks<NT>*>(smem + C::kBarOffset + 256);
    static_assert(256 + sizeof(Marks<NT>) <= 1024 && sizeof(Marks<NT>) % 4 == 0, "room behind the barriers");

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = ptx::cluster_ctarank();
    const int n_g = (d.H + kBlockK - 1) / kBlockK, n_it = n_g + (d.d_l + kBlockK - 1) / kBlockK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::kStages; ++s) { ptx::mbar_init(&full_bar[s], 2 * kSplitThreads / 32); ptx::mbar_init(&empty_bar[s], 1); }
        for (int r = 0; r < C::kRaw; ++r) { ptx::mbar_init(&raw_full[r], 1); ptx::mbar_init(&raw_empty[r], kSplitThreads / 32); }
        for (int s = 0; s < 2; ++s) { ptx::mbar_init(&acc_full[s], 1); ptx::mbar_init(&acc_free[s], 2 * kAddWarps); }
        ptx::mbar_init(drain_bar, 1);
        *abort_flag = 0;
        *drain_flag = 0;
        *any_bad = 0;
        ptx::fence_mbar_init();
    }
    if (threadIdx.x < sizeof(Marks<NT>) / 4) reinterpret_cast<uint32_t*>(marks)[threadIdx.x] = 0;
    if (warp == 0) ptx::tmem_alloc_pair(tmem_slot, 2 * NT);
    ptx::tc_fence_before_sync();
    __syncthreads();
    ptx::cluster_arrive();         // the peer's barriers exist before anything is signalled to them
    ptx::cluster_wait();
    ptx::tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_slot;
    // Accumulators take turns up to the gates' last; it keeps the gates, and the decoded values have the other to themselves.
    const auto buf_of = [&](int it) { return (it < n_g ? it : n_g) & 1; };
    const auto use_of = [&](int it) { return it < n_g ? it >> 1 : (n_g >> 1) + (it - n_g); };      // how often it was used before

    const auto wait = [&](uint64_t* bar, uint32_t parity) { return ptx::mbar_wait_sleep(bar, parity, abort_flag, 0, c_wait.limit_ns); };

    if (warp < kSplitWarp0) {
        ptx::set_max_regs_dec<kIssueRegs>();
        if (warp == 0 && rank == 0 && ptx::elect_one()) {
            const uint32_t idesc = ptx::make_idesc_bf16(2 * kTileM, NT, 0, 1);   // A K-major, B MN-major
            const uint64_t a_desc = ptx::make_smem_desc_sw64(ptx::smem_addr(smem), 512);
            const uint64_t b_desc = ptx::make_smem_desc(ptx::smem_addr(smem) + 3 * kAPlane, kBlockK * 128, 1024);
            const uint32_t a_lo0 = (uint32_t)a_desc, a_hi = (uint32_t)(a_desc >> 32), b_lo0 = (uint32_t)b_desc, b_hi = (uint32_t)(b_desc >> 32);
            bool ok = true;
            int s = 0;
            uint32_t ph = 0;
            for (int it = 0; it < n_it; ++it, s = (s + 1 == C::kStages) ? 0 : s + 1, ph ^= (s == 0)) {
                const int buf = buf_of(it);
                if (it == n_g) ptx::grid_dependency_wait();      // (every waiting role: how long the attention kernel takes is not bounded
                                                                 // by the waits' limit, and the CTA does not end before it)
                ok = wait(&acc_free[buf], (use_of(it) & 1) ^ 1) && wait(&full_bar[s], ph);
                if (!ok) break;
                ptx::mbar_try_wait_acquire_cluster(&full_bar[s], ph);    // (both CTAs' pieces, written by ordinary stores)
                ptx::tc_fence_after_sync();
                const uint32_t a_lo = a_lo0 + s * (C::kStageBytes >> 4), b_lo = b_lo0 + s * (C::kStageBytes >> 4);
                const uint32_t d_tmem = tmem_base + buf * NT;
                constexpr int kPa[6] = {2, 1, 0, 1, 0, 0}, kPb[6] = {0, 1, 2, 0, 1, 0};       // pieces, the smallest products first
#pragma unroll
                for (int u = 0; u < 6; ++u)
#pragma unroll
                    for (int k2 = 0; k2 < kBlockK / 16; ++k2)
                        ptx::mma_ss_pair(d_tmem, ptx::desc_of(a_lo + ((kPa[u] * kAPlane + k2 * 32) >> 4), a_hi),
                                         ptx::desc_of(b_lo + ((kPb[u] * C::kBPlane + k2 * 16 * 128) >> 4), b_hi), idesc, (u | k2) ? 1u : 0u);
                ptx::tc_commit_pair(&empty_bar[s], 3);
                if (it != 0 || c_wait.withhold == 0) ptx::tc_commit_pair(&acc_full[buf], 3);
            }
        }
        if (warp == 1 && ptx::elect_one()) {
            const Block w = block_of<NT>(d, row_tiles, col_tiles, blockIdx.x);
            ptx::prefetch_tensormap(&tm_x); ptx::prefetch_tensormap(&tm_wg);
            ptx::prefetch_tensormap(&tm_l); ptx::prefetch_tensormap(&tm_wp);
            const int col = w.g * w.map_cols + w.n0 + (int)rank * C::kCols;      // this CTA's first output column (of n_h d_h)
            const int m0 = (int)w.m0;
            int r = 0;
            uint32_t ph = 1;
            bool ok = true;
            int it = 0;
            for (; it < n_it; ++it) {
                ok = wait(&raw_empty[r], ph);
                if (!ok) break;
                const bool gate = it < n_g;
                const int k0 = (gate ? it : it - n_g) * kBlockK;
                uint8_t* dst = raw + r * C::kRawBytes;
                uint8_t* dst_w = dst + kTileM * kBlockK * 4;
                if (it == n_g) {                // L is the attention kernel's; X and the weights are older
                    ptx::grid_dependency_wait();
                    ptx::grid_launch_dependents();
                }
                ptx::mbar_arrive_expect_tx(&raw_full[r], C::kRawBytes);
                if (gate) {
                    ptx::tma_load_2d(dst, &tm_x, &raw_full[r], k0, m0);
                    for (int u = 0; u < C::kCols / 64; ++u) ptx::tma_load_2d(dst_w + u * kRawBlock, &tm_wg, &raw_full[r], col + 64 * u, k0);
                } else {
                    ptx::tma_load_3d(dst, &tm_l, &raw_full[r], k0, m0, w.g);
                    for (int u = 0; u < C::kCols / 64; ++u)
                        ptx::tma_load_3d(dst_w + u * kRawBlock, &tm_wp, &raw_full[r], (col + 64 * u) % d.d_h, k0, (col + 64 * u) / d.d_h);
                }
                r = r + 1 == C::kRaw ? 0 : r + 1;
                ph ^= r == 0;
            }
            *armed = it;
        }
    } else if (warp < kAddWarp0) {
        ptx::set_max_regs_dec<kSplitRegs>();
        const int tid = threadIdx.x - 32 * kSplitWarp0;
        // this thread's pieces: A row 32 i + tid / 8, elements 4 (tid % 8) of the block; of the i-th 16 k of the weights (64 columns
        // after 64 columns) k = tid / 16, columns 4 (tid % 16) of the 64
        const int a_row = tid >> 3, b_k = tid >> 4, b_vec = tid & 15;
        // four floats -> 8 bytes of each piece.  What two pieces leave of a number has eight bits, which are the upper half of its
        // word; the lower half of `odd` is not zero where one leaves more: it ends below bf16's range, or has no pieces
        uint32_t odd = 0u;
        auto split = [&](const ulonglong2 v, uint8_t* dst, uint32_t plane) {
            uint64_t r0 = v.x, r1 = v.y;
            float a, b, e, f;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                ptx::f32x2_split(r0, a, b);
                ptx::f32x2_split(r1, e, f);
                const uint32_t h0 = ptx::cvt_bf16x2(a, b), h1 = ptx::cvt_bf16x2(e, f);
                *reinterpret_cast<uint2*>(dst + p * plane) = make_uint2(h0, h1);
                r0 = ptx::sub2(r0, ptx::f32x2(__uint_as_float(h0 << 16), __uint_as_float(h0 & 0xffff0000u)));
                r1 = ptx::sub2(r1, ptx::f32x2(__uint_as_float(h1 << 16), __uint_as_float(h1 & 0xffff0000u)));
            }
            ptx::f32x2_split(r0, a, b);
            ptx::f32x2_split(r1, e, f);
            const uint32_t wa = __float_as_uint(a), wb = __float_as_uint(b), we = __float_as_uint(e), wf = __float_as_uint(f);
            *reinterpret_cast<uint2*>(dst + 2 * plane) = make_uint2(ptx::upper_halves(wa, wb), ptx::upper_halves(we, wf));
            odd |= wa | wb;
            odd |= we | wf;
        };
        auto note_odd = [&](const uint8_t* src) {
            auto is_odd = [](float v) { return fabsf(v) >= 3.38e38f; };         // (3.3895e38 is bf16's largest; what is not a number
                                                                               // makes the row or column none by itself)
            auto any_odd = [&](const float4 v) { return is_odd(v.x) || is_odd(v.y) || is_odd(v.z) || is_odd(v.w); };
            auto is_small = [](float v) { return v != 0.f && fabsf(v) < 0x1p-109f; };
            auto any_small = [&](const float4 v) { return is_small(v.x) || is_small(v.y) || is_small(v.z) || is_small(v.w); };
            for (int i = 0; i < C::kAPieces; ++i) {
                const float4 v = *reinterpret_cast<const float4*>(src + i * kSplitThreads * 16);
                if (any_odd(v)) { marks->row_bad[a_row + 32 * i] = 1; *any_bad = 1; }
                else if (any_small(v)) { marks->row_small[a_row + 32 * i] = 1; *any_bad = 1; }
            }
            for (int i = 0; i < C::kBPieces; ++i) {
                const float4 v = *reinterpret_cast<const float4*>(src + (C::kAPieces + i) * kSplitThreads * 16);
                const bool bad = any_odd(v);
                if (bad || any_small(v))
                    for (uint32_t r = 0; r < 2; ++r) {       // both CTAs have these columns
                        uint8_t* mark = (bad ? marks->col_bad : marks->col_small) + rank * (C::kCols / 4) + (i >> 1) * 16 + b_vec;
                        ptx::st_cluster_u8(ptx::map_to_cta(ptx::smem_addr(mark), r), 1);
                        ptx::st_cluster_u32(ptx::map_to_cta(ptx::smem_addr(any_bad), r), 1);
                    }
            }
        };
        // where the pieces go: A rows of 64 bytes (64-byte swizzle), weights [64 columns][k][128 bytes] (128-byte swizzle); rows 32 i
        // and k 16 i apart have the same swizzle
        const uint32_t a_dst = a_row * 64 + ((((tid & 7) >> 1) ^ ((a_row >> 1) & 3)) << 4) + 8 * (tid & 1);
        const uint32_t b_dst = 3 * kAPlane + b_k * 128 + (((b_vec >> 1) ^ (b_k & 7)) << 4) + 8 * (b_vec & 1);
        const uint32_t full_leader = ptx::map_to_cta(ptx::smem_addr(full_bar), 0);
        // (a wait that has given up makes every later one return at once: the loops run to their end on meaningless data)
        int s = 0, r = 0;
        uint32_t ph = 1, raw_ph = 0;
        for (int it = 0; it < n_it; ++it) {
            if (it == n_g) ptx::grid_dependency_wait();
            wait(&raw_full[r], raw_ph);
            wait(&empty_bar[s], ph);
            __syncwarp();
            const uint8_t* src = raw + r * C::kRawBytes + tid * 16;
            uint8_t* st = smem + s * C::kStageBytes;
            // (four loads ahead of the stores, which the compiler cannot move them across)
            ulonglong2 v[4];
            constexpr int kPieces = C::kAPieces + C::kBPieces;
#pragma unroll
            for (int i0 = 0; i0 < kPieces; i0 += 4) {
#pragma unroll
                for (int i = i0; i < i0 + 4 && i < kPieces; ++i) v[i & 3] = *reinterpret_cast<const ulonglong2*>(src + i * kSplitThreads * 16);
#pragma unroll
                for (int i = i0; i < i0 + 4 && i < kPieces; ++i)
                    if (i < C::kAPieces) split(v[i & 3], st + a_dst + i * 32 * 64, kAPlane);
                    else split(v[i & 3], st + b_dst + (i - C::kAPieces) * 16 * 128, C::kBPlane);
            }
            if ((odd & 0xffffu) != 0u) {
                note_odd(src);
                odd = 0u;
            }
            ptx::fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) {
                ptx::mbar_arrive_release_smem_cluster(full_leader + 8 * s);      // (the leader's issuing thread acquires the pieces)
                ptx::mbar_arrive(&raw_empty[r]);
            }
            s = s + 1 == C::kStages ? 0 : s + 1;
            ph ^= s == 0;
            r = r + 1 == C::kRaw ? 0 : r + 1;
            raw_ph ^= r == 0;
        }
        // the gates, in place, while the last decoded values are summed up (the adding warps, with their registers full, would take
        // 5 us more for a pair's 65536)
        ptx::named_sync(1, kBoth);
        ptx::tc_fence_after_sync();
        const uint32_t z_tmem = tmem_base + ((uint32_t)((warp & 3) * 32) << 16) + ((n_g - 1) & 1) * NT + ((warp - kSplitWarp0) >> 2) * C::kCols;
#pragma unroll 1
        for (int ch = 0; ch < C::kCols / 16; ++ch) {
            uint32_t z[16];
            ptx::tmem_ld16(z_tmem + ch * 16, z);
            ptx::tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; ++e) z[e] = __float_as_uint(sigmoid(__uint_as_float(z[e])));
            ptx::tmem_st16(z_tmem + ch * 16, z);
        }
        ptx::tmem_wait_st();
        ptx::tc_fence_before_sync();
        ptx::named_arrive(2, kBoth);
    } else {
        ptx::set_max_regs_inc<kAddRegs>();
        const Block w = block_of<NT>(d, row_tiles, col_tiles, blockIdx.x);
        const int quarter = warp & 3, half = (warp - kAddWarp0) >> 2;    // TMEM lanes, columns
        const uint32_t d_tmem = tmem_base + ((uint32_t)(quarter * 32) << 16) + half * C::kCols;
        const uint32_t free_leader = ptx::map_to_cta(ptx::smem_addr(acc_free), 0);
        uint64_t acc[C::kCols / 2];
#pragma unroll
        for (int e = 0; e < C::kCols / 2; ++e) acc[e] = 0ull;
        for (int it = 0; it < n_it; ++it) {
            const int buf = buf_of(it);
            if (it == n_g) ptx::grid_dependency_wait();
            wait(&acc_full[buf], use_of(it) & 1);
            __syncwarp();
            ptx::tc_fence_after_sync();
#pragma unroll
            for (int ch = 0; ch < C::kCols / 16; ++ch) {
                uint32_t v[16];
                ptx::tmem_ld16(d_tmem + buf * NT + ch * 16, v);
                ptx::tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    acc[ch * 8 + e] = ptx::add2(acc[ch * 8 + e], ptx::f32x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1])));
            }
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_release_smem_cluster(free_leader + 8 * buf);
            if (it == n_g - 1) {                // the gates' sums are complete: the splitting warps make gates of them
#pragma unroll
                for (int ch = 0; ch < C::kCols / 16; ++ch) {
                    uint32_t v[16];
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        float z0, z1;
                        ptx::f32x2_split(acc[ch * 8 + e], z0, z1);
                        acc[ch * 8 + e] = 0ull;
                        v[2 * e] = __float_as_uint(z0);
                        v[2 * e + 1] = __float_as_uint(z1);
                    }
                    ptx::tmem_st16(d_tmem + buf * NT + ch * 16, v);
                }
                ptx::tmem_wait_st();
                ptx::tc_fence_before_sync();
                ptx::named_arrive(1, kBoth);
            }
        }
        ptx::named_sync(2, kBoth);               // the gates are there
        ptx::tc_fence_after_sync();
        // out = decoded value x gate: 32 rows x 32 columns at a time through the ring's memory, which nothing uses any more (rows
        // of 128 bytes, 128-byte swizzle), and out by TMA: whole lines, and rows past the last are not written
        const int g_buf = (n_g - 1) & 1;
        uint8_t* stage = smem + (warp - kAddWarp0) * (C::kCols * 32 * 4);
#pragma unroll
        for (int ch = 0; ch < C::kCols / 16; ++ch) {
            uint32_t z[16];
            ptx::tmem_ld16(d_tmem + g_buf * NT + ch * 16, z);
            ptx::tmem_wait_ld();
            uint8_t* box = stage + (ch >> 1) * 4096 + lane * 128;
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                float y[4];
                ptx::f32x2_split(acc[ch * 8 + 2 * h], y[0], y[1]);
                ptx::f32x2_split(acc[ch * 8 + 2 * h + 1], y[2], y[3]);
                *reinterpret_cast<float4*>(box + (((4 * (ch & 1) + h) ^ (lane & 7)) << 4)) =
                    make_float4(y[0] * __uint_as_float(z[4 * h]), y[1] * __uint_as_float(z[4 * h + 1]),
                                y[2] * __uint_as_float(z[4 * h + 2]), y[3] * __uint_as_float(z[4 * h + 3]));
            }
            if (ch & 1) {
                ptx::fence_proxy_async_smem();
                __syncwarp();
                const int c = half * C::kCols + 16 * (ch - 1);         // (a map's columns are a multiple of 64)
                if (lane == 0 && c < w.n_cols && quarter * 32 < w.rows) {
                    ptx::tma_store_2d(&tm_out, stage + (ch >> 1) * 4096, w.g * w.map_cols + w.n0 + c, (int)w.m0 + quarter * 32);
                    ptx::bulk_commit_group();
                }
            }
        }
        ptx::bulk_wait_group_all();        // (rows done again below come after this; and the memory may go)
    }
    ptx::tc_fence_before_sync();
    __syncthreads();
    if (*abort_flag) {             // a wait gave up, maybe behind the last one of the threads that issue: what is on its way comes to its end
        if (warp == 0 && rank == 0 && ptx::elect_one()) {        // (the thread that issued the MMAs: the election is the same each time)
            ptx::tc_commit_pair(drain_bar, 1);
            ptx::mbar_wait_drain(drain_bar, 0, drain_flag);
        }
        if (warp == 1 && ptx::elect_one())
            for (int n = *armed, back = 1; back <= C::kRaw && n - back >= 0; ++back)
                ptx::mbar_wait_drain(&raw_full[(n - back) % C::kRaw], ((n - back) / C::kRaw) & 1, drain_flag);
        __syncwarp();
    }
    ptx::cluster_arrive();         // neither CTA leaves (or frees tensor memory) while the other may still signal it
    ptx::cluster_wait();
    if (warp == 0) ptx::tmem_dealloc_pair(tmem_base, 2 * NT);
    if (warp >= kAddWarp0 && *any_bad) {
        uint32_t block;             // (worked out anew: nothing of this is kept in registers until here)
        asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(block));
        redo<NT>(d, o_lat, x, w_p, w_g, out, row_tiles, col_tiles, block, marks, reinterpret_cast<float*>(smem));
    }
    if (threadIdx.x == 0 && *abort_flag) raise_status(status_word, GTA_ERR_TIMEOUT);
}

template <int NT>
cudaError_t launch_tile(const Dims& d, const float* o_lat, const float* x, const float* w_p, const float* w_g, float* out,
                        int32_t* status_word, cudaStream_t stream, bool behind) {
    auto kern = sm100_decoder_f32_kernel<NT>;
    const uint64_t M = (uint64_t)d.B * d.N, n_out = (uint64_t)d.n_h * d.d_h;
    CUtensorMap tm_l, tm_x, tm_wp, tm_wg, tm_out;
    {
        const uint64_t dl[3] = {(uint64_t)d.d_l, M, (uint64_t)d.n_q}, dx[2] = {(uint64_t)d.H, M};
        const uint64_t dp[3] = {(uint64_t)d.d_h, (uint64_t)d.d_l, (uint64_t)d.n_h}, dg[2] = {n_out, (uint64_t)d.H};
        const uint64_t dout[2] = {n_out, M};
        const uint32_t rows[3] = {kBlockK, kTileM, 1}, cols[3] = {64, kBlockK, 1}, box[2] = {32, 32};
        if (!make_f32_map(&tm_l, o_lat, 3, dl, rows) || !make_f32_map(&tm_x, x, 2, dx, rows) ||
            !make_f32_map(&tm_wp, w_p, 3, dp, cols) || !make_f32_map(&tm_wg, w_g, 2, dg, cols) ||
            !make_f32_map(&tm_out, out, 2, dout, box, true))
            return cudaErrorInvalidValue;
    }
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg<NT>::kSmem);
    if (err != cudaSuccess) return err;
    const int row_tiles = (int)((M + 2 * kTileM - 1) / (2 * kTileM));
    const int col_tiles = (d.n_h / d.n_q * d.d_h + NT - 1) / NT;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2u * row_tiles * col_tiles * d.n_q);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = Cfg<NT>::kSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = behind ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kern, tm_l, tm_x, tm_wp, tm_wg, tm_out, d, o_lat, x, w_p, w_g, out, row_tiles, col_tiles,
                              status_word);
}

}  // namespace

gta_status_t sm100_decoder_f32_debug_wait(unsigned long long limit_ns, int withhold_first_arrive) {
    const WaitHook w = {limit_ns ? limit_ns : ptx::kWaitLimitNs, withhold_first_arrive ? 1 : 0};
    if (cudaMemcpyToSymbol(c_wait, &w, sizeof(w)) == cudaSuccess) return GTA_OK;
    cudaGetLastError();
    return GTA_ERR_CUDA;
}

long long sm100_decoder_f32_units(const Dims& d, int nt) {
    return (((long long)d.B * d.N + 2 * kTileM - 1) / (2 * kTileM)) * ((d.n_h / d.n_q * d.d_h + nt - 1) / nt) * d.n_q;
}

cudaError_t launch_sm100_decoder_f32(const Dims& d, const float* o_lat, const float* x, const float* w_p, const float* w_g,
                                     float* out, int32_t* status_word, cudaStream_t stream, bool behind, int nt) {
    if (nt == 256) return launch_tile<256>(d, o_lat, x, w_p, w_g, out, status_word, stream, behind);
    return launch_tile<128>(d, o_lat, x, w_p, w_g, out, status_word, stream, behind);
}

}  // namespace gta
