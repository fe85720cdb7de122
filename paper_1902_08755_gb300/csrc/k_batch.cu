// k_batch.cu -- many independent composites in a few persistent launches.
//
// Thesis 4.2.4 ("tile" compounds): fixed-size work packages sit in a queue
// and resources pull them until the queue is empty, which balances uneven
// work without a static assignment.  Here a work item is one output tile of
// one job (a job is a full composite: its inputs, mode and destination); a
// grid sized to the resident-CTA count of the device loops, each CTA taking
// the next item with one atomicAdd on a queue head.  Items are sorted by
// estimated cost, largest first (longest-processing-time order), so the tail
// of the launch is made of small items.  No CTA ever waits for another.
//
// There is a kernel, and a queue, per kind of item: one for all of them held
// every kind's loop to what they share of its registers, and spilled with more.
// The kernels of a batch run side by side (a later one's CTAs take the place
// of an earlier one's as its queue runs out).  HBM-bound: 128 uneven
// composites, half depth and half alpha, 3.77 GB: 642 us, 0.87 of the measured
// copy rate; one kernel with one shared loop body 852 us (640 M warp
// instructions, four inputs' loads in flight whatever the kind); a kernel per
// kind 783, with items fetched ahead and the kernels overlapped 756, and with
// the lean items below 642.
//
// Every item runs exactly the per-pixel arithmetic of the one-frame kernels
// (composite_body.cuh), so results are bit-identical to per-job launches and
// independent of the tile shape the autotuner picks.
#include <type_traits>

#include "composite_body.cuh"

namespace ec {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// Kinds of jobs:
//   kDepth8 (RGBA8, 4 adjacent px/lane), kDepth8Far (the same, a lane's pixels
//   32 apart; see depth_px4), kDepth32 (RGBA32F, 1 px/lane),
//   kAlpha32 (RGBA32F, 1 px/lane), kAlpha16 (RGBA16F, 2 px/lane)
enum { kDepth8, kDepth32, kAlpha32, kAlpha16, kDepth8Far };
constexpr int kJobKinds = kDepth8Far + 1;
static_assert(2 * kJobKinds == kBatchKinds, "general and lean items of each");

// Depth merge of RGBA32F, one pixel per lane (depth_px4's order of operations).
__device__ __forceinline__ void px_depth32(const SrcDesc* sd, const int16_t* act, int nact, int x, int y, const DstDesc& D)
{
    constexpr int U = 4;
    float bd = 1.0f;
    int bi = -1;
    uint4 bc = make_uint4(0u, 0u, 0u, 0u);
    for (int a = 0; a < nact; a += U) {
        uint4 c[U];
        float d[U];
        bool live[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            live[u] = false;
            if (a + u >= nact) continue;
            const SrcDesc& s = sd[act[a + u]];
            live[u] = y >= s.y0 && y < s.y1 && x >= s.x0 && x < s.x1;
            if (!live[u]) continue;
            const size_t e = (size_t)(y - s.oy) * (size_t)s.pitch + (size_t)(x - s.ox);
            const uint4* p = reinterpret_cast<const uint4*>(s.color) + e;
            if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
                c[u] = ld_stream(p);
            } else {
                const unsigned int* f = reinterpret_cast<const unsigned int*>(p);
                c[u] = make_uint4(__ldcs(f), __ldcs(f + 1), __ldcs(f + 2), __ldcs(f + 3));
            }
            d[u] = __ldcs(s.depth + e);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (live[u] && d[u] < bd) { bd = d[u]; bc = c[u]; bi = act[a + u]; }
    }
    const size_t o = (size_t)y * (size_t)D.pitch + (size_t)x;
    uint4* oc = reinterpret_cast<uint4*>(D.color) + o;
    if ((reinterpret_cast<uintptr_t>(oc) & 15u) == 0) st_stream(oc, bc);
    else { uint32_t* w = reinterpret_cast<uint32_t*>(oc); w[0] = bc.x; w[1] = bc.y; w[2] = bc.z; w[3] = bc.w; }
    if (D.depth) D.depth[o] = bd;
    if (D.winner) D.winner[(size_t)y * D.W + x] = (int16_t)bi;
}

// Lean items, whose tile every active input covers (with 16-byte rows where the
// kind reads them): folded without range tests, from compact records: the
// address of an input's pixel (0, 0) of the destination, its pitch, and its
// depth's address.  They have kernels of their own; with the general path in
// one kernel, both spill registers.
struct Lean {
    uint64_t color;
    int32_t pitch;
    int32_t pad;
};

template <int KIND>
__device__ __forceinline__ void lean_px(const Lean* rec, const uint64_t* rdepth, const int16_t* act, int nact, int x,
                                        int y, const DstDesc& D)
{
    if constexpr (KIND == kAlpha32 || KIND == kAlpha16) {
        constexpr bool F16 = KIND == kAlpha16;
        constexpr int U = 8, PX = F16 ? 2 : 1, B = F16 ? 8 : 16;
        float4 acc[PX];
        float T[PX];
#pragma unroll
        for (int j = 0; j < PX; ++j) { acc[j] = make_float4(0.f, 0.f, 0.f, 0.f); T[j] = 1.0f; }
        for (int a = 0; a < nact; a += U) {
            uint4 raw[U];
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (a + u < nact) {
                    const Lean r = rec[a + u];
                    raw[u] = ld_stream(reinterpret_cast<const uint4*>(r.color + (int64_t)B * ((int64_t)y * r.pitch + x)));
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (a + u < nact)
#pragma unroll
                    for (int j = 0; j < PX; ++j) over(pixel_of<F16>(raw[u], j), acc[j], T[j]);
        }
        store_alpha<F16>(D, x, y, acc, T);
    } else {
        constexpr int U = 4, STEP = KIND == kDepth8Far ? 32 : 1;
        float bd[4] = {1.0f, 1.0f, 1.0f, 1.0f};
        uint32_t bc[4] = {0u, 0u, 0u, 0u};
        int bi[4] = {-1, -1, -1, -1};
        for (int a = 0; a < nact; a += U) {
            uint32_t c[U][4];
            float d[U][4];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (a + u >= nact) continue;
                const Lean r = rec[a + u];
                const int64_t e = (int64_t)y * r.pitch + x;
                const uint32_t* pc = reinterpret_cast<const uint32_t*>(r.color + 4 * e);
                const float* pd = reinterpret_cast<const float*>(rdepth[a + u] + 4 * e);
                if constexpr (STEP == 1) {
                    const uint4 c4 = ld_stream(reinterpret_cast<const uint4*>(pc));
                    const float4 d4 = ld_stream(reinterpret_cast<const float4*>(pd));
                    c[u][0] = c4.x; c[u][1] = c4.y; c[u][2] = c4.z; c[u][3] = c4.w;
                    d[u][0] = d4.x; d[u][1] = d4.y; d[u][2] = d4.z; d[u][3] = d4.w;
                } else {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const bool in = x + STEP * j < D.W;
                        c[u][j] = in ? __ldcs(pc + STEP * j) : 0u;
                        d[u][j] = in ? __ldcs(pd + STEP * j) : 1.0f;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (a + u >= nact) continue;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (d[u][j] < bd[j]) { bd[j] = d[u][j]; bc[j] = c[u][j]; bi[j] = a + u; }
            }
        }
        if (D.winner)
#pragma unroll
            for (int j = 0; j < 4; ++j) bi[j] = bi[j] < 0 ? -1 : act[bi[j]];
        store_depth4<4, STEP>(D, x, y, bd, bc, bi);
    }
}

// f(x, y) for the first pixel of every lane's group in the item's tile, the row
// segments shared out over the warps.
template <int KIND, class F>
__device__ __forceinline__ void for_rows(int tx0, int ty0, int TW, int TH, int W, int H, F f)
{
    constexpr int kPx = KIND == kDepth8 || KIND == kDepth8Far ? 4 : (KIND == kAlpha16 ? 2 : 1);   // per lane
    constexpr int kNext = KIND == kDepth8Far ? 1 : kPx;                                           // lane to lane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, segs = TW / (32 * kPx), tasks = TH * segs;
    for (int r = warp; r < tasks; r += kWarps) {
        const int row = r / segs, y = ty0 + row, x = tx0 + (r - row * segs) * 32 * kPx + lane * kNext;
        if (y < H && x < min(tx0 + TW, W)) f(x, y);
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Work items are fetched ahead, so that no CTA stands still between two of
// them: while an item is composited, the next one's job and input descriptors
// are copied into shared memory, the record of the one after it is fetched, and
// the queue is asked for the one after that.  A CTA's first two items are given
// to it (in snake order over the sorted list), so that a short list is spread
// over all CTAs; the others come from the queue.  What an item needs later is
// kept in shared memory: registers held across the compositing loops would
// cost them loads in flight.  General items are folded by the one-frame
// kernels' bodies from the staged descriptors.
//
// The kernels of a batch are chained but do not wait for one another until
// they end, so the last items of one overlap the first of the next: no job may
// read what another one writes, and the first kernel is launched plainly, so
// that it and all of them start after whatever came before the batch.
template <int KIND, bool LEAN>
__global__ void __launch_bounds__(kThreads, 4)
k_batch(const BatchJob* __restrict__ jobs, const SrcDesc* __restrict__ srcs,
        const BatchItem* __restrict__ items, int n_items, uint32_t* head, int TW, int TH)
{
    __shared__ int16_t act[EC_MAX_BATCH_INPUTS];
    __shared__ __align__(16) SrcDesc sdesc[2][EC_MAX_BATCH_INPUTS];
    __shared__ __align__(16) BatchJob sjob[2];
    __shared__ __align__(16) BatchItem sitem[4];
    __shared__ __align__(16) Lean lean[EC_MAX_BATCH_INPUTS];
    __shared__ uint64_t ldepth[EC_MAX_BATCH_INPUTS];
    __shared__ int nact_s;
    const int tid = threadIdx.x;
    chain_next();

    // the record of ticket t into slot k: n = -1 past the list's end (thread 0)
    auto fetch_item = [&](uint32_t t, uint32_t k) {
        if (t < (uint32_t)n_items) cp_async16(&sitem[k & 3u], items + t);
        else sitem[k & 3u].n = -1;
    };
    // copy item k's job and inputs into its buffer (48-byte descriptors, 64-byte jobs)
    auto stage = [&](uint32_t k) {
        const BatchItem& b = sitem[k & 3u];
        const uint4* from = reinterpret_cast<const uint4*>(srcs + b.first);
        uint4* to = reinterpret_cast<uint4*>(sdesc[k & 1u]);
        for (int j = tid; j < 3 * b.n; j += kThreads) cp_async16(to + j, from + j);
        if (tid < 4 && b.n >= 0)
            cp_async16(reinterpret_cast<uint4*>(&sjob[k & 1u]) + tid, reinterpret_cast<const uint4*>(jobs + b.job) + tid);
    };
    // wait for what was copied; list the inputs that meet item k's tile
    auto open = [&](uint32_t k) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();                                // the buffer is there; the previous item is done
        const BatchItem& b = sitem[k & 3u];
        if (b.n < 0) return;                            // (uniform)
        const DstDesc& D = sjob[k & 1u].D;
        const SrcDesc* sd = sdesc[k & 1u];
        const int tx0 = b.tx * TW, ty0 = b.ty * TH;
        build_active([&](int, int i) -> const SrcDesc& { return sd[i]; }, b.n, tx0, ty0, min(tx0 + TW, D.W),
                     min(ty0 + TH, D.H), act, &nact_s);
        __syncthreads();
        if constexpr (LEAN) {
            for (int j = tid; j < nact_s; j += kThreads) {
                const SrcDesc& s = sd[act[j]];
                const int64_t e = -((int64_t)s.oy * s.pitch + s.ox);
                const int bpp = KIND == kAlpha32 ? 16 : KIND == kAlpha16 ? 8 : 4;
                lean[j].color = (uint64_t)(reinterpret_cast<uintptr_t>(s.color) + (uintptr_t)(e * bpp));
                lean[j].pitch = s.pitch;
                if (KIND == kDepth8 || KIND == kDepth8Far)
                    ldepth[j] = (uint64_t)(reinterpret_cast<uintptr_t>(s.depth) + (uintptr_t)(e * 4));
            }
            __syncthreads();
        }
    };

    uint32_t tick = 0u;
    if (tid == 0) {
        fetch_item(blockIdx.x, 0u);
        fetch_item(2u * gridDim.x - 1u - blockIdx.x, 1u);
        tick = 2u * gridDim.x + atomicAdd(head, 1u);      // the third item's ticket
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    stage(0u);
    open(0u);
    for (uint32_t i = 0; sitem[i & 3u].n >= 0; ++i) {   // (uniform; a CTA's items past the end are its last)
        if (tid == 0) {
            fetch_item(tick, i + 2u);                     // used in the next round
            tick = 2u * gridDim.x + atomicAdd(head, 1u);
        }
        stage(i + 1u);
        const SrcDesc* const sd = sdesc[i & 1u];
        const DstDesc& D = sjob[i & 1u].D;
        const int nact = nact_s;
        auto at = [&](int, int j) -> const SrcDesc& { return sd[j]; };
        for_rows<KIND>(sitem[i & 3u].tx * TW, sitem[i & 3u].ty * TH, TW, TH, D.W, D.H, [&](int x, int y) {
            if constexpr (LEAN) lean_px<KIND>(lean, ldepth, act, nact, x, y, D);
            else if constexpr (KIND == kDepth8) depth_px4<4, 1>(at, act, nact, x, y, D);
            else if constexpr (KIND == kDepth8Far) depth_px4<4, 32>(at, act, nact, x, y, D);
            else if constexpr (KIND == kDepth32) px_depth32(sd, act, nact, x, y, D);
            else if constexpr (KIND == kAlpha32) alpha_px<false>(at, act, nact, x, y, D);
            else alpha_px<true>(at, act, nact, x, y, D);
        });
        open(i + 1u);
    }
    chain_wait();                                         // the kinds before this one have ended too
}

// The items of one kernel.  first: the batch's first, which starts after
// everything before the batch; the later ones start once its CTAs have.
template <int KIND, bool LEAN>
cudaError_t launch_kind(const BatchJob* jobs, const SrcDesc* srcs, const BatchItem* items, const int* n_items,
                        uint32_t* head, const BatchShape& shape, int grid, cudaStream_t s, bool& first)
{
    constexpr int k = KIND + (LEAN ? kJobKinds : 0), m = KIND == kDepth8Far ? 0 : KIND;
    const int n = n_items[k], g = grid < n ? grid : n;
    if (n <= 0) return cudaSuccess;
    for (int j = 0; j < k; ++j) items += n_items[j];
    if (!first) return launch_chained(k_batch<KIND, LEAN>, g, kThreads, 0, s, jobs, srcs, items, n, head + k, shape.tw[m], shape.th[m]);
    first = false;
    k_batch<KIND, LEAN><<<g, kThreads, 0, s>>>(jobs, srcs, items, n, head + k, shape.tw[m], shape.th[m]);
    return cudaGetLastError();
}

}  // namespace

int batch_warp_px(int mode) { return 32 * (mode == 0 ? 4 : (mode == 3 ? 2 : 1)); }

int batch_ctas_per_sm()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_batch<kAlpha32, true>, kThreads, 0) != cudaSuccess) return 1;
    return n > 0 ? n : 1;
}

int batch_kind(const BatchJob& j, bool covered)
{
    const int k = j.mode == 0 && j.step != 1 ? kDepth8Far : j.mode;
    return k + (covered && k != kDepth32 ? kJobKinds : 0);
}

cudaError_t launch_batch(const BatchJob* jobs, const SrcDesc* srcs, const BatchItem* items,
                         const int* n_items, uint32_t* head, const BatchShape& shape, int grid,
                         cudaStream_t s)
{
    cudaError_t e = cudaMemsetAsync(head, 0, kBatchKinds * sizeof(uint32_t), s);
    bool first = true;
    auto run = [&](auto kind, auto lean) {
        if (e == cudaSuccess)
            e = launch_kind<decltype(kind)::value, decltype(lean)::value>(jobs, srcs, items, n_items, head, shape, grid, s, first);
    };
    using std::integral_constant;
    auto both = [&](auto kind) {
        run(kind, std::true_type{});
        run(kind, std::false_type{});
    };
    both(integral_constant<int, kAlpha32>{});
    both(integral_constant<int, kAlpha16>{});
    run(integral_constant<int, kDepth32>{}, std::false_type{});
    both(integral_constant<int, kDepth8>{});
    both(integral_constant<int, kDepth8Far>{});
    return e;
}

}  // namespace ec
