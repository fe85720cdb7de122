// k_rle.cu -- run-length pixel codec kernels for sm_103a (thesis 5.5.1:
// per-component RLE, bit-swizzle preconditioner, data decomposition).
//
// Compress: a pipeline of kernels with no waits between warps.
//   1. Coding, a chunk of 4096 elements at a time: the chunk's change points are
//      listed; a chunk with few of them (sparse) is coded at once from the list
//      into a scratch pool, the others (dense) are listed.
//      Modes 1, 2: element change points, four byte planes (mode 2 swizzled;
//      the swizzle permutes bits, so it commutes with the comparison); runs of
//      three or more bytes become repeat tokens, maximal spans of shorter runs
//      literal tokens.  Mode 0 (basic RLE): change points of 8-byte units,
//      one stream; runs of two or more units repeat, single units literal.
//   2. The dense chunks, coded from the image: all four planes classified
//      at once with byte-SIMD masks (a byte is part of a repeat iff one of the
//      three windows of 3 around it is constant), max- and sum-scans over the
//      CTA, and the streams to the pool where it has room; in mode 0 a CTA per
//      chunk with block scans, which sizes them.
//   3. Placing: a chunk's offset is the sum of its image's chunks before it
//      (taken from sums over 32 chunks; in mode 0 a scan launch computes the
//      offsets); the pooled chunks are copied to their place with their end-table
//      entries, the header and the stream size are written, and chunks that are
//      not in the pool are coded again.
// Every wait (for copies into shared memory) is bounded (EC_ERR_TIMEOUT).
//
// Decompress: one CTA of four warps per chunk.  Every warp fetches the header
// and the chunk's end-table entries in one round trip and validates them.
// Warp p walks plane p's tokens; each is checked against its stream and chunk bounds.  A
// chunk of few runs is written from the runs' starts and bytes (16-byte stores
// of constant groups); the planes of the others are decoded into shared memory
// and transposed back into elements with byte permutes.
#include "ec_internal.cuh"
#include "rle_codec.cuh"

#include <algorithm>
#include <atomic>

namespace ec {
namespace {

constexpr int kChunk = EC_RLE_CHUNK;                 // 4096 elements
constexpr int kT = 256;                              // threads per mode-0 CTA
constexpr uint32_t kMagic = 0x31524345u;             // "ECR1"
constexpr int kSpinLimit = 1 << 20;            // tries of a bounded mbarrier wait

using rlec::swizzle;
using rlec::transpose4;

template <int N>
__device__ __forceinline__ int find_job(const RleJobList<N>& J, uint32_t unit)
{
    int lo = 0, hi = J.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (J.j[mid].first_unit <= unit) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ void put_u32(uint8_t* p, uint32_t v)
{
    p[0] = (uint8_t)v; p[1] = (uint8_t)(v >> 8); p[2] = (uint8_t)(v >> 16); p[3] = (uint8_t)(v >> 24);
}


// Row of element q: q / w from the reciprocal winv = floor((2^32 - 1) / w).
// q winv / 2^32 lies in (q / w - 2 q / 2^32, q / w], and q < 2^27, so its floor
// is the quotient or one less.
__device__ __forceinline__ uint32_t row_of(const RleJobDesc& jb, uint32_t q)
{
    const uint32_t y = __umulhi(q, jb.winv);
    return q - y * (uint32_t)jb.w >= (uint32_t)jb.w ? y + 1u : y;
}

// Element q of a job's image.
__device__ __forceinline__ size_t elem_off(const RleJobDesc& jb, uint32_t q)
{
    const uint32_t y = row_of(jb, q);
    return (size_t)y * jb.pitch + (q - y * (uint32_t)jb.w);
}

__device__ void write_header(uint8_t* d, const RleJobDesc& jb)
{
    put_u32(d + 0, kMagic);
    d[4] = 1; d[5] = 0;                               // version
    d[6] = (uint8_t)jb.mode; d[7] = 0;
    put_u32(d + 8, (uint32_t)jb.w);
    put_u32(d + 12, (uint32_t)jb.h);
    put_u32(d + 16, 4u);
    put_u32(d + 20, (uint32_t)kChunk);
    put_u32(d + 24, jb.n_chunks);
    put_u32(d + 28, jb.mode == 0 ? 1u : 4u);       // streams per chunk
}

// ------------------------------------------------------------- compress ----

// Copy n stage bytes (src 4-byte aligned) to o, threads t, t+nt, ...: byte
// stores up to o's first word boundary and after its last, word stores of
// funnel-shifted stage words between.  The two buffers never overlap, and a
// thread's loads (eight words at a time, and its head and tail bytes) are all
// issued before its stores.  Reads up to one word past src + n.
__device__ __forceinline__ void copy_out(uint8_t* __restrict__ o, const uint8_t* __restrict__ src, uint32_t n,
                                         uint32_t t, uint32_t nt)
{
    const uintptr_t a0 = reinterpret_cast<uintptr_t>(o), a1 = a0 + n;
    const uintptr_t w0 = (a0 + 3) & ~(uintptr_t)3, w1 = a1 & ~(uintptr_t)3;
    if (w0 >= w1) {
        for (uint32_t i = t; i < n; i += nt) o[i] = src[i];
        return;
    }
    const uint32_t head = (uint32_t)(w0 - a0), tail0 = (uint32_t)(w1 - a0);   // head, n - tail0 < 4 <= nt
    const bool hh = t < head, th = tail0 + t < n;
    const uint8_t hb = hh ? src[t] : 0, tb = th ? src[tail0 + t] : 0;
    const uint32_t nw = (uint32_t)((w1 - w0) >> 2);
    const uint32_t* __restrict__ s32 = reinterpret_cast<const uint32_t*>(src);
    const uint32_t sh = 8u * head;
    uint32_t* __restrict__ o32 = reinterpret_cast<uint32_t*>(w0);
    for (uint32_t k0 = t; k0 < nw; k0 += 8u * nt) {
        uint32_t v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            // bytes [head + 4k, head + 4k + 4), head < 4
            const uint32_t k = k0 + (uint32_t)j * nt;
            v[j] = k < nw ? __funnelshift_r(s32[k], s32[k + 1], sh) : 0u;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t k = k0 + (uint32_t)j * nt;
            if (k < nw) o32[k] = v[j];
        }
    }
    if (hh) o[t] = hb;
    if (th) o[tail0 + t] = tb;
}

// ---- compressor --------------------------------------------------------------
// The coding kernels list each chunk's change points.  A chunk of few of them
// (sparse) is coded at once from the list, its streams left in a scratch pool;
// the others (dense) are listed, and a recoding kernel codes them from the
// image.  A chunk's offset is the sum of its image's chunk sizes before it (sums
// over 32 chunks are taken while they are coded; mode 0 scans them); the placing
// kernels copy the pooled chunks to their place, and code those that the pool
// had no room for again.  No kernel waits for another's warps.
//
// Four-plane modes: a CTA of four warps per chunk (k_rle_code).  Mode 0: every
// warp of a persistent kernel works alone, chunk after chunk (k_rle_compress0):
// it streams each chunk through a ring of two 2 KB quarter buffers in shared
// memory, filled by asynchronous copies (bulk copies of row segments, or 4-byte
// copies where rows are not 16-byte aligned) that complete on the buffer's
// mbarrier; a buffer is refilled with the next quarter (of this chunk or the
// next) as soon as it has been read.
constexpr int kWPB = 2;                       // warps per CTA
constexpr int kCap = 128;                     // change points the sparse path takes
constexpr int kQ = 512;                       // elements per quarter buffer
constexpr int kQPC = kChunk / kQ;             // quarters per chunk
constexpr int kSlots = 2;                     // quarter buffers per warp

// Each plane of a sparse chunk has at most kCap runs and codes to at most
// 3 kCap + kChunk / 64 bytes (a repeat run of length L to 2 ceil(L / 128) <=
// 2 + L / 64 bytes, a literal span of k short runs to at most 3k bytes).
constexpr int kStagePlane = 3 * kCap + kChunk / 64;
constexpr uint32_t kRecode = 0xFFFFFFFFu;      // record: coded again when placed
constexpr uint32_t kDense = 0x80000000u;       // record: a pooled dense chunk (offset / 16 in the low bits)

// One warp's shared memory.  Quarter s of the warp's sequence of quarters
// (kQPC per chunk) goes to buf[s % kSlots].
struct WarpRing {
    uint32_t buf[kSlots][kQ + 4];   // + 16 guard bytes before each quarter
    uint64_t full[kSlots];
    uint64_t pad[4 - kSlots];       // (keeps what follows 16-byte aligned)
    uint8_t stage[4 * kStagePlane]; // the chunk's plane streams (plane p at p * kStagePlane)
    uint32_t ce[kCap];              // the chunk being read: first element of each change point's unit,
    uint32_t ch[kCap];              // its second element
    uint16_t cq[kCap];              // and its position
};
static_assert((kQ + 4) * 4 % 16 == 0 && sizeof(WarpRing) % 16 == 0, "16-byte aligned buffers");

// A coded chunk, as the coding kernels leave it for the placing kernels: its
// four plane stream sizes, where its streams wait in the pool (a sparse chunk's
// offset / 4, a dense chunk's offset / 16 with kDense, or kRecode: not kept,
// coded again from the image when placed), and, in mode 0, its offset inside the
// stream's payload (written by the scan).
struct ChunkRec {
    uint16_t T[4];
    uint32_t pool;
    uint32_t off;
};
static_assert(sizeof(ChunkRec) == 16, "chunk record");

// A launch's scratch.
constexpr uint32_t kGroup = 32;                // chunks whose sizes are summed up while they are coded
struct RleScratch {
    uint32_t* counters;     // [0] mode 0: ticket, else sparse chunks to code again; [1] listed chunks; [2, 3] pool cursor
    ChunkRec* rec;          // per chunk
    uint32_t* recode;       // listed chunks: the dense ones, in mode 0 also those that found the pool full
    uint32_t* again;        // sparse chunks that found the pool full
    uint32_t* groups;       // bytes coded per kGroup chunks
    uint8_t* pool;
    size_t pool_bytes;
    size_t slots;           // of them the first: a slot of kRlePoolPerUnit bytes per chunk, or none
};
constexpr size_t kCompressSmem = kWPB * sizeof(WarpRing);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* b)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_u32(b)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_tx(uint64_t* b, uint32_t bytes)
{
    asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}"
                 ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}

// One try of a wait for the phase of the given parity; the thread may sleep
// in it (up to about a microsecond) until the phase completes.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* b, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(b)), "r"(parity), "r"(1000u) : "memory");
    return ok != 0u;
}

// Wait for the phase of the given parity to complete; gives up after
// kSpinLimit tries (recording EC_ERR_TIMEOUT) instead of spinning forever.
__device__ __forceinline__ void mbar_wait(uint64_t* b, uint32_t parity, uint32_t* status)
{
    for (int i = 0; i < kSpinLimit; ++i)
        if (mbar_try_wait(b, parity)) return;
    set_status(status, EC_ERR_TIMEOUT);
}

// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) from
// global to shared memory, completing on mbarrier b.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* b)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(b)) : "memory");
}

// Elements [q, q + 4) of a chunk that starts at element q0 (q a multiple of
// 4; zeros past len).  16-byte loads where the image allows them (the four
// elements then lie in one row), else one load per element.
__device__ __forceinline__ uint4 load_elems(const RleJobDesc& jb, uint32_t q0, int len, int q)
{
    if (q >= len) return make_uint4(0u, 0u, 0u, 0u);
    const uint32_t w = (uint32_t)jb.w;
    if (jb.vec && q + 4 <= len) {
        const size_t e = jb.pitch == jb.w ? q0 + (uint32_t)q : elem_off(jb, q0 + (uint32_t)q);
        return __ldg(reinterpret_cast<const uint4*>(jb.src + e));
    }
    uint32_t v[4];
    uint32_t y = row_of(jb, q0 + (uint32_t)q), x = q0 + (uint32_t)q - y * w;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[k] = q + k < len ? __ldg(jb.src + (size_t)y * jb.pitch + x) : 0u;
        if (++x == w) { x = 0u; ++y; }
    }
    return make_uint4(v[0], v[1], v[2], v[3]);
}

// Asynchronous 4-byte copy from global to shared memory, and the arrival on
// mbarrier b once all of this thread's earlier such copies have landed (the
// barrier's pending count is raised by one now and lowered by the arrival).
__device__ __forceinline__ void cp_async4(void* dst, const void* src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_arrive(uint64_t* b)
{
    asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];" ::"r"(smem_u32(b)) : "memory");
}

// Start the copy of quarter qi of chunk `unit` into W.buf[slot].  Images whose
// rows are 16-byte aligned: lane 0 sets the expected bytes, every lane copies
// row segments with bulk copies.  Other images: every lane copies elements
// lane, lane + 32, ... with 4-byte asynchronous copies, and the barrier
// completes once all of them have landed.  Quarters with nothing to copy (past
// the image's end, an empty image) just arrive.
__device__ void issue_quarter(const RleJobDesc& jb, uint32_t unit, int qi, int slot, WarpRing& W)
{
    const int lane = threadIdx.x & 31;
    int qlen = 0;
    uint32_t qs = 0u;
    if (jb.n_chunks > 0) {
        const uint32_t q0 = (unit - jb.first_unit) * (uint32_t)kChunk;
        const int len = (int)min((uint32_t)kChunk, (uint32_t)jb.w * (uint32_t)jb.h - q0);
        qlen = min(max(len - kQ * qi, 0), kQ);
        qs = q0 + (uint32_t)(kQ * qi);
    }
    if (qlen == 0) {
        if (lane == 0) mbar_arrive(&W.full[slot]);
        return;
    }
    uint32_t* dst = W.buf[slot] + 4;
    const uint32_t w = (uint32_t)jb.w;
    if (!jb.vec || (qlen & 3)) {                       // (a contiguous image may end inside a 16-byte group)
        uint32_t y = row_of(jb, qs + (uint32_t)lane), x = qs + (uint32_t)lane - y * w;
        for (int i = lane; i < qlen; i += 32) {
            cp_async4(dst + i, jb.src + (size_t)y * jb.pitch + x);
            x += 32u;
            while (x >= w) { x -= w; ++y; }
        }
        cp_async_arrive(&W.full[slot]);
        __syncwarp();                                  // every lane's pending count is in
        if (lane == 0) mbar_arrive(&W.full[slot]);
        return;
    }
    if (lane == 0) mbar_arrive_tx(&W.full[slot], 4u * (uint32_t)qlen);
    __syncwarp();
    if (jb.pitch == jb.w) {
        if (lane == 0) bulk_load(dst, jb.src + qs, 4u * (uint32_t)qlen, &W.full[slot]);
        return;
    }
    const uint32_t y0 = row_of(jb, qs), y1 = row_of(jb, qs + (uint32_t)qlen - 1u);
    for (uint32_t y = y0 + (uint32_t)lane; y <= y1; y += 32) {
        const uint32_t a = y == y0 ? qs - y0 * w : 0u;                   // first column of the segment
        const uint32_t b = min(w, qs + (uint32_t)qlen - y * w);          // its end column
        bulk_load(dst + (y * w + a - qs), jb.src + (size_t)y * jb.pitch + a, 4u * (b - a), &W.full[slot]);
    }
}

// ---- coding kernel of the four-plane modes: a CTA of four warps per chunk ----
// The chunk is copied into shared memory (bulk copies, or 4-byte asynchronous
// copies where rows are not 16-byte aligned); twelve CTAs are resident on an
// SM, so the copies of most overlap the work of the others.  Lane l of warp k
// holds positions [1024 k + 32 l, + 32) and flags those whose element differs
// from its predecessor in the bits of one word.  One scan over the CTA lists
// the change points of the whole chunk in order.  A byte plane can change only
// where the element does, so each plane's runs are the change points where that
// plane's byte differs from the previous change point's, and every run's value
// is the byte at its start: warp p then codes plane p from the list alone.  A
// chunk with more than kCap change points is dense and left to the recoding
// kernel.
//
// Bound by instruction issue up to a few thousand chunks per launch, by HBM and
// issue alike beyond (2110 warp instructions per chunk, issue 65% active, DRAM
// 75%).  16 flat sources, colour and depth: 1920x1080 54 -> 33.4 us, 7680x4320
// (1.87 GB) 357 -> 307 us, against persistent warps that each streamed a chunk
// through two 2 KB buffers (2930 instructions per chunk, and a chunk's whole
// latency on one warp: the pieces of a binary-swap stage took 34 us whatever
// their number, 10 to 24 here).  Holding the chunk in registers (eight 16-byte groups
// per lane, eight CTAs per SM) took 3220 instructions per chunk and 465 us.
constexpr int kCT = 128;

// Bytes that a plane of at most kCap runs codes to: r repeat runs to 2 r +
// kChunk / 64 (2 ceil(L / 128) <= 2 + L / 64 for a run of L), k short ones, of
// at most two bytes, in s literal spans to 2 k + s + k / 64.  A repeat run lies
// between two spans, so s <= kCap / 2.  (With the tables, 18.3 KB per CTA: twelve
// fit on an SM.  With 3 kCap + kChunk / 64 eleven did: 313 -> 307 us for 16 flat
// 7680x4320 sources.)
constexpr int kStagePlane4 = 2 * kCap + kCap / 2 + kCap / 64 + kChunk / 64 + 6;
static_assert(kStagePlane4 % 8 == 0, "planes' stages are aligned");

// Pool space of a chunk of `total` bytes: the copy to its place reads up to one
// word past them, and the last 32-byte sector is filled up (a sector written in
// part would be fetched from memory when it is read).
__host__ __device__ constexpr uint32_t pool_need(uint32_t total) { return (total + 4u + 31u) & ~31u; }

// The pool of a launch.  Where it has room behind them for every few-run chunk,
// chunks of up to kRlePoolPerUnit bytes have slots of their own, and only the
// others take space with an atomic (2025 flat chunks: 8.2 us, 8.7 with an atomic
// for each).  Otherwise (the least pool, the allocation-free entry point's,
// launches of more than 167 thousand chunks) all take what they need: the slots
// would leave the others no room, and those would be coded twice (8192 few-run
// chunks of 512 to 770 bytes: 188 us, 75 to 98 so).
constexpr size_t pool_slots(size_t units, size_t pool_bytes)
{
    return pool_bytes >= (kRlePoolPerUnit + pool_need(4 * kStagePlane4)) * units ? kRlePoolPerUnit * units : 0;
}

// Plane stream of a chunk of len elements from its m <= 32 change points, run
// by run, where every run is at least 3 bytes (so all of it is repeat tokens).
// Lane i holds change point i: byte v at position q (valid: i < m); out is even.
// Returns the bytes written, or 0 (nothing written) when a run is shorter.
__device__ __forceinline__ uint32_t code_plane_few(bool valid, uint32_t v, int q, int len, uint8_t* out)
{
    const int lane = threadIdx.x & 31;
    const uint32_t before = __shfl_up_sync(0xffffffffu, v, 1);
    const bool keep = valid && (lane == 0 || v != before);          // starts a run
    const uint32_t K = __ballot_sync(0xffffffffu, keep);
    const uint32_t nm = lane == 31 ? 0u : K & ~((2u << lane) - 1u);
    const int qn = __shfl_sync(0xffffffffu, q, nm ? __ffs(nm) - 1 : 0);
    const int L = (nm ? qn : len) - q;
    if (__any_sync(0xffffffffu, keep && L < 3)) return 0u;
    const uint32_t cost = keep ? 2u * (uint32_t)((L + 127) >> 7) : 0u;
    const uint32_t incl = (uint32_t)rlec::warp_incl_sum((int)cost, lane);
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    if (keep) {                                       // (out and every token's place are even)
        uint16_t* o = reinterpret_cast<uint16_t*>(out + (incl - cost));
        int r = L;
        for (; r > 128; r -= 128) *o++ = (uint16_t)(0xFFu | (v << 8));
        *o = (uint16_t)((uint32_t)(127 + r) | (v << 8));
    }
    return total;
}

// Plane stream of a chunk of len elements from its m <= 128 change points
// (positions cq of the elements el, the plane's byte at bit `shift`; swizzled on
// reading when sw).  Lane l takes change points 4l .. 4l+3.  A run of three or
// more bytes becomes repeat tokens; a shorter one belongs to a literal span (a
// maximal sequence of short runs), whose start a warp max-scan finds.  A short
// run at byte offset b of its span writes its bytes, the control byte of a
// token that ends among them (127 for a full one), and, if the span ends with
// it, the last token's control byte.  A plane without short runs (three in four
// of those of flat-shaded sources) needs no spans, and its tokens are whole
// 16-bit stores (out is even): a binary swap of 16 1920x1080 sources 199.5 us
// without that path, 197.0 with it.  Returns the bytes written (at most
// kStagePlane4).
__device__ __forceinline__ uint32_t code_plane_many(const uint32_t* el, const uint16_t* cq, int m, int shift, bool sw,
                                                    int len, uint8_t* out)
{
    const int lane = threadIdx.x & 31, i0 = 4 * lane;
    const uint32_t below = (1u << lane) - 1u, above = lane == 31 ? 0u : ~((2u << lane) - 1u);
    uint32_t v[4];
    int q[4], L[4];
    uint32_t keep = 0u;                               // bit k: change point i0 + k starts a run of this plane
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const bool ok = i0 + k < m;
        q[k] = ok ? (int)cq[i0 + k] : len;
        uint32_t e = ok ? el[q[k]] : 0u;
        if (sw) e = swizzle(e);
        v[k] = (e >> shift) & 0xFFu;
        if (ok && k > 0 && v[k] != v[k - 1]) keep |= 1u << k;
    }
    const uint32_t vp = __shfl_up_sync(0xffffffffu, v[3], 1);
    if (i0 < m && (lane == 0 || v[0] != vp)) keep |= 1u;
    // where the next run starts: the lanes' first runs, then right to left
    const uint32_t has = __ballot_sync(0xffffffffu, keep != 0u);
    int first = len;
#pragma unroll
    for (int k = 3; k >= 0; --k)
        if ((keep >> k) & 1u) first = q[k];
    const int nl = (has & above) ? __ffs(has & above) - 1 : 0;
    int next = __shfl_sync(0xffffffffu, first, nl);
    if (!(has & above)) next = len;
    uint32_t sh = 0u;                                 // bit k: a short run
    uint32_t first_short = 0u, last_short = 0u;
    bool any = false;
#pragma unroll
    for (int k = 3; k >= 0; --k) {
        L[k] = 0;
        if (!((keep >> k) & 1u)) continue;
        L[k] = next - q[k];
        next = q[k];
        const uint32_t s = L[k] < 3 ? 1u : 0u;
        sh |= s << k;
        first_short = s;
        if (!any) { last_short = s; any = true; }
    }
    if (!__any_sync(0xffffffffu, sh != 0u)) {         // repeat tokens only
        uint32_t cost = 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if ((keep >> k) & 1u) cost += (uint32_t)((L[k] + 127) >> 7);
        const uint32_t incl = (uint32_t)rlec::warp_incl_sum((int)cost, lane);
        uint16_t* o = reinterpret_cast<uint16_t*>(out) + (incl - cost);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (!((keep >> k) & 1u)) continue;
            int r = L[k];
            for (; r > 128; r -= 128) *o++ = (uint16_t)(0xFFu | (v[k] << 8));
            *o++ = (uint16_t)((uint32_t)(127 + r) | (v[k] << 8));
        }
        return 2u * __shfl_sync(0xffffffffu, incl, 31);
    }
    const uint32_t ps = __shfl_sync(0xffffffffu, last_short, (has & below) ? 31 - __clz(has & below) : 0);
    const uint32_t ns = __shfl_sync(0xffffffffu, first_short, nl);
    const bool prev_short = (has & below) && ps, next_short = (has & above) && ns;
    // the last span start up to each lane (position + 1; 0: none)
    uint32_t start = 0u;
    bool p = prev_short;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!((keep >> k) & 1u)) continue;
        const bool s = (sh >> k) & 1u;
        if (s && !p) start = (uint32_t)q[k] + 1u;
        p = s;
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, start, o);
        if (lane >= o) start = max(start, y);
    }
    uint32_t span0 = __shfl_up_sync(0xffffffffu, start, 1);    // the span open at the lane's first run, if any
    if (lane == 0) span0 = 0u;
    uint32_t cost = 0u, sp = span0;
    p = prev_short;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!((keep >> k) & 1u)) continue;
        const bool s = (sh >> k) & 1u;
        if (s && !p) sp = (uint32_t)q[k] + 1u;
        p = s;
        if (!s) cost += 2u * (uint32_t)((L[k] + 127) >> 7);
        else {
            const uint32_t b = (uint32_t)q[k] + 1u - sp;
            cost += (uint32_t)L[k] + (((b + (uint32_t)L[k] + 127u) >> 7) - ((b + 127u) >> 7));
        }
    }
    const uint32_t incl = (uint32_t)rlec::warp_incl_sum((int)cost, lane);
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
    uint32_t o = incl - cost;
    sp = span0;
    p = prev_short;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!((keep >> k) & 1u)) continue;
        const bool s = (sh >> k) & 1u;
        if (s && !p) sp = (uint32_t)q[k] + 1u;
        p = s;
        if (!s) {
            for (int r = L[k]; r > 0; r -= 128) {
                out[o] = (uint8_t)(127 + min(r, 128));
                out[o + 1] = (uint8_t)v[k];
                o += 2;
            }
        } else {
            const uint32_t b = (uint32_t)q[k] + 1u - sp;
            const uint32_t so = o - b - ((b + 127u) >> 7);   // the span's first control byte
            for (uint32_t x = b; x < b + (uint32_t)L[k]; ++x) {
                out[so + x + (x >> 7) + 1u] = (uint8_t)v[k];
                if ((x & 127u) == 127u) out[so + 129u * (x >> 7)] = 127u;
            }
            const uint32_t later = keep >> (k + 1);          // the lane's later runs
            const bool more = later ? (sh >> (k + __ffs(later))) & 1u : next_short;
            const uint32_t last = b + (uint32_t)L[k] - 1u;
            if (!more) out[so + 129u * (last >> 7)] = (uint8_t)(last & 127u);
            o += (uint32_t)L[k] + (((b + (uint32_t)L[k] + 127u) >> 7) - ((b + 127u) >> 7));
        }
    }
    return total;
}

template <int N>
__global__ void __launch_bounds__(kCT, 12)
k_rle_code(const __grid_constant__ RleJobList<N> J, const RleScratch W, uint32_t* status)
{
    __shared__ __align__(16) uint32_t raw[4 + kChunk];      // the chunk, after a guard
    __shared__ __align__(16) uint8_t stage[4][kStagePlane4];
    __shared__ uint16_t cq[kCap];                            // the change points' positions
    __shared__ uint64_t full;
    __shared__ uint32_t s_cnt[4], s_T[4], s_po;
    __shared__ int s_ji;
    uint32_t* const el = raw + 4;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t unit = blockIdx.x;
    if (warp == 0) {                                         // find the job, start the copies
        if (lane == 0) {
            mbar_init(&full, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        const int ji = find_job(J, unit);
        const RleJobDesc& jb = J.j[ji];
        const uint32_t q0 = (unit - jb.first_unit) * (uint32_t)kChunk, n = (uint32_t)jb.w * (uint32_t)jb.h;
        const uint32_t w = (uint32_t)jb.w, len = n ? min((uint32_t)kChunk, n - q0) : 0u;
        if (lane == 0) s_ji = ji;
        chain_wait();
        if (len > 0 && jb.vec && !(len & 3u)) {
            __syncwarp();
            if (lane == 0) mbar_arrive_tx(&full, 4u * len);
            __syncwarp();
            if (jb.pitch == jb.w) {
                if (lane == 0) bulk_load(el, jb.src + q0, 4u * len, &full);
            } else {
                const uint32_t y0 = row_of(jb, q0), y1 = row_of(jb, q0 + len - 1u);
                for (uint32_t y = y0 + (uint32_t)lane; y <= y1; y += 32) {
                    const uint32_t a = y == y0 ? q0 - y0 * w : 0u;           // first column of the row's part
                    const uint32_t b = min(w, q0 + len - y * w);             // its end column
                    bulk_load(el + (y * w + a - q0), jb.src + (size_t)y * jb.pitch + a, 4u * (b - a), &full);
                }
            }
        }
    }
    chain_wait();
    __syncthreads();
    const RleJobDesc& jb = J.j[s_ji];
    if (jb.n_chunks == 0) return;                     // an empty image: placing writes its header
    const uint32_t q0 = (unit - jb.first_unit) * (uint32_t)kChunk;
    const int len = (int)min((uint32_t)kChunk, (uint32_t)jb.w * (uint32_t)jb.h - q0);
    if (jb.vec && !(len & 3)) {
        mbar_wait(&full, 0u, status);
    } else {                                          // (also a contiguous image that ends inside a 16-byte group)
        const uint32_t w = (uint32_t)jb.w;
        if (w >= 32u) {                               // a warp takes a quarter of the chunk, a row's part at a time
            int q = kChunk / 4 * warp;
            const int qe = min(len, q + kChunk / 4);
            const uint32_t y = row_of(jb, q0 + (uint32_t)min(q, len - 1));
            uint32_t x = q0 + (uint32_t)q - y * w;
            const uint32_t* row = jb.src + (size_t)y * jb.pitch;
            while (q < qe) {
                const int n = min((int)(w - x), qe - q);
                const uint32_t* from = row + x + lane;
                uint32_t* to = el + q + lane;
                for (int i = lane; i < n; i += 256) {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (i + 32 * k < n) cp_async4(to + 32 * k, from + 32 * k);
                    from += 256;
                    to += 256;
                }
                q += n;
                x = 0u;
                row += jb.pitch;
            }
        } else {
            for (int i = tid; i < len; i += kCT) cp_async4(el + i, jb.src + elem_off(jb, q0 + (uint32_t)i));
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
    }
    // flags of the lane's 32 elements; its 16-byte groups are taken from the
    // (lane mod 8)-th on, so that eight lanes' reads meet different banks
    const int p0 = 1024 * warp + 32 * lane;
    uint32_t F = 0u, pv = el[p0 + 4 * (lane & 7) - 1];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int g = (j + lane) & 7;
        const uint4 v = *reinterpret_cast<const uint4*>(el + p0 + 4 * g);
        if (j > 0 && g == 0) pv = el[p0 - 1];
        uint32_t f = v.x != pv ? 1u : 0u;
        if (v.y != v.x) f |= 2u;
        if (v.z != v.y) f |= 4u;
        if (v.w != v.z) f |= 8u;
        F |= f << (4 * g);
        pv = v.w;
    }
    if (tid == 0) F |= 1u;                            // position 0 is always listed
    if (len < kChunk) {
        const int left = len - p0;
        if (left < 32) F &= left <= 0 ? 0u : (1u << left) - 1u;
    }
    const int own = __popc(F), incl = rlec::warp_incl_sum(own, lane);
    if (lane == 31) s_cnt[warp] = (uint32_t)incl;
    __syncthreads();
    const uint32_t n0 = s_cnt[0], n1 = s_cnt[1], n2 = s_cnt[2], n3 = s_cnt[3];
    const int m = (int)(n0 + n1 + n2 + n3);
    if (m > kCap) {                                   // dense: coded by the recoding kernel
        if (tid == 0) {
            W.recode[atomicAdd(W.counters + 1, 1u)] = unit;
        }
        return;
    }
    {
        uint32_t o = (uint32_t)(incl - own) + (warp > 0 ? n0 : 0u) + (warp > 1 ? n1 : 0u) + (warp > 2 ? n2 : 0u);
        for (; F; F &= F - 1u) cq[o++] = (uint16_t)(p0 + __ffs(F) - 1);
    }
    __syncthreads();
    const bool sw = jb.mode == 2;
    uint32_t T = 0u;
    if (m <= 32) {
        const int q = lane < m ? (int)cq[lane] : 0;
        uint32_t e = el[q];
        if (sw) e = swizzle(e);
        T = code_plane_few(lane < m, (e >> (8 * warp)) & 0xFFu, q, len, stage[warp]);
    }
    if (T == 0u) T = code_plane_many(el, cq, m, 8 * warp, sw, len, stage[warp]);
    if (lane == 0) s_T[warp] = T;
    __syncthreads();
    const uint32_t T0 = s_T[0], T1 = s_T[1], T2 = s_T[2], T3 = s_T[3], total = T0 + T1 + T2 + T3;
    // the unit's own slot, or space behind the slots
    const uint32_t need = pool_need(total);
    uint32_t po = unit * (uint32_t)(kRlePoolPerUnit / 4);
    if (W.slots == 0 || need > kRlePoolPerUnit) {
        if (tid == 0) {
            const unsigned long long a = W.slots + atomicAdd(reinterpret_cast<unsigned long long*>(W.counters + 2),
                                                             (unsigned long long)need);
            s_po = a + need <= W.pool_bytes ? (uint32_t)(a >> 2) : kRecode;
        }
        __syncthreads();
        po = s_po;
    }
    if (po != kRecode) {                              // the streams one after the other, then whole sectors
        uint8_t* flat = reinterpret_cast<uint8_t*>(el) + (warp > 0 ? T0 : 0u) + (warp > 1 ? T1 : 0u) + (warp > 2 ? T2 : 0u);
        for (uint32_t i = lane; i < T; i += 32) flat[i] = stage[warp][i];
        __syncthreads();
        uint4* o = reinterpret_cast<uint4*>(W.pool + 4 * (size_t)po);
        for (uint32_t i = tid; 16u * i < need; i += kCT) o[i] = reinterpret_cast<const uint4*>(el)[i];
    }
    if (tid == 0) {
        W.rec[unit] = ChunkRec{{(uint16_t)T0, (uint16_t)T1, (uint16_t)T2, (uint16_t)T3}, po, 0u};
        atomicAdd(W.groups + unit / kGroup, total);
        if (po == kRecode) W.again[atomicAdd(W.counters, 1u)] = unit;
    }
}

// Four 16-bit lanes in two words (planes 0,1 | planes 2,3).
struct P4 { uint32_t a, b; };

template <bool MAX>
__device__ __forceinline__ P4 combine(P4 x, P4 y)
{
    if (MAX) return {__vmaxu2(x.a, y.a), __vmaxu2(x.b, y.b)};
    return {x.a + y.a, x.b + y.b};   // lanes never carry: every sum < 65536
}

__device__ __forceinline__ uint32_t lane16(P4 v, int p)
{
    const uint32_t w = p < 2 ? v.a : v.b;
    return (p & 1) ? (w >> 16) : (w & 0xFFFFu);
}

// Warp-wide exclusive scan of P4 values; *total receives the warp's total.
template <bool MAX>
__device__ __forceinline__ P4 warp_scan4(P4 v, int lane, P4* total)
{
    P4 inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        P4 y;
        y.a = __shfl_up_sync(0xffffffffu, inc.a, o);
        y.b = __shfl_up_sync(0xffffffffu, inc.b, o);
        if (lane >= o) inc = combine<MAX>(inc, y);
    }
    total->a = __shfl_sync(0xffffffffu, inc.a, 31);
    total->b = __shfl_sync(0xffffffffu, inc.b, 31);
    P4 ex;
    ex.a = __shfl_up_sync(0xffffffffu, inc.a, 1);
    ex.b = __shfl_up_sync(0xffffffffu, inc.b, 1);
    if (lane == 0) ex = {0u, 0u};
    return ex;
}

// The most significant bit of each byte of w, gathered into bits 0..3.
__device__ __forceinline__ uint32_t byte_msbs(uint32_t w)
{
    return ((w & 0x80808080u) * 0x00204081u) >> 28;
}

// 4-bit mask of the bytes of a and b that are equal (bit i = byte i).
__device__ __forceinline__ uint32_t eq_bytes(uint32_t a, uint32_t b)
{
    const uint32_t x = a ^ b;                                   // zero byte <=> equal
    const uint32_t t = ~(((x & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | x | 0x7F7F7F7Fu);
    return byte_msbs(t);
}

// Bits [lo, hi) set (0 <= lo, hi <= 31).
__device__ __forceinline__ uint32_t bit_range(int lo, int hi)
{
    lo = max(lo, 0);
    hi = min(hi, 31);
    return hi > lo ? ((1u << hi) - 1u) & ~((1u << lo) - 1u) : 0u;
}

// Dense path, a CTA of 8 warps per chunk: every position is classified with
// byte-SIMD bit masks, all four planes at once.  Warp k takes positions
// [512 k, 512 k + 512): lane l holds positions [P0, P0 + 16), P0 = 16 (32 k +
// l), in registers, and the bytes just before and after them come from its
// neighbours (shuffles; lane 0 and lane 31 load the neighbouring words).  A
// byte lies in a repeat iff one of the three windows of 3 around it is
// constant.  A max-scan of segment starts (warp scans, then the warps' totals
// through shared memory) cuts tokens every 128 bytes of a segment, and a
// sum-scan of output bytes (likewise) places them.  The four streams go to
// `stage` back to back, their sizes to T.  The stage takes the scattered bytes:
// a lane's literals are written in position order, one predicated store each,
// so the lanes of a warp stay together whatever their tokens.  xw: 16 P4 of
// shared memory.  The caller synchronises before it reads the stage.
// Bound by instruction issue: the dense chunks of 8 shaded 1920x1080 sources
// (colour and depth, 68 MB) take 95 us, and 16 us to be placed;
// sizing them (45 us) and coding them again to their place with scattered
// byte stores (134 us) came before.
__device__ __forceinline__ void dense_chunk(const RleJobDesc& jb, uint32_t q0, int len, bool sw, uint32_t* T,
                                            uint8_t* stage, P4* xw)
{
    const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
    const bool act = 512 * k < len;                          // (uniform in the warp)
    const int P0 = 16 * (32 * k + lane);
    uint32_t REP[4] = {0u, 0u, 0u, 0u}, SEG[4] = {0u, 0u, 0u, 0u};
    uint4 bytes[4];
    uint32_t VALID = 0u;
    P4 mine = {0u, 0u};
    // plane words of positions [q, q + 4) (word b = plane b)
    auto load_planes = [&](int q) {
        const uint4 g = load_elems(jb, q0, len, q);
        uint4 t = transpose4(g.x, g.y, g.z, g.w);
        if (sw) rlec::swizzle_planes(t.x, t.y, t.z, t.w);
        return t;
    };
    if (act) {
        uint4 t[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) t[i] = load_planes(P0 + 4 * i);
        uint4 tn = make_uint4(0u, 0u, 0u, 0u), tp = make_uint4(0u, 0u, 0u, 0u);
        if (lane == 31) tn = load_planes(P0 + 16);
        if (lane == 0 && P0 > 0) tp = load_planes(P0 - 4);
        const uint32_t VQ = bit_range(4 - P0, len - P0 + 4);          // 0 <= q < len
        const uint32_t VEQ = bit_range(5 - P0, len - P0 + 4);         // 1 <= q < len
        const uint32_t HIGH = bit_range(len - P0 + 4, 24);            // q >= len
        const uint32_t Q0 = P0 == 0 ? (1u << 4) : 0u;                 // q == 0
        VALID = (VQ >> 4) & 0xFFFFu;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            auto pw = [&](const uint4& x) { return b == 0 ? x.x : b == 1 ? x.y : b == 2 ? x.z : x.w; };
            const uint4 v = make_uint4(pw(t[0]), pw(t[1]), pw(t[2]), pw(t[3]));
            uint32_t wm = __shfl_up_sync(0xffffffffu, v.w, 1);
            if (lane == 0) wm = pw(tp);
            uint32_t wp = __shfl_down_sync(0xffffffffu, v.x, 1);
            if (lane == 31) wp = pw(tn);
            bytes[b] = v;
            // eq bit i: byte at position P0-4+i equals its predecessor
            uint32_t EQ = eq_bytes(wm, wm << 8);
            EQ |= eq_bytes(v.x, __funnelshift_l(wm, v.x, 8)) << 4;
            EQ |= eq_bytes(v.y, __funnelshift_l(v.x, v.y, 8)) << 8;
            EQ |= eq_bytes(v.z, __funnelshift_l(v.y, v.z, 8)) << 12;
            EQ |= eq_bytes(v.w, __funnelshift_l(v.z, v.w, 8)) << 16;
            EQ |= eq_bytes(wp, __funnelshift_l(v.w, wp, 8)) << 20;
            EQ &= VEQ & ~1u;                                          // bit 0 has no predecessor here
            const uint32_t T3 = EQ & (EQ << 1);                       // positions i-2, i-1, i equal
            const uint32_t R = (T3 | (T3 >> 1) | (T3 >> 2)) & VQ;     // byte lies in a run >= 3
            const uint32_t Sg = (((R & ~EQ) | (~R & (R << 1))) & VQ) | HIGH | Q0;
            REP[b] = (R >> 4) & 0xFFFFu;
            SEG[b] = (Sg >> 4) & 0x1FFFFu;                            // bit 16: position P0+16
        }
        // last segment start in each lane's range (position + 1)
        uint32_t l[4];
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const uint32_t m = SEG[b] & 0xFFFFu;
            l[b] = m ? (uint32_t)(P0 + 31 - __clz(m) + 1) : 0u;
        }
        mine.a = l[0] | (l[1] << 16);
        mine.b = l[2] | (l[3] << 16);
    }
    // max-scan over the chunk: in the warp, then over the warps before
    P4 tmax = {0u, 0u}, smax = {0u, 0u};
    if (act) smax = warp_scan4<true>(mine, lane, &tmax);
    if (lane == 0) xw[k] = tmax;
    __syncthreads();
    P4 before = smax;
    for (int j = 0; j < k; ++j) before = combine<true>(before, xw[j]);
    // piece starts (tokens hold <= 128 bytes) and output sizes
    uint32_t PSV[4], PE[4], cost[4];
    int sbin[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const uint32_t seg16 = SEG[b] & 0xFFFFu;
        const int sb_in = (int)lane16(before, b) - 1;            // -1 only for position 0
        sbin[b] = sb_in;
        uint32_t PS = seg16;
        const int first = seg16 ? __ffs(seg16) - 1 : 16;
        if (sb_in >= 0) {                                        // continuing segment
            const int r = (P0 - sb_in) & 127;
            const int d = r ? 128 - r : 0;
            if (d < first) PS |= 1u << d;
        }
        const int sb15 = seg16 ? P0 + 31 - __clz(seg16) : sb_in;
        const uint32_t next = ((SEG[b] >> 16) & 1u) | (((P0 + 16 - sb15) & 127) == 0 ? 1u : 0u);
        PSV[b] = PS & VALID;
        PE[b] = ((PS | (next << 16)) >> 1) & VALID;
        cost[b] = __popc((~REP[b] & VALID) | (PSV[b] & REP[b])) + __popc(PSV[b]);
    }
    P4 tsum = {0u, 0u}, ssum = {0u, 0u};
    if (act) ssum = warp_scan4<false>(P4{cost[0] | (cost[1] << 16), cost[2] | (cost[3] << 16)}, lane, &tsum);
    if (lane == 0) xw[8 + k] = tsum;
    __syncthreads();
    P4 off0 = ssum, total = {0u, 0u};
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const P4 x = xw[8 + j];
        if (j < k) off0 = combine<false>(off0, x);
        total = combine<false>(total, x);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b) T[b] = lane16(total, b);
    uint8_t* plane = stage;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        if (act) {
            uint8_t* const o = plane + lane16(off0, b);
            const uint32_t lit = ~REP[b] & VALID, psv = PSV[b], rep = REP[b], seg16 = SEG[b] & 0xFFFFu;
            const uint4 v = bytes[b];
            // literal bytes in position order; a piece start leaves room for its
            // control byte, a repeat's for its value too.  Warps without
            // literals skip the pass, warps of literals only (noise) need no
            // tests for them.
            uint8_t* w = o;
            if (__all_sync(0xffffffffu, lit == 0xFFFFu)) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const uint32_t wd = i < 4 ? v.x : i < 8 ? v.y : i < 12 ? v.z : v.w;
                    w += (psv >> i) & 1u;
                    w[i] = (uint8_t)(wd >> (8 * (i & 3)));
                }
            } else if (__any_sync(0xffffffffu, lit != 0u)) {
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const uint32_t wd = i < 4 ? v.x : i < 8 ? v.y : i < 12 ? v.z : v.w;
                    if ((psv >> i) & 1u) w += 1 + ((rep >> i) & 1u);
                    if ((lit >> i) & 1u) *w++ = (uint8_t)(wd >> (8 * (i & 3)));
                }
            }
            // control bytes, at the pieces' ends
            for (uint32_t m = PE[b]; m; m &= m - 1u) {
                const int i = __ffs(m) - 1;
                const uint32_t le = (2u << i) - 1u;
                uint8_t* const e = o + __popc((lit | (psv & rep)) & le) + __popc(psv & le);   // past the piece
                const uint32_t h = seg16 & le;
                const int sbk = h ? P0 + 31 - __clz(h) : sbin[b];
                const uint32_t jj = (uint32_t)(P0 + i - sbk) & 127u;
                if ((rep >> i) & 1u) {
                    const uint32_t wd = i < 8 ? (i < 4 ? v.x : v.y) : (i < 12 ? v.z : v.w);
                    e[-2] = (uint8_t)(0x80u + jj);
                    e[-1] = (uint8_t)(wd >> (8 * (i & 3)));
                } else {
                    *(e - 2 - jj) = (uint8_t)jj;
                }
            }
        }
        plane += T[b];
    }
}

// ---- basic RLE (mode 0) on the same pipeline --------------------------------
// Thesis 5.5.1's basic RLE codes 8-byte units (element pairs) in one stream
// per chunk.  The coding kernel lists the chunk's unit change points (units
// that differ from their predecessor) as it lists element change points for
// the four-plane modes; a run of one unit is literal, maximal spans of literal
// units become literal tokens and longer runs repeat tokens, both at most 128
// units per token, full tokens first.  Chunks with more change points than the
// list holds are coded by a CTA per chunk from the image (code0_block).
constexpr int kU = kChunk / 2;                       // units per chunk
constexpr int kUPer = kU / kT;                       // 8 per thread of a CTA
constexpr int kStage0 = 8 * kU + kU / 128 + 32;      // worst case + room for copy_out's read-ahead

__device__ __forceinline__ void put8(uint8_t* p, uint32_t lo, uint32_t hi)
{
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        p[k] = (uint8_t)(lo >> (8 * k));
        p[4 + k] = (uint8_t)(hi >> (8 * k));
    }
}

// Append the unit change points among units [kQ/2 qi, kQ/2 qi + kQ/2) of the
// chunk (unit k = elements 2k, 2k + 1) to W.cq (the unit's index) and W.ce,
// W.ch (its two elements); a lane's 16-byte group holds two units.  Every lane
// flags the changes in its group of each of the quarter's four 128-element
// groups; one warp scan of the four per-lane counts, packed in the bytes of a
// word (a group has at most 64 changes, so no byte carries into the next),
// places them all in order.  carry: the unit before the quarter (updated to the
// quarter's last).  Returns false once the chunk has more than kCap change
// points.
__device__ bool detect_quarter0(const uint32_t* data, int len, int qi, WarpRing& W, int& m, uint2& carry)
{
    const int lane = threadIdx.x & 31;
    constexpr int G = kQ / 128;
    static_assert(G == 4, "four groups' counts in the bytes of one word");
    uint4 vv[G];
    uint2 pv[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
        vv[g] = *reinterpret_cast<const uint4*>(data + 128 * g + 4 * lane);
        pv[g] = *reinterpret_cast<const uint2*>(data + 128 * g + 4 * lane - 2);   // g = lane = 0: guard words
    }
    if (lane == 0) pv[0] = qi == 0 ? make_uint2(~vv[0].x, vv[0].y) : carry;     // unit 0 is always listed
    carry = make_uint2(__shfl_sync(0xffffffffu, vv[G - 1].z, 31), __shfl_sync(0xffffffffu, vv[G - 1].w, 31));
    const int uend = min(len / 2 - kQ / 2 * qi, kQ / 2);                         // units of this quarter
    uint32_t f[G], packed = 0u;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const uint4 v = vv[g];
        const int u = 64 * g + 2 * lane;                  // within the quarter
        f[g] = (uint32_t)(v.x != pv[g].x || v.y != pv[g].y) | ((uint32_t)(v.z != v.x || v.w != v.y) << 1);
        if (u + 2 > uend) f[g] &= u >= uend ? 0u : 1u;
        packed |= (uint32_t)__popc(f[g]) << (8 * g);
    }
    // one warp scan of the four groups' per-lane counts (bytes of a word)
    uint32_t inc = packed;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31), exc = inc - packed;
    const int cnt = (int)((tot & 0xFFu) + ((tot >> 8) & 0xFFu) + ((tot >> 16) & 0xFFu) + (tot >> 24));
    if (m + cnt > kCap) return false;
    int base = m;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        if (f[g]) {
            const uint4 v = vv[g];
            const int uu = kQ / 2 * qi + 64 * g + 2 * lane;
            int o = base + (int)((exc >> (8 * g)) & 0xFFu);
            if (f[g] & 1u) { W.cq[o] = (uint16_t)uu; W.ce[o] = v.x; W.ch[o] = v.y; ++o; }
            if (f[g] & 2u) { W.cq[o] = (uint16_t)(uu + 1); W.ce[o] = v.z; W.ch[o] = v.w; }
        }
        base += (int)((tot >> (8 * g)) & 0xFFu);
    }
    m += cnt;
    return true;
}

// Mode 0, sparse path: the tokens of a chunk of nu units from its m <= 128
// unit change points (run i starts at unit cq[i], its unit is (ce[i], ch[i]),
// and it ends where run i + 1 starts, or at nu).  Lane l takes runs 4l .. 4l+3.
// A warp max-scan gives every literal run the start of its span, a sum-scan
// the place of its bytes; a repeat run writes its tokens, a literal unit its
// 8 bytes, and the unit that ends a literal token the token's control byte.
// Returns the bytes written.
__device__ uint32_t code_sparse0(const uint32_t* ce, const uint32_t* ch, const uint16_t* cq, int m, int nu,
                                 uint8_t* out)
{
    const int lane = threadIdx.x & 31;
    const int i0 = 4 * lane;
    int s[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) s[k] = i0 + k < m ? (int)cq[i0 + k] : nu;
    uint32_t lit = 0u;                                    // bit k: run i0 + k is one unit
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (i0 + k < m && s[k + 1] - s[k] == 1) lit |= 1u << k;
    const uint32_t litn = __shfl_down_sync(0xffffffffu, lit, 1);
    const uint32_t litp = __shfl_up_sync(0xffffffffu, lit, 1);
    const uint32_t lx = lit | ((lane < 31 ? (litn & 1u) : 0u) << 4);   // bit 4: the next lane's first run
    const uint32_t pre = (lit << 1) | (lane > 0 ? ((litp >> 3) & 1u) : 0u);   // bit k: run i0 + k - 1 literal
    const uint32_t starts = lit & ~pre;                   // literal runs that start a span
    // the last span start up to each lane (index + 1; 0: none)
    uint32_t last = starts ? (uint32_t)(i0 + 32 - __clz(starts)) : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, last, o);
        if (lane >= o) last = max(last, y);
    }
    uint32_t S0 = __shfl_up_sync(0xffffffffu, last, 1);
    if (lane == 0) S0 = 0u;
    uint32_t sz = 0u, S = S0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (i0 + k >= m) break;
        if ((starts >> k) & 1u) S = (uint32_t)(i0 + k + 1);
        if ((lit >> k) & 1u) sz += ((uint32_t)(i0 + k) - (S - 1u)) % 128u == 0u ? 9u : 8u;
        else sz += 9u * (((uint32_t)(s[k + 1] - s[k]) + 127u) / 128u);
    }
    uint32_t inc = sz;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
    uint32_t P = inc - sz;
    S = S0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = i0 + k;
        if (i >= m) break;
        const uint32_t lo = ce[i], hi = ch[i];
        if ((starts >> k) & 1u) S = (uint32_t)(i + 1);
        if ((lit >> k) & 1u) {
            const uint32_t p = ((uint32_t)i - (S - 1u)) % 128u;   // place in its token
            const uint32_t ts = p == 0u ? 1u : 0u;
            put8(out + P + ts, lo, hi);
            P += 8u + ts;
            if (p == 127u || !((lx >> (k + 1)) & 1u)) out[P - 8u * (p + 1u) - 1u] = (uint8_t)p;
        } else {
            for (uint32_t L = (uint32_t)(s[k + 1] - s[k]); L > 0u;) {
                const uint32_t piece = min(L, 128u);
                out[P] = (uint8_t)(127u + piece);
                put8(out + P + 1u, lo, hi);
                P += 9u;
                L -= piece;
            }
        }
    }
    return total;
}

// Exclusive block scan (sum, or max with identity 0) of one value per thread;
// *total receives the reduction over the block.
template <bool MAX>
__device__ __forceinline__ uint32_t block_excl(uint32_t v, uint32_t* wt, uint32_t* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc = MAX ? max(inc, y) : inc + y;
    }
    if (lane == 31) wt[warp] = inc;
    __syncthreads();
    uint32_t pre = 0, tot = 0;
#pragma unroll
    for (int w = 0; w < kT / 32; ++w) {
        const uint32_t t = wt[w];
        if (w < warp) pre = MAX ? max(pre, t) : pre + t;
        tot = MAX ? max(tot, t) : tot + t;
    }
    uint32_t ex = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) ex = 0u;
    *total = tot;
    __syncthreads();                                  // wt is reused by the next scan
    return MAX ? max(pre, ex) : pre + ex;
}

// Mode 0, dense path: one CTA of kT threads codes chunk [q0, q0 + len) of the
// job into stage and returns its size (the odd tail element included).  The
// chunk's elements go to e in shared memory; each thread reads its 8
// consecutive units and the two on either side into registers once (16-byte
// reads).  A unit equal to a neighbour belongs to a repeat run, the others form
// literal spans; a block max-scan gives every unit its segment's start (a run,
// or a maximal span of single units), a block sum-scan the place of its bytes,
// and the unit that ends a token writes the token's control byte.
__device__ uint32_t code0_block(const RleJobDesc& jb, uint32_t q0, int len, uint32_t* e, uint8_t* stage,
                                uint32_t* wt)
{
    const int tid = threadIdx.x;
    for (int t = tid; 4 * t < len; t += kT)
        *reinterpret_cast<uint4*>(e + 4 * t) = load_elems(jb, q0, len, 4 * t);
    __syncthreads();
    const int nu = len / 2;
    const int k0 = tid * kUPer;
    uint32_t ul[kUPer + 4], uh[kUPer + 4];           // [0,1] = k0-2, k0-1; [2..9] = k0..k0+7; [10,11] = k0+8, k0+9
    {
        const uint4* e4 = reinterpret_cast<const uint4*>(e);
        const uint4 m = tid > 0 ? e4[4 * tid - 1] : make_uint4(0u, 0u, 0u, 0u);
        ul[0] = m.x; uh[0] = m.y; ul[1] = m.z; uh[1] = m.w;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const uint4 v = e4[4 * tid + g];
            ul[2 + 2 * g] = v.x; uh[2 + 2 * g] = v.y; ul[3 + 2 * g] = v.z; uh[3 + 2 * g] = v.w;
        }
        const uint4 n = tid + 1 < kT ? e4[4 * tid + 4] : make_uint4(0u, 0u, 0u, 0u);
        ul[10] = n.x; uh[10] = n.y; ul[11] = n.z; uh[11] = n.w;
    }
    // eqp bit i: unit k0-2+i equals its predecessor (both exist), i = 0 .. 11
    uint32_t eqp = 0u;
#pragma unroll
    for (int i = 1; i < kUPer + 4; ++i) {
        const int k = k0 - 2 + i;
        if (k >= 1 && k < nu && ul[i] == ul[i - 1] && uh[i] == uh[i - 1]) eqp |= 1u << i;
    }
    // lit bit i, i = 1 .. 10: unit k0-2+i exists and equals neither neighbour
    uint32_t lit = 0u;
#pragma unroll
    for (int i = 1; i < kUPer + 3; ++i) {
        const int k = k0 - 2 + i;
        if (k >= 0 && k < nu && !((eqp >> i) & 1u) && !((eqp >> (i + 1)) & 1u)) lit |= 1u << i;
    }
    // seg bit i, i = 2 .. 10: unit k0-2+i starts a run or a span
    uint32_t seg = 0u;
#pragma unroll
    for (int i = 2; i < kUPer + 3; ++i) {
        const int k = k0 - 2 + i;
        if (k >= nu) continue;
        const bool l = (lit >> i) & 1u, lp = (lit >> (i - 1)) & 1u;
        if (k == 0 || l != lp || (!l && !((eqp >> i) & 1u))) seg |= 1u << i;
    }
    uint32_t smax = 0, ssum = 0, tot = 0;
#pragma unroll
    for (int j = 0; j < kUPer; ++j)
        if (k0 + j < nu && ((seg >> (j + 2)) & 1u)) smax = (uint32_t)(k0 + j);
    const uint32_t carry = block_excl<true>(smax, wt, &tot);
    uint32_t S = carry;
#pragma unroll
    for (int j = 0; j < kUPer; ++j) {
        const int k = k0 + j;
        if (k >= nu) break;
        if ((seg >> (j + 2)) & 1u) S = (uint32_t)k;
        const bool ts = ((uint32_t)k - S) % 128u == 0u;
        ssum += ((lit >> (j + 2)) & 1u) ? 8u + (ts ? 1u : 0u) : (ts ? 9u : 0u);
    }
    uint32_t body = 0;
    uint32_t P = block_excl<false>(ssum, wt, &body);
    S = carry;
#pragma unroll
    for (int j = 0; j < kUPer; ++j) {
        const int k = k0 + j;
        if (k >= nu) break;
        if ((seg >> (j + 2)) & 1u) S = (uint32_t)k;
        const bool l = (lit >> (j + 2)) & 1u;
        const uint32_t pos = (uint32_t)k - S;
        const bool ts = pos % 128u == 0u;
        const uint32_t sz = l ? 8u + (ts ? 1u : 0u) : (ts ? 9u : 0u);
        const bool te = k + 1 == nu || ((seg >> (j + 3)) & 1u) || ((uint32_t)k + 1u - S) % 128u == 0u;
        const uint32_t L = pos % 128u + 1u;          // units of the token so far
        if (l) {
            put8(stage + P + (ts ? 1u : 0u), ul[j + 2], uh[j + 2]);
            if (te) stage[P + sz - 1u - 8u * L] = (uint8_t)(L - 1u);
        } else {
            if (ts) put8(stage + P + 1u, ul[j + 2], uh[j + 2]);
            if (te) stage[P + sz - 9u] = (uint8_t)(128u + L - 1u);
        }
        P += sz;
    }
    if ((len & 1) && tid == 0) {
        const uint32_t v = e[len - 1];
#pragma unroll
        for (int k = 0; k < 4; ++k) stage[body + k] = (uint8_t)(v >> (8 * k));
    }
    __syncthreads();                                  // the stage is complete
    return body + ((len & 1) ? 4u : 0u);
}

// Mode-0 coding kernel.  Per chunk a warp: takes its next ticket; reads the
// chunk's eight quarters, refilling each slot as soon as it has been read (with
// the next quarter of this chunk or of the next one); codes the stream; and
// leaves the chunk's record and, for a sparse chunk, its stream in the
// pool (space from the warp's slab, a fresh slab taken with one atomic on the
// pool cursor when the chunk does not fit, or from the cursor chunk by chunk
// when slab is 0; a chunk that finds the pool full is coded again when
// placed, like a dense one; such chunks are listed for the recoding kernel).
// No warp waits for another.
template <int N>
__global__ void __launch_bounds__(32 * kWPB, 16)
k_rle_compress0(const __grid_constant__ RleJobList<N> J, ChunkRec* rec, uint32_t* recode, uint8_t* pool,
                uint32_t pool_bytes, uint32_t slab, uint32_t* ticket, uint32_t* status)
{
    extern __shared__ __align__(16) uint8_t smem[];
    WarpRing& W = reinterpret_cast<WarpRing*>(smem)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const uint32_t T = J.total_units;
    chain_wait();
    unsigned long long* cursor = reinterpret_cast<unsigned long long*>(ticket + 2);   // pool bytes taken
    if (lane == 0) {
        for (int q = 0; q < kSlots; ++q) mbar_init(&W.full[q], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    uint32_t sb = 0u, sl = 0u;                          // lane 0: the warp's pool slab (base, bytes left)
    uint32_t cur = 0u;
    if (lane == 0) cur = atomicAdd(ticket, 1u);
    cur = __shfl_sync(0xffffffffu, cur, 0);
    int ji = cur < T ? find_job(J, cur) : 0;            // job of the current chunk
    if (cur < T)
        for (int q = 0; q < kSlots; ++q) issue_quarter(J.j[ji], cur, q, q, W);
    for (uint32_t qs = 0; cur < T;) {                   // qs: the warp's quarter sequence number
        uint32_t nxt = 0u;
        if (lane == 0) nxt = atomicAdd(ticket, 1u);
        nxt = __shfl_sync(0xffffffffu, nxt, 0);
        const RleJobDesc& jb = J.j[ji];
        const int jn = nxt < T ? find_job(J, nxt) : 0;
        const uint32_t nc = jb.n_chunks;
        const uint32_t q0 = nc ? (cur - jb.first_unit) * (uint32_t)kChunk : 0u;
        const int len = nc ? (int)min((uint32_t)kChunk, (uint32_t)jb.w * (uint32_t)jb.h - q0) : 0;
        int m = 0;
        uint2 carry = make_uint2(0u, 0u);
        bool fits = true;
        // quarters [0, issued) of this chunk are in flight or read; once the chunk
        // proves dense its remaining quarters are not fetched, and the slots go
        // to the next chunk
        int issued = kSlots;
        for (int q = 0; q < issued; ++q, ++qs) {
            const int slot = (int)(qs % kSlots);
            mbar_wait(&W.full[slot], (qs / kSlots) & 1u, status);
            if (fits && kQ * q < len) fits = detect_quarter0(W.buf[slot] + 4, len, q, W, m, carry);
            // the quarter's values have all been consumed (compared, voted on) by
            // now, so its reads are complete before the refill below starts
            __syncwarp();
            // refill the slot with the next quarter, of this chunk or of the next
            if (fits && issued < kQPC) issue_quarter(jb, cur, issued++, slot, W);
            else if (nxt < T) issue_quarter(J.j[jn], nxt, q + kSlots - issued, slot, W);
        }
        if (nc > 0) {
            uint32_t total = 0u;                        // (a dense chunk is sized by the recoding kernel)
            if (fits) {
                __syncwarp();
                total = code_sparse0(W.ce, W.ch, W.cq, m, len / 2, W.stage);
                if (len & 1) {                            // the odd last element follows the tokens
                    if (lane == 0) put_u32(W.stage + total, __ldg(jb.src + elem_off(jb, q0 + (uint32_t)len - 1u)));
                    total += 4u;
                }
            }
            uint32_t po = kRecode;
            if (fits && lane == 0) {
                // (+ 4: the copy-out reads up to one word past a chunk's bytes)
                const uint32_t need = (total + 15u) & ~15u;
                if (slab == 0u) {                         // small pools: space per chunk
                    const unsigned long long a = atomicAdd(cursor, (unsigned long long)need);
                    if (a + total + 4u <= pool_bytes) po = (uint32_t)a;
                } else {
                    // space from the warp's own slab, one atomic per slab (a
                    // sparse chunk codes to at most 4 kStagePlane <= slab bytes)
                    if (need > sl) {
                        const unsigned long long a = atomicAdd(cursor, (unsigned long long)slab);
                        sl = a + slab + 4u <= pool_bytes ? slab : 0u;
                        sb = (uint32_t)a;
                    }
                    if (need <= sl) { po = sb; sb += need; sl -= need; }
                }
            }
            po = __shfl_sync(0xffffffffu, po, 0);
            __syncwarp();
            if (po != kRecode)
                for (uint32_t i = lane; i < total; i += 32) pool[po + i] = W.stage[i];
            if (lane == 0) {
                ChunkRec r;
                r.T[0] = (uint16_t)total; r.T[1] = r.T[2] = r.T[3] = 0;
                r.pool = po == kRecode ? kRecode : po >> 2;
                r.off = 0u;
                rec[cur] = r;
                if (po == kRecode) recode[atomicAdd(ticket + 1, 1u)] = cur;   // coded again when placed
            }
            __syncwarp();
        }
        cur = nxt;
        ji = jn;
    }
}

// Clears the counters and the groups' sums.
__global__ void k_rle_begin(uint4* counters, uint32_t* groups, uint32_t n)
{
    chain_wait();
    const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *counters = make_uint4(0u, 0u, 0u, 0u);
    if (i < n) groups[i] = 0u;
}

// Mode 0's scan kernel: one CTA per job.  The exclusive prefix of the job's
// chunk sizes gives every chunk its offset in the payload (written to its
// record); the job's header and stream size are written here too.
template <int N>
__global__ void __launch_bounds__(1024)
k_rle_scan(const __grid_constant__ RleJobList<N> J, ChunkRec* rec)
{
    __shared__ uint32_t wsum[32];
    const RleJobDesc& jb = J.j[blockIdx.x];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    chain_wait();
    uint8_t* dst = reinterpret_cast<uint8_t*>(jb.dst);
    const uint32_t nc = jb.n_chunks;
    if (nc == 0) {                                    // empty image: header only
        if (tid == 0) {
            write_header(dst, jb);
            *jb.d_size = 32u;
        }
        return;
    }
    ChunkRec* R = rec + jb.first_unit;
    const uint32_t per = (nc + blockDim.x - 1) / blockDim.x;   // contiguous chunks per thread
    const uint32_t c0 = min(nc, tid * per), c1 = min(nc, c0 + per);
    uint32_t mine = 0u;
    for (uint32_t c = c0; c < c1; ++c) mine += (uint32_t)R[c].T[0] + R[c].T[1] + R[c].T[2] + R[c].T[3];
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    uint32_t base = inc - mine;
    for (int k = 0; k < warp; ++k) base += wsum[k];
    for (uint32_t c = c0; c < c1; ++c) {
        R[c].off = base;
        base += (uint32_t)R[c].T[0] + R[c].T[1] + R[c].T[2] + R[c].T[3];
    }
    if (tid == (int)blockDim.x - 1) {                 // its base is now the job's total
        write_header(dst, jb);
        *jb.d_size = 32ull + (jb.mode == 0 ? 4ull : 16ull) * nc + base;
    }
}

constexpr int kPlaceLanes = 8;

// Mode 0's placing kernel: kPlaceLanes lanes (a quarter-warp) per chunk copy its
// stream from the pool to its place and write its end-table entry, so a warp's
// four chunks have their loads in flight together.  Listed chunks are left to
// the recoding kernel.
template <int N>
__global__ void __launch_bounds__(128, 8)
k_rle_place(const __grid_constant__ RleJobList<N> J, const ChunkRec* rec, const uint8_t* pool)
{
    chain_wait();
    const uint32_t unit = blockIdx.x * (128u / kPlaceLanes) + threadIdx.x / kPlaceLanes;
    const int lane = (int)threadIdx.x % kPlaceLanes;
    if (unit >= J.total_units) return;
    const ChunkRec r = rec[unit];                     // (in flight during the job search)
    const RleJobDesc& jb = J.j[find_job(J, unit)];
    const uint32_t nc = jb.n_chunks;
    if (nc == 0 || r.pool == kRecode) return;         // (an empty image's header is written by the scan)
    uint8_t* dst = reinterpret_cast<uint8_t*>(jb.dst);
    copy_out(dst + 32 + 4ull * nc + r.off, pool + 4ull * r.pool, r.T[0], lane, kPlaceLanes);
    if (lane == 0) put_u32(dst + 32 + 4ull * (unit - jb.first_unit), r.off + r.T[0]);
}

// Bytes of the chunks [f, u), from the groups' sums where they lie inside: the
// part of one of kRT threads.
constexpr uint32_t kRT = 256;
__device__ __forceinline__ uint32_t bytes_between(const RleScratch& W, uint32_t f, uint32_t u, uint32_t tid)
{
    auto of = [&](uint32_t c) {
        const ChunkRec& r = W.rec[c];
        return (uint32_t)r.T[0] + r.T[1] + r.T[2] + r.T[3];
    };
    const uint32_t g0 = (f + kGroup - 1) / kGroup, g1 = u / kGroup;
    uint32_t sum = 0u;
    if (g0 >= g1) {                                   // (then fewer than 2 kGroup chunks)
        if (f + tid < u) sum = of(f + tid);
        return sum;
    }
    if (tid < kGroup) {
        if (f + tid < kGroup * g0) sum = of(f + tid);
    } else if (tid < 2 * kGroup) {
        if (kGroup * g1 + tid - kGroup < u) sum = of(kGroup * g1 + tid - kGroup);
    }
    for (uint32_t g = g0 + tid; g < g1; g += kRT) sum += W.groups[g];
    return sum;
}

__device__ __forceinline__ uint32_t warp_sum(uint32_t v)
{
    return __reduce_add_sync(0xffffffffu, v);
}

// Placing, a CTA per kGroup chunks.  A chunk's place is the sum of its image's
// chunks before it: the groups' sums up to the CTA's first chunk and a scan of
// the CTA's own.  kPlaceLanes lanes copy a sparse chunk, so a warp's four have
// their loads in flight together (a dense one is another CTA's); the end-table
// entries, and with an image's last chunk its header and stream size, are
// written here for all chunks.  (A scan launch of a CTA per image between the
// coding and the placing launch took 2.9 us more: 8.1 us for both against 5.2 us
// for the 32 pieces of a 1920x1080 swap's level.)
template <int N>
__device__ __forceinline__ void place_group(const RleJobList<N>& J, const RleScratch& W, uint32_t group, uint32_t* sum)
{
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = kGroup * group;
    const uint32_t k = tid / kPlaceLanes, sub = tid % kPlaceLanes, unit = b + k;
    const bool in = unit < J.total_units;
    const ChunkRec r = in ? W.rec[unit] : ChunkRec{{0, 0, 0, 0}, kRecode, 0u};
    uint32_t own = 0u;                                // lane i: the size of the group's i-th chunk
    if (b + lane < J.total_units) {
        const ChunkRec& o = W.rec[b + lane];
        own = (uint32_t)o.T[0] + o.T[1] + o.T[2] + o.T[3];
    }
    const RleJobDesc& jb = J.j[find_job(J, in ? unit : J.total_units - 1u)];
    const uint32_t nc = jb.n_chunks, f = jb.first_unit, f0 = J.j[find_job(J, b)].first_unit;
    const uint32_t part = warp_sum(bytes_between(W, f0, b, tid));
    if (lane == 0) sum[warp] = part;
    __syncthreads();
    uint32_t base = 0u;
#pragma unroll
    for (int i = 0; i < (int)kRT / 32; ++i) base += sum[i];
    const uint32_t ex = (uint32_t)rlec::warp_incl_sum((int)own, (int)lane) - own;
    const uint32_t pk = __shfl_sync(0xffffffffu, ex, k), pf = __shfl_sync(0xffffffffu, ex, (f - b) & 31u);
    const uint32_t off = f < b ? base + pk : pk - pf;
    const uint32_t T0 = r.T[0], T1 = r.T[1], T2 = r.T[2], T3 = r.T[3], total = T0 + T1 + T2 + T3;
    uint8_t* const dst = reinterpret_cast<uint8_t*>(jb.dst);
    if (!in) return;
    if (nc > 0 && !(r.pool & kDense)) copy_out(dst + 32 + 16ull * nc + off, W.pool + 4ull * r.pool, total, sub, kPlaceLanes);
    if (nc > 0) {
        const uint32_t mine = sub == 0 ? T0 : sub == 1 ? T0 + T1 : sub == 2 ? T0 + T1 + T2 : total;
        if (sub < 4) put_u32(dst + 32 + 16ull * (unit - f) + 4u * sub, off + mine);
    }
    if (sub == 0 && (nc == 0 || unit - f == nc - 1u)) {
        write_header(dst, jb);
        *jb.d_size = 32ull + 16ull * nc + (nc ? off + total : 0u);
    }
}

// Recoding kernels, a CTA of 8 warps per listed chunk over a persistent grid.
// Before placing (PLACE false) the dense chunks are coded from the image into
// the stage; their sizes go to their records and their groups' sums and, where
// the pool has room, their streams to the pool with 16-byte stores.  The
// placing launch (PLACE true) copies the pooled ones to their place; the others,
// and the sparse ones that found the pool full, are coded (again) from the image
// and copied from the stage.  Its first CTAs place the sparse chunks.
constexpr int kDenseStage = 4 * (kChunk + kChunk / 128) + 64;   // all literals, copy_out's read-ahead, whole sectors

template <int N, bool PLACE>
__global__ void __launch_bounds__(kRT, 4)
k_rle_recode(const __grid_constant__ RleJobList<N> J, const RleScratch W, uint32_t grid)
{
    __shared__ P4 xw[16];
    __shared__ __align__(16) uint8_t stage[kDenseStage];
    __shared__ uint32_t s_pool, s_sum[kRT / 32];
    chain_wait();
    const int tid = threadIdx.x;
    uint32_t first = blockIdx.x;
    if (PLACE) {
        const uint32_t groups = gridDim.x - grid;
        if (first < groups) {
            place_group(J, W, first, s_sum);
            return;
        }
        first -= groups;
    }
    const uint32_t dense = W.counters[1], n = dense + (PLACE ? W.counters[0] : 0u);
    for (uint32_t i = first; i < n; i += grid) {
        const uint32_t unit = i < dense ? W.recode[i] : W.again[i - dense];
        const RleJobDesc& jb = J.j[find_job(J, unit)];
        const uint32_t q0 = (unit - jb.first_unit) * (uint32_t)kChunk;
        const int len = (int)min((uint32_t)kChunk, (uint32_t)jb.w * (uint32_t)jb.h - q0);
        uint32_t T[4];
        if (!PLACE) {
            dense_chunk(jb, q0, len, jb.mode == 2, T, stage, xw);
            const uint32_t total = T[0] + T[1] + T[2] + T[3];
            if (tid == 0) {
                const uint32_t need = pool_need(total);
                const unsigned long long a = W.slots + atomicAdd(reinterpret_cast<unsigned long long*>(W.counters + 2), (unsigned long long)need);
                s_pool = a + need <= W.pool_bytes ? kDense | (uint32_t)(a >> 4) : kRecode;
                W.rec[unit] = ChunkRec{{(uint16_t)T[0], (uint16_t)T[1], (uint16_t)T[2], (uint16_t)T[3]}, s_pool, 0u};
                atomicAdd(W.groups + unit / kGroup, total);
            }
            __syncthreads();                                  // the stage is complete
            if (s_pool != kRecode) {
                uint4* to = reinterpret_cast<uint4*>(W.pool + ((size_t)(s_pool & ~kDense) << 4));
                for (uint32_t j = tid; 32u * (j >> 1) < total + 4u; j += kRT)    // (whole 32-byte sectors)
                    to[j] = reinterpret_cast<const uint4*>(stage)[j];
            }
        } else {
            const ChunkRec r = W.rec[unit];
            const uint32_t part = warp_sum(bytes_between(W, jb.first_unit, unit, (uint32_t)tid));
            if ((tid & 31) == 0) s_sum[tid >> 5] = part;
            if (r.pool == kRecode) dense_chunk(jb, q0, len, jb.mode == 2, T, stage, xw);
            __syncthreads();                                  // (the stage is complete, too)
            uint32_t off = 0u;
#pragma unroll
            for (int k = 0; k < (int)kRT / 32; ++k) off += s_sum[k];
            const uint8_t* from = r.pool == kRecode ? stage : W.pool + ((size_t)(r.pool & ~kDense) << 4);
            copy_out(reinterpret_cast<uint8_t*>(jb.dst) + 32 + 16ull * jb.n_chunks + off, from,
                     (uint32_t)r.T[0] + r.T[1] + r.T[2] + r.T[3], tid, kRT);
        }
        __syncthreads();                                      // stage, xw and s_sum are reused
    }
}

// Mode-0 recoding kernels: as k_rle_recode, with one CTA per listed chunk
// (code0_block).  Before the scan (EMIT false) the dense chunks are sized;
// after it (EMIT true) every listed chunk is written to its place with its
// end-table entry.
template <int N, bool EMIT>
__global__ void __launch_bounds__(kT)
k_rle0_recode(const __grid_constant__ RleJobList<N> J, ChunkRec* rec, const uint32_t* recode, const uint32_t* count)
{
    __shared__ __align__(16) uint32_t e[kChunk];
    __shared__ __align__(16) uint8_t stage[kStage0];
    __shared__ uint32_t wt[kT / 32];
    const int tid = threadIdx.x;
    chain_wait();
    const uint32_t n = *count;
    for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) {
        const uint32_t unit = recode[i];
        const RleJobDesc& jb = J.j[find_job(J, unit)];
        const uint32_t nc = jb.n_chunks, c = unit - jb.first_unit;
        const ChunkRec r = rec[unit];
        if (!EMIT && r.T[0] != 0u) continue;              // sized already (a sparse chunk)
        const uint32_t q0 = c * (uint32_t)kChunk;
        const int len = (int)min((uint32_t)kChunk, (uint32_t)jb.w * (uint32_t)jb.h - q0);
        const uint32_t total = code0_block(jb, q0, len, e, stage, wt);
        if (!EMIT) {
            if (tid == 0) rec[unit].T[0] = (uint16_t)total;
        } else {
            uint8_t* dst = reinterpret_cast<uint8_t*>(jb.dst);
            copy_out(dst + 32 + 4ull * nc + r.off, stage, total, tid, kT);
            if (tid == 0) put_u32(dst + 32 + 4ull * c, r.off + total);
        }
        __syncthreads();                                  // e and stage are reused
    }
}

// Self-test of the bounded waits: a warp waits on an mbarrier that nothing
// arrives on; the wait gives up after its try limit, records EC_ERR_TIMEOUT
// and the kernel returns.
__global__ void k_selftest_wait(uint32_t* status)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    mbar_wait(&bar, 0u, status);
}

// ----------------------------------------------------------- decompress ----

constexpr int kDT = 128;        // decoder CTA: one warp per byte plane


// Mode 0 (basic 64-bit RLE): the chunk's one stream [b, e) of the payload is
// staged in shared memory.  Then, up to kTok0 tokens at a time, one thread
// walks the tokens (control byte, size, bounds) and lists each token's first
// unit and stream offset in tok, and the four warps write the listed tokens,
// one token per warp and a unit per lane (8-byte stores of the unit's two
// elements where the image allows).  A unit's 8 stream bytes are funnel-
// shifted out of three aligned shared-memory words.
constexpr int kTok0 = 256;

__device__ void decode_mode0(const RleJobDesc& jb, const uint8_t* pay, uint32_t b, uint32_t e, uint32_t q0,
                             int len, uint8_t* sbuf, uint32_t* tok, uint32_t* status)
{
    __shared__ uint32_t s_ntok, s_i, s_o, s_bad;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t w0 = b >> 2, wl = e >> 2;          // whole words [w0, wl), then bytes [4 wl, e)
    uint32_t* st = reinterpret_cast<uint32_t*>(sbuf);
    const uint32_t* p32 = reinterpret_cast<const uint32_t*>(pay);
    for (uint32_t i = tid; w0 + i < wl; i += kDT) st[i] = __ldg(p32 + w0 + i);
    if (tid < (int)(e - 4u * wl) && wl >= w0) sbuf[4u * (wl - w0) + tid] = __ldg(pay + 4u * wl + tid);
    if (tid == 0) { s_i = b; s_o = 0u; s_bad = 0u; }
    __syncthreads();
    const uint8_t* sb = sbuf - 4u * w0;                // stream byte i at sb[i]
    const uint32_t* sw = st - w0;                      // stream word j (bytes 4j .. 4j+3) at sw[j]
    uint32_t* dst = reinterpret_cast<uint32_t*>(jb.dst);
    const bool pairs = jb.vec != 0u;                   // a unit's elements are adjacent, 8-byte aligned
    const bool dense = jb.pitch == jb.w;
    const uint32_t nu = (uint32_t)len / 2u;
    for (;;) {
        if (tid == 0) {
            uint32_t i = s_i, o = s_o, k = 0u, bad = 0u;
            while (o < nu && k < (uint32_t)kTok0) {
                if (i >= e) { bad = 1u; break; }
                const uint32_t ctl = sb[i];
                const uint32_t m = ctl < 128u ? ctl + 1u : ctl - 127u;
                const uint32_t need = ctl < 128u ? 1u + 8u * m : 9u;
                if (o + m > nu || i + need > e) { bad = 1u; break; }
                tok[k++] = o | ((i - b) << 12);
                i += need;
                o += m;
            }
            s_ntok = k; s_i = i; s_o = o; s_bad = bad;
        }
        __syncthreads();
        const uint32_t ntok = s_ntok;
        for (uint32_t t = (uint32_t)warp; t < ntok; t += kDT / 32) {
            const uint32_t r = tok[t], o = r & 0xFFFu, i = b + (r >> 12);
            const uint32_t ctl = sb[i];
            const bool lit = ctl < 128u;
            const uint32_t m = lit ? ctl + 1u : ctl - 127u;
            for (uint32_t k = (uint32_t)lane; k < m; k += 32u) {
                const uint32_t x = i + 1u + (lit ? 8u * k : 0u);   // the unit's first stream byte
                const uint32_t sh = 8u * (x & 3u), j = x >> 2;
                const uint32_t a0 = sw[j], a1 = sw[j + 1], a2 = sw[j + 2];
                const uint32_t lo = __funnelshift_r(a0, a1, sh), hi = __funnelshift_r(a1, a2, sh);
                const uint32_t q = q0 + 2u * (o + k);
                if (pairs) {
                    const size_t eo = dense ? q : elem_off(jb, q);
                    __stcs(reinterpret_cast<uint2*>(dst + eo), make_uint2(lo, hi));
                } else {
                    dst[elem_off(jb, q)] = lo;
                    dst[elem_off(jb, q + 1u)] = hi;
                }
            }
        }
        const bool done = s_bad != 0u || s_o >= nu;
        __syncthreads();                              // tok and the shared words are reused
        if (done) break;
    }
    if (tid != 0) return;
    uint32_t i = s_i;
    bool bad = s_bad != 0u;
    if (!bad && (len & 1)) {
        if (i + 4u > e) bad = true;
        else {
            dst[elem_off(jb, q0 + (uint32_t)len - 1u)] =
                (uint32_t)sb[i] | ((uint32_t)sb[i + 1] << 8) | ((uint32_t)sb[i + 2] << 16) | ((uint32_t)sb[i + 3] << 24);
            i += 4u;
        }
    }
    if (!bad && i != e) bad = true;
    if (bad) set_status(status, EC_ERR_CORRUPT);
}

// Run path of the decoder (few runs): the chunk's elements are constant
// between the union of the four planes' run starts, so each such segment's
// element is assembled once (one byte per plane, found by the rank of the
// segment's start among that plane's run starts) and written with 16-byte
// stores of constant groups.  bm: the planes' run-start bitmaps [4][128];
// val: their run bytes [4][256]; work: shared scratch of kRunArea bytes
// (bitmaps included).
constexpr int kRunCap = 255;                        // runs per plane the run path takes
constexpr int kRunArea = 2048 + 1024 + 64;          // bitmaps, union with its prefix, warp totals

__device__ __forceinline__ void fill_segments(const RleJobDesc& jb, uint32_t q0, int len, bool sw, const uint32_t* bm,
                                              const uint8_t* val, uint8_t* work, uint32_t* dstp)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint2* UP = reinterpret_cast<uint2*>(work + 2048);           // [128] union of run starts, segments before it - 1
    uint2* wt = UP + 128;                                         // per-warp totals (scan)
    uint32_t* SV = reinterpret_cast<uint32_t*>(work + kRunArea + 1024);   // segment elements
    // word tid of every bitmap; exclusive prefixes of their bit counts
    const uint32_t b0 = bm[tid], b1 = bm[128 + tid], b2 = bm[256 + tid], b3 = bm[384 + tid];
    const uint32_t u = b0 | b1 | b2 | b3;
    const uint32_t cu = __popc(u);
    const uint32_t cb = __popc(b0) | (__popc(b1) << 8) | (__popc(b2) << 16) | ((uint32_t)__popc(b3) << 24);
    uint32_t iu = cu, ib = cb;                   // (each plane has <= 255 runs: its byte never carries)
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t yu = __shfl_up_sync(0xffffffffu, iu, o), yb = __shfl_up_sync(0xffffffffu, ib, o);
        if (lane >= o) { iu += yu; ib += yb; }
    }
    if (lane == 31) wt[warp] = make_uint2(iu, ib);
    __syncthreads();
    uint32_t eu = iu - cu, eb = ib - cb;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const uint2 t = wt[k];
        if (k < warp) { eu += t.x; eb += t.y; }
    }
    UP[tid] = make_uint2(u, eu - 1u);
    // the element of every segment starting in word tid
    for (uint32_t m = u; m; m &= m - 1u) {
        const int b = __ffs(m) - 1;
        const uint32_t le = (2u << b) - 1u;      // bits 0..b
        const uint32_t r0 = ((eb >> 0) & 0xFFu) + __popc(b0 & le) - 1u;
        const uint32_t r1 = ((eb >> 8) & 0xFFu) + __popc(b1 & le) - 1u;
        const uint32_t r2 = ((eb >> 16) & 0xFFu) + __popc(b2 & le) - 1u;
        const uint32_t r3 = (eb >> 24) + __popc(b3 & le) - 1u;
        uint32_t e = (uint32_t)val[r0] | ((uint32_t)val[256 + r1] << 8) | ((uint32_t)val[512 + r2] << 16) |
                     ((uint32_t)val[768 + r3] << 24);
        if (sw) e = swizzle(e);
        SV[eu + __popc(u & (le >> 1))] = e;
    }
    __syncthreads();
    const bool dense = jb.pitch == jb.w;
    const int bb = (tid & 7) << 2;               // a thread's groups start at one bit of their words
    const uint32_t le = (2u << bb) - 1u;
    auto group = [&](int i) {                    // elements [4 (tid + 128 i), + 4)
        const uint2 up = UP[(tid >> 3) + 16 * i];
        const uint32_t k0 = up.y + __popc(up.x & le);
        const uint32_t in = (up.x >> (bb + 1)) & 7u;             // segments starting inside the group
        const uint32_t v0 = SV[k0];
        uint4 v = make_uint4(v0, v0, v0, v0);
        if (in) {
            const uint32_t k1 = k0 + (in & 1u), k2 = k1 + ((in >> 1) & 1u), k3 = k2 + (in >> 2);
            v.y = SV[k1]; v.z = SV[k2]; v.w = SV[k3];
        }
        return v;
    };
    if (jb.vec && len == kChunk) {               // whole chunks: every group is one 16-byte store
        const uint32_t q = q0 + 4u * (uint32_t)tid;
        if (dense) {
            uint4* o = reinterpret_cast<uint4*>(dstp + q);
#pragma unroll
            for (int i = 0; i < kChunk / 4 / kDT; ++i) st_stream(o + kDT * i, group(i));
        } else {
#pragma unroll 2
            for (int i = 0; i < kChunk / 4 / kDT; ++i)
                st_stream(reinterpret_cast<uint4*>(dstp + elem_off(jb, q + 4u * kDT * i)), group(i));
        }
        return;
    }
    for (int i = 0; 4 * (tid + kDT * i) < len; ++i) {
        const uint4 v = group(i);
        const int g = tid + kDT * i;
        const uint32_t q = q0 + 4u * (uint32_t)g;
        if (jb.vec && 4 * g + 4 <= len) {
            st_stream(reinterpret_cast<uint4*>(dstp + (dense ? (size_t)q : elem_off(jb, q))), v);
        } else {
            const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (4 * g + j < len) dstp[elem_off(jb, q + (uint32_t)j)] = vv[j];
        }
    }
}

template <int N>
__global__ void __launch_bounds__(kDT, 12)
k_rle_decompress(const __grid_constant__ RleJobList<N> J, uint32_t* status)
{
    // the four decoded planes; a mode-0 chunk's stream (at most 8 * 2048 + 16
    // bytes) is staged here instead
    __shared__ __align__(16) uint8_t sbuf[4 * kChunk + 64];
    uint8_t (*planes)[kChunk] = reinterpret_cast<uint8_t (*)[kChunk]>(sbuf);
    __shared__ uint32_t s_tok[kTok0];                 // mode 0: listed tokens

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t unit = blockIdx.x;
    const RleJobDesc& jb = J.j[find_job(J, unit)];
    const uint8_t* src = reinterpret_cast<const uint8_t*>(jb.src);
    const uint64_t size = jb.capacity;
    const uint32_t nc = jb.n_chunks;
    const uint32_t c = unit - jb.first_unit;
    chain_wait();
    const rlec::ChunkEnds E = rlec::check_chunk(src, size, size, (uint32_t)jb.w, (uint32_t)jb.h, nc, c, true);
    if (E.bad) {
        if (tid == 0) set_status(status, EC_ERR_CORRUPT);
        return;
    }
    if (nc == 0) return;

    const uint32_t n = (uint32_t)jb.w * (uint32_t)jb.h;
    const uint32_t q0 = c * (uint32_t)kChunk;
    const int len = (int)min((uint32_t)kChunk, n - q0);
    if (E.mode == 0) {
        decode_mode0(jb, src + 32 + 4ull * nc, (uint32_t)E.beg(5), (uint32_t)E.end(5), q0, len, sbuf, s_tok, status);
        return;
    }
    const uint8_t* payload = src + 32 + 16ull * nc;
    uint32_t* dstp = reinterpret_cast<uint32_t*>(jb.dst);
    const bool sw = E.mode == 2;
    const int beg = E.beg(warp), end = E.end(warp);

    // Runs first: warp p walks plane p's tokens, marking where each run starts
    // (every repeat token, every literal byte) and keeping its byte.  A token of
    // k bytes starts at least k / 2 runs, so a stream of more than 2 kRunCap
    // bytes has too many for this path, and its walk is not begun.
    if (!E.any_longer(2u * (uint32_t)kRunCap)) {
        uint32_t* bm = reinterpret_cast<uint32_t*>(sbuf);          // [4][128] run starts per plane
        uint8_t* val = sbuf + kRunArea;                             // [4][256] run bytes per plane
        reinterpret_cast<uint4*>(bm + 128 * warp)[lane] = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
        int nr = 0;
        const int r = rlec::decode_plane_runs(rlec::GlobalBytes{payload}, beg, end, len, bm + 128 * warp,
                                              val + 256 * warp, kRunCap, &nr, lane);
        if (!__syncthreads_or(r)) {
            fill_segments(jb, q0, len, sw, bm, val, sbuf, dstp);
            return;
        }
        if (__syncthreads_or(r == 1)) {
            if (tid == 0) set_status(status, EC_ERR_CORRUPT);
            return;
        }
    }

    // many runs: warp p decodes byte plane p into shared memory
    if (__syncthreads_or(rlec::decode_plane_dense(rlec::GlobalWords{payload}, beg, end, len, planes[warp], lane))) {
        if (tid == 0) set_status(status, EC_ERR_CORRUPT);
        return;
    }

    // transpose planes back into elements, 16 per thread; the swizzle is undone
    // on the plane words, four elements at a time
    const int whole = jb.vec ? len & ~3 : 0;                  // elements written by 16-byte groups
    const bool dense = jb.pitch == jb.w;
    for (int g16 = tid; 16 * g16 < whole; g16 += kDT) {
        const uint4 A = *reinterpret_cast<const uint4*>(&planes[0][16 * g16]);
        const uint4 B = *reinterpret_cast<const uint4*>(&planes[1][16 * g16]);
        const uint4 C = *reinterpret_cast<const uint4*>(&planes[2][16 * g16]);
        const uint4 D = *reinterpret_cast<const uint4*>(&planes[3][16 * g16]);
        uint32_t a4[4] = {A.x, A.y, A.z, A.w}, b4[4] = {B.x, B.y, B.z, B.w};
        uint32_t c4[4] = {C.x, C.y, C.z, C.w}, d4[4] = {D.x, D.y, D.z, D.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int g = 4 * g16 + k;
            if (4 * g >= whole) break;
            if (sw) rlec::swizzle_planes(a4[k], b4[k], c4[k], d4[k]);
            const uint4 v = transpose4(a4[k], b4[k], c4[k], d4[k]);
            const uint32_t q = q0 + 4u * g;
            st_stream(reinterpret_cast<uint4*>(dstp + (dense ? (size_t)q : elem_off(jb, q))), v);
        }
    }
    for (int t = whole + tid; t < len; t += kDT) {
        uint32_t v = (uint32_t)planes[0][t] | ((uint32_t)planes[1][t] << 8) |
                     ((uint32_t)planes[2][t] << 16) | ((uint32_t)planes[3][t] << 24);
        if (sw) v = swizzle(v);
        dstp[elem_off(jb, q0 + t)] = v;
    }
}

template <int N>
RleJobList<N> make_jobs(const RleJobDesc* jobs, int n, uint32_t total)
{
    RleJobList<N> J;
    J.n = n;
    J.total_units = total;
    J.pad[0] = J.pad[1] = 0;
    for (int i = 0; i < n; ++i) J.j[i] = jobs[i];
    return J;
}

}  // namespace

namespace {

// Mode 0's persistent grid: as many coding CTAs as fit on the device at once.
template <int N>
cudaError_t compress_grid(int* grid)
{
    constexpr int kMaxDev = 64;
    static std::atomic<int> cache[kMaxDev];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < kMaxDev && (*grid = cache[dev].load(std::memory_order_relaxed)) > 0) return cudaSuccess;
    e = cudaFuncSetAttribute(k_rle_compress0<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCompressSmem);
    if (e != cudaSuccess) return e;
    // the persistent grid is sized for the largest shared-memory carveout:
    // ask for it, so that every CTA of the grid is resident at once
    e = cudaFuncSetAttribute(k_rle_compress0<N>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             (int)cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    int per_sm = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rle_compress0<N>, 32 * kWPB, kCompressSmem);
    if (e != cudaSuccess) return e;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    *grid = std::max(1, per_sm) * sms;
    if (dev < kMaxDev) cache[dev].store(*grid, std::memory_order_relaxed);
    return cudaSuccess;
}

// Mode 0: code (persistent warps), size the dense chunks, scan the sizes (a CTA
// per job), place (a quarter-warp per chunk), write the listed chunks.
template <int N>
cudaError_t compress0(const RleJobDesc* jobs, int n, uint32_t total_units, const RleScratch& W, int rgrid,
                      uint32_t* status, cudaStream_t s)
{
    cudaError_t e;
    const RleJobList<N> J = make_jobs<N>(jobs, n, total_units);
    int grid = 0;
    if ((e = compress_grid<N>(&grid)) != cudaSuccess) return e;
    grid = (int)std::min<uint32_t>((uint32_t)grid, (total_units + kWPB - 1) / kWPB);
    // pool space is taken in slabs of up to 16 KB per warp where the pool
    // has room for eight slabs per warp of the grid (their unused tails are
    // then at most an eighth of it), else chunk by chunk
    const uint32_t pb = (uint32_t)std::min<size_t>(W.pool_bytes, 0xFFFFFFF0u);
    uint32_t slab = std::min<uint32_t>(pb / (8u * (uint32_t)grid * kWPB), 16384u) & ~255u;
    if (slab < 4u * kStagePlane) slab = 0u;
    e = launch_chained(k_rle_compress0<N>, grid, 32 * kWPB, kCompressSmem, s, J, W.rec, W.recode, W.pool, pb, slab,
                       W.counters, status);
    if (e != cudaSuccess) return e;
    const uint32_t* count = W.counters + 1;
    if ((e = launch_chained(k_rle0_recode<N, false>, rgrid, kT, 0, s, J, W.rec, W.recode, count)) != cudaSuccess) return e;
    if ((e = launch_chained(k_rle_scan<N>, n, 1024, 0, s, J, W.rec)) != cudaSuccess) return e;
    constexpr uint32_t per = 128 / kPlaceLanes;
    e = launch_chained(k_rle_place<N>, (total_units + per - 1) / per, 128, 0, s, J, W.rec, W.pool);
    if (e != cudaSuccess) return e;
    return launch_chained(k_rle0_recode<N, true>, rgrid, kT, 0, s, J, W.rec, W.recode, count);
}

// The four-plane modes: code (a CTA per chunk), code the dense chunks, place.
template <int N>
cudaError_t compress_n(const RleJobDesc* jobs, int n, uint32_t total_units, const RleScratch& W, int rgrid,
                       uint32_t* status, cudaStream_t s)
{
    const RleJobList<N> J = make_jobs<N>(jobs, n, total_units);
    cudaError_t e = launch_chained(k_rle_code<N>, total_units, kCT, 0, s, J, W, status);
    if (e != cudaSuccess) return e;
    if ((e = launch_chained(k_rle_recode<N, false>, rgrid, kRT, 0, s, J, W, (uint32_t)rgrid)) != cudaSuccess) return e;
    return launch_chained(k_rle_recode<N, true>, (uint32_t)rgrid + (total_units + kGroup - 1) / kGroup, kRT, 0, s, J, W,
                          (uint32_t)rgrid);
}

// Offsets of the scratch's parts after the counters; the pool starts at a 128-byte line.
constexpr size_t scratch_groups(uint32_t units) { return 16 + (sizeof(ChunkRec) + 8) * (size_t)units; }
constexpr size_t scratch_pool(uint32_t units)
{
    return (scratch_groups(units) + 4 * (((size_t)units + kGroup - 1) / kGroup) + 127) & ~(size_t)127;
}

}  // namespace

size_t rle_compress_scratch_bytes(uint32_t units, size_t pool_bytes)
{
    return scratch_pool(std::max<uint32_t>(units, 1)) + pool_bytes;
}

cudaError_t launch_rle_compress(const RleJobDesc* jobs, int n, uint32_t total_units,
                                void* scratch, size_t scratch_bytes, uint32_t* status, cudaStream_t s)
{
    if (n <= 0 || total_units == 0) return cudaSuccess;
    if (scratch_bytes < rle_compress_scratch_bytes(total_units, 0)) return cudaErrorInvalidValue;
    char* base = reinterpret_cast<char*>(scratch);
    RleScratch W;
    W.counters = reinterpret_cast<uint32_t*>(base);
    W.rec = reinterpret_cast<ChunkRec*>(base + 16);
    W.recode = reinterpret_cast<uint32_t*>(W.rec + total_units);
    W.again = W.recode + total_units;
    W.groups = reinterpret_cast<uint32_t*>(base + scratch_groups(total_units));
    W.pool = reinterpret_cast<uint8_t*>(base + scratch_pool(total_units));
    W.pool_bytes = scratch_bytes - scratch_pool(total_units);
    W.slots = pool_slots(total_units, W.pool_bytes);
    int sms = 0, dev = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const int rgrid = std::max(1, sms) * 4;
    // (a memset between the kernels would end the chain)
    const uint32_t ng = jobs[0].mode == 0 ? 0u : (total_units + kGroup - 1) / kGroup;
    e = launch_chained(k_rle_begin, std::max(1u, (ng + 255) / 256), 256, 0, s, reinterpret_cast<uint4*>(scratch), W.groups, ng);
    if (e != cudaSuccess) return e;
    if (jobs[0].mode == 0) {                      // (one launch codes one mode family)
        if (n <= 8) return compress0<8>(jobs, n, total_units, W, rgrid, status, s);
        if (n <= 64) return compress0<64>(jobs, n, total_units, W, rgrid, status, s);
        return compress0<kRleJobsPerLaunch>(jobs, n, total_units, W, rgrid, status, s);
    }
    if (n <= 8) return compress_n<8>(jobs, n, total_units, W, rgrid, status, s);
    if (n <= 64) return compress_n<64>(jobs, n, total_units, W, rgrid, status, s);
    return compress_n<kRleJobsPerLaunch>(jobs, n, total_units, W, rgrid, status, s);
}

cudaError_t launch_selftest_wait(uint32_t* status, cudaStream_t s)
{
    k_selftest_wait<<<1, 32, 0, s>>>(status);
    return cudaGetLastError();
}

cudaError_t launch_rle_decompress(const RleJobDesc* jobs, int n, uint32_t total_units,
                                  uint32_t* status, cudaStream_t s)
{
    if (n <= 0 || total_units == 0) return cudaSuccess;
    if (n <= 8) return launch_chained(k_rle_decompress<8>, total_units, kDT, 0, s, make_jobs<8>(jobs, n, total_units), status);
    if (n <= 64) return launch_chained(k_rle_decompress<64>, total_units, kDT, 0, s, make_jobs<64>(jobs, n, total_units), status);
    return launch_chained(k_rle_decompress<kRleJobsPerLaunch>, total_units, kDT, 0, s,
                          make_jobs<kRleJobsPerLaunch>(jobs, n, total_units), status);
}

}  // namespace ec
