// k_fused.cu -- fused decode-and-composite for the stages of multi-stage
// compositing schedules (thesis 5.2.2 binary swap, 5.2.3 streaming
// compositing): a resource receives RLE-coded pieces (thesis 5.5.1) of another
// resource's partial frame and depth-merges them with its own image
// (thesis 5.2.1) without writing the decoded pieces to memory first.
//
// One CTA of eight warps per work unit.  A decode unit is one 4096-element
// chunk of a received piece: warps 0-3 walk the colour stream's four byte
// planes and warps 4-7 the depth stream's (the decoder of the RLE kernels,
// including its validation).  When every plane has at most 255 runs they
// record the runs only: between the union of the eight planes' run starts
// colour and depth are constant, so each segment's pair is assembled once and
// a pixel's pair is found by its rank among the run starts.  Otherwise they
// decode the planes into shared memory, and pixels are transposed back from
// them with funnel shifts.  The threads take the chunk's pixels four at a
// time (quads aligned to the output's 16-byte boundaries), read the local
// input at the same frame pixels and write the merge.  A fill unit,
// a band of rows that no piece reaches, writes the local input (or the
// background) there.
//
// The merge of a front and a back partial: the front is first merged with the
// cleared background (depth not below 1.0, or NaN, gives the background), then
// the back replaces it where its depth is strictly smaller.  A partial that is
// already a composite is unchanged by the first step, a raw source image is
// made one, and ties stay with the front, the lower source indices.
#include "ec_internal.cuh"
#include "rle_codec.cuh"

namespace ec {
namespace {

constexpr int kFT = 256;
constexpr int kChunk = rlec::kChunk;
constexpr uint32_t kBgDepth = 0x3F800000u;   // 1.0f
constexpr int kStageWords = 1024;             // staged stream bytes per stream: 4 KB
// The run path's tables: bitmaps, run bytes, their union with its prefix, scan
// scratch, segments (at most 8 * 255).
constexpr int kRunArea = 4096 + 2048 + 512 + 512 + 128 + 8 * 2040;
static_assert(kRunArea % 16 == 0 && kRunArea + 2 * 4 * kStageWords <= 8 * kChunk, "run path in the planes' space");

__device__ __forceinline__ bool below_one(uint32_t d) { return __uint_as_float(d) < 1.0f; }
__device__ __forceinline__ bool less(uint32_t a, uint32_t b) { return __uint_as_float(a) < __uint_as_float(b); }

// A front pixel over the cleared background.
__device__ __forceinline__ void clear_far(uint32_t& c, uint32_t& d)
{
    if (!below_one(d)) { c = 0u; d = kBgDepth; }
}

// A cleared front pixel (fc, fd) and a back one (bc, bd), as raw bits.
__device__ __forceinline__ void over(uint32_t fc, uint32_t fd, uint32_t bc, uint32_t bd, uint32_t& oc, uint32_t& od)
{
    const bool b = less(bd, fd);
    oc = b ? bc : fc;
    od = b ? bd : fd;
}

// Merge one pixel.
__device__ __forceinline__ void merge(uint32_t fc, uint32_t fd, uint32_t bc, uint32_t bd, uint32_t& oc, uint32_t& od)
{
    clear_far(fc, fd);
    over(fc, fd, bc, bd, oc, od);
}

// Pixels are handled in quads: four horizontally adjacent pixels whose first
// one sits at a 16-byte boundary of the output buffer (x - ox a multiple of
// 4), so that a quad inside the unit is one 16-byte store.  A unit covers
// `nrows` rows of its rectangle from row `ra`; a decode unit only the elements
// [q0, q0 + len) of its chunk (element q = row * w + column).
struct Quad {
    int r, x, lo, hi;             // row after the unit's first, column of pixel 0, pixels [lo, hi) inside the unit
    uint32_t lc[4], ld[4];        // the receiver's own image there
};

// What the quads of a unit share.  Columns are the rectangle's, rows count from
// the unit's first.
struct Grid {
    const uint32_t *lc, *ld;      // the local image at row 0, column 0
    uint32_t *oc, *od;            // the output there
    int lpitch, opitch;
    int rx0, rx1, ry0, ry1;       // the local image's ROI
    int w, e0, e1;                // columns; element of row 0, column 0 in the chunk; the chunk's length
    bool lvec, ovec, front;
};

template <bool CODED>
__device__ __forceinline__ bool bounds(const Grid& g, Quad& Q)
{
    Q.lo = max(0, -Q.x);
    Q.hi = min(4, g.w - Q.x);
    if (CODED) {
        const int i0 = g.e0 + Q.r * g.w + Q.x;
        Q.lo = max(Q.lo, -i0);
        Q.hi = min(Q.hi, g.e1 - i0);
    }
    return Q.lo < Q.hi;
}

// The receiver's own image at the quad (background outside its ROI).
__device__ __forceinline__ void load_local(const Grid& g, Quad& Q)
{
    const bool in_y = Q.r >= g.ry0 && Q.r < g.ry1;
    const int64_t le = (int64_t)Q.r * g.lpitch + Q.x;
    if (in_y && Q.x >= g.rx0 && Q.x + 3 < g.rx1 && g.lvec) {
        const uint4 c = __ldcs(reinterpret_cast<const uint4*>(g.lc + le));
        const uint4 d = __ldcs(reinterpret_cast<const uint4*>(g.ld + le));
        Q.lc[0] = c.x; Q.lc[1] = c.y; Q.lc[2] = c.z; Q.lc[3] = c.w;
        Q.ld[0] = d.x; Q.ld[1] = d.y; Q.ld[2] = d.z; Q.ld[3] = d.w;
        return;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        Q.lc[k] = 0u;
        Q.ld[k] = kBgDepth;
        if (k >= Q.lo && k < Q.hi && in_y && Q.x + k >= g.rx0 && Q.x + k < g.rx1) {
            Q.lc[k] = __ldcs(g.lc + le + k);
            Q.ld[k] = __ldcs(g.ld + le + k);
        }
    }
}

// Run path of a decode unit: the chunk's elements are constant between the
// union of its eight planes' run starts.  U: that union (128 words), PU: the
// segments starting before each word, S: each segment's colour and depth.
struct Segs {
    const uint32_t* U;
    const uint32_t* PU;
    const uint2* S;
};

template <bool CODED>
__device__ __forceinline__ void finish(const Grid& g, const Quad& Q, const uint8_t (*planes)[kChunk], bool csw, bool dsw,
                                       const Segs* G = nullptr)
{
    uint32_t oc[4], od[4];
    if (CODED && G) {
        // the segment of the quad's first element in the chunk, and the starts
        // after it (bit k: pixel k starts one); most quads lie inside one segment
        const int i0 = g.e0 + Q.r * g.w + Q.x, a = max(i0, 0);
        const uint32_t u0 = G->U[a >> 5], u1 = G->U[min((a >> 5) + 1, kChunk / 32 - 1)];
        const uint2* s0 = G->S + (G->PU[a >> 5] + __popc(u0 & ((2u << (a & 31)) - 1u)) - 1u);
        const uint32_t nb = (__funnelshift_r(u0, u1, a & 31) & 0xEu) << (a - i0);
        uint2 v[4];
        v[0] = v[1] = v[2] = v[3] = *s0;
        if (nb & 0xEu) {
            v[1] = s0[__popc(nb & 0x2u)];
            v[2] = s0[__popc(nb & 0x6u)];
            v[3] = s0[__popc(nb & 0xEu)];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (g.front) over(v[k].x, v[k].y, Q.lc[k], Q.ld[k], oc[k], od[k]);   // (cleared when the segment was made)
            else merge(Q.lc[k], Q.ld[k], v[k].x, v[k].y, oc[k], od[k]);
        }
    } else if (CODED) {
        // bytes of elements i0 .. i0 + 3 of every plane: two words and a funnel shift
        const int i0 = g.e0 + Q.r * g.w + Q.x;
        const int wi = i0 >> 2, sh = 8 * (i0 & 3);
        const int w0 = max(wi, 0), w1 = min(wi + 1, kChunk / 4 - 1);
        uint32_t pb[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) {
            const uint32_t* pl = reinterpret_cast<const uint32_t*>(planes[p]);
            pb[p] = __funnelshift_r(pl[w0], pl[w1], sh);
        }
        const uint4 C = rlec::transpose4(pb[0], pb[1], pb[2], pb[3]);
        const uint4 D = rlec::transpose4(pb[4], pb[5], pb[6], pb[7]);
        uint32_t ic[4] = {C.x, C.y, C.z, C.w}, id[4] = {D.x, D.y, D.z, D.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (csw) ic[k] = rlec::swizzle(ic[k]);
            if (dsw) id[k] = rlec::swizzle(id[k]);
            if (g.front) merge(ic[k], id[k], Q.lc[k], Q.ld[k], oc[k], od[k]);
            else merge(Q.lc[k], Q.ld[k], ic[k], id[k], oc[k], od[k]);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool keep = below_one(Q.ld[k]);
            oc[k] = keep ? Q.lc[k] : 0u;
            od[k] = keep ? Q.ld[k] : kBgDepth;
        }
    }
    const int64_t oe = (int64_t)Q.r * g.opitch + Q.x;
    if (Q.lo == 0 && Q.hi == 4 && g.ovec) {
        st_stream(reinterpret_cast<uint4*>(g.oc + oe), make_uint4(oc[0], oc[1], oc[2], oc[3]));
        st_stream(reinterpret_cast<uint4*>(g.od + oe), make_uint4(od[0], od[1], od[2], od[3]));
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k >= Q.lo && k < Q.hi) {
                g.oc[oe + k] = oc[k];
                g.od[oe + k] = od[k];
            }
    }
}

// The unit's quads in row order, from the one of its first element to the one of
// its last: thread t takes the t-th of every kFT, two at a time, so that both
// local loads are in flight together.  The step from one quad to the next is the
// same for all of a thread's quads but for a wrap into the next row.
template <bool CODED>
__device__ __forceinline__ void compose(const FusedStage& S, const FusedUnit& u, int ra, int nrows,
                                        int q0, int len, const uint8_t (*planes)[kChunk], bool csw, bool dsw,
                                        const Segs* G = nullptr)
{
    const int head = (u.x - S.ox) & 3;                        // pixels of a row's first quad before the unit
    const int nq = (u.w + head + 3) >> 2;                     // quads of a row
    Grid g;
    const int64_t lo = (int64_t)(u.y + ra - S.ly) * S.lpitch + (u.x - S.lx);
    const int64_t oo = (int64_t)(u.y + ra - S.oy) * S.opitch + (u.x - S.ox);
    g.lc = S.lc + lo;
    g.ld = reinterpret_cast<const uint32_t*>(S.ld) + lo;
    g.oc = S.oc + oo;
    g.od = reinterpret_cast<uint32_t*>(S.od) + oo;
    g.lpitch = S.lpitch;
    g.opitch = S.opitch;
    g.rx0 = S.r0x - u.x;
    g.rx1 = S.r1x - u.x;
    g.ry0 = S.r0y - u.y - ra;
    g.ry1 = S.r1y - u.y - ra;
    g.w = u.w;
    g.e0 = CODED ? ra * u.w - q0 : 0;
    g.e1 = len;
    g.lvec = S.lvec && ((u.x - head - S.lx) & 3) == 0;
    g.ovec = S.ovec;
    g.front = S.front;
    const int s0 = CODED ? (head - g.e0) >> 2 : 0;
    const int s1 = CODED ? (nrows - 1) * nq + ((head + len - 1 - g.e0 - (nrows - 1) * u.w) >> 2) + 1 : nrows * nq;
    const int dr = kFT / nq, dx = 4 * (kFT - dr * nq);
    const int s = s0 + (int)threadIdx.x, r = s / nq;
    Quad A, B;
    B.r = r;
    B.x = 4 * (s - r * nq) - head;
    const int end = 4 * nq - head;
    auto step = [&](const Quad& from, Quad& to) {
        to.r = from.r + dr;
        to.x = from.x + dx;
        if (to.x >= end) { to.x -= 4 * nq; ++to.r; }
    };
    for (int left = s1 - s; left > 0; left -= 2 * kFT) {
        A.r = B.r;
        A.x = B.x;
        step(A, B);
        const bool a = bounds<CODED>(g, A), b = left > kFT && bounds<CODED>(g, B);
        if (a) load_local(g, A);
        if (b) load_local(g, B);
        if (a) finish<CODED>(g, A, planes, csw, dsw, G);
        if (b) finish<CODED>(g, B, planes, csw, dsw, G);
        step(B, B);
    }
}

// Bound by instruction issue, and in small launches by the chain from a unit's
// header to its last pixel.  The four fused launches of a binary swap of 16
// 1920x1080 sources (about 1100 x 1000 pixels each, 30 % covered) take 104 us;
// with rows walked quad by quad with a division each, every warp checking the
// headers and 41 KB of shared memory they took 123 us.  Four CTAs per SM: six
// (40 registers) took 114 us, five (48) 105 us.
__global__ void __launch_bounds__(kFT, 4)
k_fused_depth(const FusedStage* __restrict__ stages, const FusedUnit* __restrict__ units, uint32_t* status)
{
    // the decoded planes; before them, the run path's tables and staged streams
    __shared__ __align__(16) uint8_t planes[8][kChunk];
    uint32_t (*staged)[kStageWords] = reinterpret_cast<uint32_t (*)[kStageWords]>(&planes[0][0] + kRunArea);
    __shared__ uint32_t s_beg[2][5];
    __shared__ int s_mode[2];
    __shared__ int s_fail, s_over;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // (the plan's own arrays: written when it was made)
    const FusedUnit u = units[blockIdx.x];
    const FusedStage S = stages[u.stage];
    chain_wait();

    if (u.cs == nullptr) {                    // fill: rows [chunk, chunk + nrows) of the rectangle
        compose<false>(S, u, (int)u.chunk, u.nrows, 0, 0, planes, false, false);
        return;
    }
    const uint32_t n = (uint32_t)u.w * (uint32_t)u.h;
    const uint32_t q0 = u.chunk * (uint32_t)kChunk;
    const int len = (int)min((uint32_t)kChunk, n - q0);
    const uint32_t nc = (n + kChunk - 1) / kChunk;
    const int ra = (int)(q0 / (uint32_t)u.w), rb = (int)((q0 + (uint32_t)len - 1u) / (uint32_t)u.w);
    // header bytes are read within the streams' capacity, in parallel with
    // their sizes; the validation then uses the sizes
    const uint64_t csz = *u.csize, dsz = *u.dsize;
    // the run bitmaps (aliased with the planes) start empty
    uint32_t* bm = reinterpret_cast<uint32_t*>(&planes[0][0]);       // [8][128] run starts per plane
    reinterpret_cast<uint4*>(bm)[tid] = make_uint4(0u, 0u, 0u, 0u);
    // a warp checks the colour stream, another the depth stream
    bool bad = false;
    if ((warp & 3) == 0) {
        const rlec::ChunkEnds E = warp == 0
            ? rlec::check_chunk(u.cs, u.cap, csz, (uint32_t)u.w, (uint32_t)u.h, nc, u.chunk, false)
            : rlec::check_chunk(u.ds, u.cap, dsz, (uint32_t)u.w, (uint32_t)u.h, nc, u.chunk, false);
        if (lane >= 8 && lane < 13) s_beg[warp >> 2][lane - 8] = E.v;
        if (lane == 0) s_mode[warp >> 2] = E.mode;
        bad = E.bad;
    }
    if (tid == 0) { s_fail = 0; s_over = 0; }
    if (__syncthreads_or(bad)) {
        if (tid == 0) set_status(status, EC_ERR_CORRUPT);
        return;
    }
    // stage each stream's bytes of this chunk (its four planes are contiguous)
    // in shared memory when they fit, so that the decoder's dependent steps wait
    // on shared memory instead of global memory
    const uint8_t* cpay = u.cs + 32 + 16ull * nc;
    const uint8_t* dpay = u.ds + 32 + 16ull * nc;
    const int cw0 = (int)(s_beg[0][0] >> 2), cnw = (int)((s_beg[0][4] + 3u) >> 2) - cw0;
    const int dw0 = (int)(s_beg[1][0] >> 2), dnw = (int)((s_beg[1][4] + 3u) >> 2) - dw0;
    {
        const int k = warp >> 2, w0 = k ? dw0 : cw0, nw = k ? dnw : cnw;
        const uint32_t* from = reinterpret_cast<const uint32_t*>(k ? dpay : cpay) + w0;
        if (nw <= kStageWords)
            for (int i = tid & 127; i < nw; i += 128) staged[k][i] = __ldg(from + i);
    }
    __syncthreads();
    // run path: warp k*4+p walks stream k's plane p, recording its runs
    uint8_t* const base8 = &planes[0][0];
    {
        const int k = warp >> 2, p = warp & 3;
        const int b = (int)s_beg[k][p], e = (int)s_beg[k][p + 1];
        const int w0 = k ? dw0 : cw0, nw = k ? dnw : cnw;
        uint8_t* val = base8 + 4096 + 256 * warp;                   // [8][256] run bytes
        int nr = 0;
        const int r = nw <= kStageWords
            ? rlec::decode_plane_runs(rlec::SharedBytes{reinterpret_cast<const uint8_t*>(staged[k]), 4 * w0},
                                      b, e, len, bm + 128 * warp, val, 255, &nr, lane)
            : rlec::decode_plane_runs(rlec::GlobalBytes{k ? dpay : cpay}, b, e, len, bm + 128 * warp, val, 255,
                                      &nr, lane);
        if (r == 1 && lane == 0) s_fail = 1;
        if (r == 2 && lane == 0) s_over = 1;
    }
    __syncthreads();
    if (s_fail) {
        if (tid == 0) set_status(status, EC_ERR_CORRUPT);
        return;
    }
    if (!s_over) {
        uint32_t* U = reinterpret_cast<uint32_t*>(base8 + 6144);
        uint32_t* PU = U + 128;
        uint32_t* wt = PU + 128;                                     // scan scratch
        uint2* SS = reinterpret_cast<uint2*>(base8 + 7296);          // <= 8 * 255 segments
        const uint8_t* val = base8 + 4096;
        const bool csw = s_mode[0] == 2, dsw = s_mode[1] == 2;
        uint32_t un = 0u, eu = 0u, ec = 0u, ed = 0u, wb[8];
        if (tid < 128) {
#pragma unroll
            for (int q = 0; q < 8; ++q) { wb[q] = bm[128 * q + tid]; un |= wb[q]; }
            const uint32_t cu = __popc(un);
            const uint32_t cc = __popc(wb[0]) | (__popc(wb[1]) << 8) | (__popc(wb[2]) << 16) | ((uint32_t)__popc(wb[3]) << 24);
            const uint32_t cd = __popc(wb[4]) | (__popc(wb[5]) << 8) | (__popc(wb[6]) << 16) | ((uint32_t)__popc(wb[7]) << 24);
            uint32_t iu = cu, ic = cc, id = cd;      // (a plane has <= 255 runs: its byte never carries)
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t yu = __shfl_up_sync(0xffffffffu, iu, o), yc = __shfl_up_sync(0xffffffffu, ic, o);
                const uint32_t yd = __shfl_up_sync(0xffffffffu, id, o);
                if (lane >= o) { iu += yu; ic += yc; id += yd; }
            }
            if (lane == 31) { wt[3 * warp] = iu; wt[3 * warp + 1] = ic; wt[3 * warp + 2] = id; }
            eu = iu - cu; ec = ic - cc; ed = id - cd;
        }
        __syncthreads();
        if (tid < 128) {
            for (int w = 0; w < warp; ++w) { eu += wt[3 * w]; ec += wt[3 * w + 1]; ed += wt[3 * w + 2]; }
            U[tid] = un;
            PU[tid] = eu;
            for (uint32_t m = un; m; m &= m - 1u) {
                const int bb = __ffs(m) - 1;
                const uint32_t le = (2u << bb) - 1u;
                uint32_t c = 0u, d = 0u;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t rc = ((ec >> (8 * q)) & 0xFFu) + __popc(wb[q] & le) - 1u;
                    const uint32_t rd = ((ed >> (8 * q)) & 0xFFu) + __popc(wb[4 + q] & le) - 1u;
                    c |= (uint32_t)val[256 * q + rc] << (8 * q);
                    d |= (uint32_t)val[256 * (4 + q) + rd] << (8 * q);
                }
                const uint32_t sidx = eu + __popc(un & (le >> 1));
                if (csw) c = rlec::swizzle(c);
                if (dsw) d = rlec::swizzle(d);
                if (S.front) clear_far(c, d);
                SS[sidx] = make_uint2(c, d);
            }
        }
        __syncthreads();
        const Segs G{U, PU, SS};
        compose<true>(S, u, ra, rb - ra + 1, (int)q0, len, planes, false, false, &G);
        return;
    }
    // many runs: decode the planes into shared memory
    {
        const int k = warp >> 2, p = warp & 3;
        const int bad = rlec::decode_plane_dense(rlec::GlobalWords{k ? dpay : cpay}, (int)s_beg[k][p],
                                                 (int)s_beg[k][p + 1], len, planes[warp], lane);
        if (bad && lane == 0) s_fail = 1;
    }
    __syncthreads();
    if (s_fail) {
        if (tid == 0) set_status(status, EC_ERR_CORRUPT);
        return;
    }
    compose<true>(S, u, ra, rb - ra + 1, (int)q0, len, planes, s_mode[0] == 2, s_mode[1] == 2);
}

}  // namespace

cudaError_t launch_fused_depth(const FusedStage* stages, const FusedUnit* units, int n_units,
                               uint32_t* status, cudaStream_t s)
{
    if (n_units <= 0) return cudaSuccess;
    return launch_chained(k_fused_depth, n_units, kFT, 0, s, stages, units, status);
}

}  // namespace ec
