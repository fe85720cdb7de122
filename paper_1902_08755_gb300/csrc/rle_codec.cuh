// rle_codec.cuh -- device pieces of the RLE container (thesis 5.5.1) shared by
// the decoder kernel and the fused decode-and-composite kernel: the swizzle,
// byte transposes, header and end-table validation, and the warp-wide decoder
// of one byte-plane stream.
#pragma once

#include "ec_internal.cuh"

namespace ec {
namespace rlec {

constexpr int kChunk = EC_RLE_CHUNK;                 // 4096 elements
constexpr uint32_t kMagic = 0x31524345u;             // "ECR1"

// Bit-swizzle: byte k of the result gathers bit pair (7-2k, 6-2k) of the four
// components, component 0 (R) in the top pair.  This is a transpose of the 4x4
// matrix of 2-bit cells, done as two delta swaps; it is its own inverse.
__device__ __forceinline__ uint32_t swizzle(uint32_t x)
{
    uint32_t t = ((x >> 20) ^ x) & 0x00000F0Fu;
    x ^= t ^ (t << 20);
    t = ((x >> 10) ^ x) & 0x00330033u;
    x ^= t ^ (t << 10);
    return x;
}

// The swizzle of the four elements whose bytes lie in four plane words (word k
// = byte k of each): the same transpose of 2-bit cells, exchanged between the
// words, for four elements at once.
__device__ __forceinline__ void swap_cells(uint32_t& hi, uint32_t& lo, int s, uint32_t m)
{
    const uint32_t t = (hi ^ (lo >> s)) & m;
    hi ^= t;
    lo ^= t << s;
}

__device__ __forceinline__ void swizzle_planes(uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d)
{
    swap_cells(a, c, 4, 0x0F0F0F0Fu);
    swap_cells(b, d, 4, 0x0F0F0F0Fu);
    swap_cells(a, b, 2, 0x33333333u);
    swap_cells(c, d, 2, 0x33333333u);
}

// 4x4 byte transpose: word b of the result holds byte b of e0..e3 (e0 lowest).
__device__ __forceinline__ uint4 transpose4(uint32_t e0, uint32_t e1, uint32_t e2, uint32_t e3)
{
    const uint32_t lo01 = __byte_perm(e0, e1, 0x5140), lo23 = __byte_perm(e2, e3, 0x5140);
    const uint32_t hi01 = __byte_perm(e0, e1, 0x7362), hi23 = __byte_perm(e2, e3, 0x7362);
    return make_uint4(__byte_perm(lo01, lo23, 0x5410), __byte_perm(lo01, lo23, 0x7632),
                      __byte_perm(hi01, hi23, 0x5410), __byte_perm(hi01, hi23, 0x7632));
}

// What a warp learns about chunk c of a stream: its header and the chunk's
// end-table entries, validated.  Lane 8 + p holds the start of plane p's stream
// inside the payload and lane 9 + p its end (four-plane modes); lanes 13 and 14
// those of a one-plane stream (mode 0).
struct ChunkEnds {
    uint32_t v;                                       // this lane's word
    int mode;
    bool bad;                                         // malformed (the same on every lane)
    __device__ __forceinline__ int beg(int p) const { return (int)__shfl_sync(0xffffffffu, v, 8 + p); }
    __device__ __forceinline__ int end(int p) const { return (int)__shfl_sync(0xffffffffu, v, 9 + p); }
    // whether one of the four planes' streams has more than `most` bytes
    __device__ __forceinline__ bool any_longer(uint32_t most) const
    {
        const uint32_t up = __shfl_up_sync(0xffffffffu, v, 1);
        const int lane = threadIdx.x & 31;
        return __any_sync(0xffffffffu, lane >= 9 && lane < 13 && v - up > most);
    }
};

// Validate the header fields against the expected w x h and nc chunks, and
// chunk c's stream ends against the payload size and the all-literal bound.
// Mode 0 is accepted only with allow0.  One word per lane: the header (lanes
// 0..7), entries 4c-1 .. 4c+3 of a four-plane table (8..12), entries c-1 and c
// of a one-plane table (13, 14); entry -1 is 0, and words past `have` bytes
// read as 0.  Nothing past `have` is read; `size` (<= have) is the stream's
// size.  src is 4-byte aligned.  Every warp of a CTA checks for itself: the
// words come in one round trip, and no warp waits for another.
__device__ __forceinline__ ChunkEnds check_chunk(const uint8_t* src, uint64_t have, uint64_t size, uint32_t w,
                                                 uint32_t hgt, uint32_t nc, uint32_t c, bool allow0)
{
    const int lane = threadIdx.x & 31;
    const uint32_t* s32 = reinterpret_cast<const uint32_t*>(src);
    uint64_t at = (uint64_t)lane, need = 32u;         // word index, bytes that must be there
    bool rd = lane < 15;
    if (lane >= 13) { at = 8ull + c + (uint64_t)lane - 14u; need = 32ull + 4ull * nc; rd = rd && nc > 0 && !(c == 0 && lane == 13); }
    else if (lane >= 8) { at = 8ull + 4ull * c + (uint64_t)lane - 9u; need = 32ull + 16ull * nc; rd = rd && nc > 0 && !(c == 0 && lane == 8); }
    ChunkEnds r;
    r.v = rd && have >= need ? __ldg(s32 + at) : 0u;
    const uint32_t h1 = __shfl_sync(0xffffffffu, r.v, 1), md = h1 >> 16;
    r.mode = (int)md;
    uint32_t want = kMagic;                           // of the header's word `lane`
    if (lane == 1) want = h1;
    if (lane == 2) want = w;
    if (lane == 3) want = hgt;
    if (lane == 4) want = 4u;
    if (lane == 5) want = (uint32_t)kChunk;
    if (lane == 6) want = nc;
    if (lane == 7) want = md == 0u ? 1u : 4u;
    const uint32_t up = __shfl_up_sync(0xffffffffu, r.v, 1);
    const uint64_t tab = (md == 0u ? 4ull : 16ull) * nc;                  // bytes of the end table
    const uint64_t psize = size - 32ull - tab;                           // (used only where the table is there)
    bool bad = lane < 8 && r.v != want;
    if (nc > 0) {
        const uint32_t clen = min((uint32_t)kChunk, w * hgt - c * (uint32_t)kChunk);
        if (md == 0u) {
            const uint32_t u = clen / 2;
            bad |= lane == 14 && (r.v < up || r.v - up > 8u * u + (u + 127u) / 128u + 4u * (clen & 1u) || r.v > psize);
        } else {
            // longer than the all-literal coding: longer than any valid stream
            bad |= lane >= 9 && lane < 13 && (r.v < up || r.v - up > clen + (clen + 127u) / 128u);
            bad |= lane == 12 && r.v > psize;
        }
    }
    r.bad = __any_sync(0xffffffffu, bad) || size < 32u || (nc > 0 && size < 32u + tab) || (h1 & 0xFFFFu) != 1u ||
            md > 2u || (md == 0u && !allow0);
    return r;
}

// Readers of stream bytes: src(i) returns payload byte i.
struct GlobalBytes {
    const uint8_t* __restrict__ p;
    __device__ __forceinline__ uint32_t operator()(int i) const { return (uint32_t)__ldg(p + i); }
};
struct SharedBytes {     // bytes [off, ...) of the payload staged at p
    const uint8_t* p;
    int off;
    __device__ __forceinline__ uint32_t operator()(int i) const { return (uint32_t)p[i - off]; }
};

// Each lane's repeat token (rep): olen copies of byte tv at plane[o, o+olen).
// The lane writes the unaligned head and tail bytes and a body of at most 8
// words itself (straight-line predicated stores: loops cost three times the
// instructions); longer bodies are written by the whole warp, one per store.
__device__ __forceinline__ void write_repeats(uint8_t* plane, bool rep, int o, int olen, uint32_t tv, int lane)
{
    uint32_t* p32 = reinterpret_cast<uint32_t*>(plane);
    const int e = o + olen, w0 = (o + 3) >> 2, nw = rep ? (e >> 2) - w0 : 0;   // whole words
    const uint32_t wv = 0x01010101u * (tv & 0xFFu);
    if (rep) {
        const int he = min(4 * w0, e), tb = max(e & ~3, he);      // head [o, he), tail [tb, e)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (o + k < he) plane[o + k] = (uint8_t)tv;
            if (tb + k < e) plane[tb + k] = (uint8_t)tv;
        }
        if (nw <= 8) {
            uint32_t* q = p32 + w0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (k < nw) q[k] = wv;
        }
    }
    const uint32_t pk = (uint32_t)w0 | ((uint32_t)nw << 16);
    for (uint32_t m = __ballot_sync(0xffffffffu, nw > 8); m; m &= m - 1u) {
        const int t = __ffs(m) - 1;
        const uint32_t q = __shfl_sync(0xffffffffu, pk, t);
        const uint32_t x = __shfl_sync(0xffffffffu, wv, t);
        if ((uint32_t)lane < (q >> 16)) p32[(q & 0xFFFFu) + lane] = x;
    }
}

__device__ __forceinline__ int warp_incl_sum(int v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// One warp decodes the stream payload[beg, end) into plane[0, len) (4-byte
// aligned).  Returns nonzero (the same on every lane) when a token runs past
// its stream or the chunk, or the stream does not yield exactly len bytes.
// The stream is read a 128-byte line at a time, a word per lane, two lines
// ahead, so no step waits for memory once the first line is in; it is taken in
// windows of 64 bytes, two per lane.  Tokens take at least two bytes, so a lane's pair
// holds at most one token start.  Repeat tokens that follow one another start
// in one byte of consecutive lanes' pairs, so the start masks of the window
// come from the two ballots of the repeat controls, a bit scan per literal
// token; a scan of the tokens' lengths over the lanes places them.  Literal
// bytes go straight from the lane that holds them to their place (the shift
// from stream to plane position comes from the lane of the last token start),
// and a window inside one literal token is copied without any parsing.
//
// Bound by instruction issue (21 K warp instructions per chunk, 67 % of the issue
// slots: the planes of a chunk are of uneven length, and its warps wait for the
// longest).  Windows of 32 bytes, each with a dependent load and five levels of
// shuffles, and a loop per literal token: the decoder launch over 8 shaded
// 1920x1080 sources, RGBA8 + depth, took 265 us; this: 127 us.
struct GlobalWords {      // payload bytes; reads stay below `end`
    const uint8_t* __restrict__ p;
    __device__ __forceinline__ uint32_t operator()(int off, int end) const
    {
        if (off + 4 <= end) return __ldg(reinterpret_cast<const uint32_t*>(p + off));
        uint32_t w = 0u;
        for (int k = 0; off + k < end; ++k) w |= (uint32_t)__ldg(p + off + k) << (8 * k);
        return w;
    }
};

template <class Words>
__device__ __forceinline__ int decode_plane_dense(const Words& words, int beg, int end, int len, uint8_t* plane,
                                                  int lane)
{
    constexpr int kNone = -(1 << 20);                 // no literal token is open
    const int a0 = beg & ~3, n = end - a0;            // stream bytes [a0, end), windows relative to a0
    const uint32_t lt = (1u << lane) - 1u;
    uint32_t L0 = words(a0 + 4 * lane, end), L1 = words(a0 + 128 + 4 * lane, end);
    uint32_t L2 = words(a0 + 256 + 4 * lane, end);
    int p = beg - a0;                                 // next token start, relative to the window
    int carry = kNone;                                // literal open at the window's start: plane - window position
    int outp = 0;
    for (int wb = 0; wb < n; wb += 64) {
        const int odd = (wb >> 6) & 1;
        const uint32_t x = __shfl_sync(0xffffffffu, L0, 16 * odd + (lane >> 1));
        const uint32_t pair = (lane & 1) ? x >> 16 : x & 0xFFFFu;
        const uint32_t b0 = pair & 0xFFu, b1 = pair >> 8;
        const int lim = min(64, n - wb);
        if (p >= lim) {                               // inside one literal token (or past the stream's end)
            if (carry != kNone) {
                if (2 * lane < lim) plane[2 * lane + carry] = (uint8_t)b0;
                if (2 * lane + 1 < lim) plane[2 * lane + 1 + carry] = (uint8_t)b1;
                carry += 64;
            }
        } else {
            uint32_t nx = __shfl_down_sync(0xffffffffu, pair, 1);
            const uint32_t wn = __shfl_sync(0xffffffffu, odd ? L1 : L0, odd ? 0 : 16);   // the next window's first
            if (lane == 31) nx = wn;
            // lanes whose first / second byte would be a literal control (bytes past lim read as 0)
            const uint32_t N0 = __ballot_sync(0xffffffffu, b0 < 128u), N1 = __ballot_sync(0xffffffffu, b1 < 128u);
            uint32_t T0 = 0u, T1 = 0u;                // lanes whose first / second byte starts a token
            while (p < lim) {                         // repeats in a row and the literal (if any) behind them
                const bool s = p & 1;
                const uint32_t from = 0xFFFFFFFFu << (p >> 1), t = (s ? N1 : N0) & from, low = t & (0u - t);
                const uint32_t starts = (2u * low - 1u) & from;
                if (s) T1 |= starts;
                else T0 |= starts;
                const int k = low ? 31 - __clz(low) : 32;
                p = 2 * k + (s ? 1 : 0);
                if (p < lim) p += 2 + (int)__shfl_sync(0xffffffffu, s ? b1 : b0, k);
            }
            if (lim < 64) {                           // the stream's last bytes: no token starts past them
                T0 &= 0xFFFFFFFFu >> (31 - ((lim - 1) >> 1));
                T1 &= (1u << (lim >> 1)) - 1u;
            }
            const bool st0 = (T0 >> lane) & 1u, st1 = (T1 >> lane) & 1u, has = st0 || st1;
            const uint32_t ctl = st1 ? b1 : b0;
            const bool rep = ctl >= 128u;
            const int olen = has ? (rep ? (int)ctl - 127 : (int)ctl + 1) : 0;
            const int incl = warp_incl_sum(olen, lane);
            const int o = outp + incl - olen;
            outp += __shfl_sync(0xffffffffu, incl, 31);
            if (outp > len) return 1;                 // (every token of the window then ends inside the chunk)
            // literal bytes: plane - window position of the token that holds them
            const int dl = rep ? kNone : o - 2 * lane - (st1 ? 2 : 1);
            const uint32_t T = T0 | T1, before = T & lt;
            const int dp = __shfl_sync(0xffffffffu, dl, before ? 31 - __clz(before) : 0);
            const int d0 = before ? dp : carry;
            if (!st0 && d0 != kNone && 2 * lane < lim) plane[2 * lane + d0] = (uint8_t)b0;
            const int d1 = st0 ? dl : d0;
            if (!st1 && d1 != kNone && 2 * lane + 1 < lim) plane[2 * lane + 1 + d1] = (uint8_t)b1;
            carry = __shfl_sync(0xffffffffu, dl, 31 - __clz(T));          // (T is not empty: p was below lim)
            if (carry != kNone) carry += 64;
            write_repeats(plane, has && rep, o, olen, st1 ? nx & 0xFFu : b1, lane);
        }
        p -= 64;
        if (odd) {
            L0 = L1;
            L1 = L2;
            L2 = words(a0 + wb + 320 + 4 * lane, end);
        }
    }
    // the last token ends where the stream does (p is relative to the window after the last one)
    const int past = (n + 63) / 64 * 64;
    return p + past != n || outp != len;
}

// A token walk with decode_plane_dense's validation, recording runs instead of
// bytes: every repeat token and every literal byte starts a run, in position
// order.  A window of 32 stream bytes, one per lane: lane l knows where a token
// starting at its byte would be followed by the next one; composing these
// jumps by doubling (5 levels) gives every lane t the start of the window's
// t-th token, and a warp scan places them.  Where a window starts with repeat
// tokens no search is needed (each takes two bytes): lane l reads the pair at
// offset 2l and the leading repeats, up to 32, are placed with one scan.
// Run r starting at position o sets bit o of the plane's bitmap bm (zero on
// entry; 128 words) and stores its byte in val[r].  Returns 0 with *nruns set,
// 1 for a malformed stream, 2 once there would be more than cap runs (nothing
// about the stream's validity is then known).
template <class Src>
__device__ __forceinline__ int decode_plane_runs(const Src& src, int beg, int end, int len, uint32_t* bm,
                                                 uint8_t* val, int cap, int* nruns, int lane)
{
    int cur = beg, outp = 0, runs = 0;
    while (cur < end) {
        {
            const int i2 = cur + 2 * lane;
            const uint32_t c = i2 + 1 < end ? src(i2) : 0u;
            const uint32_t v = i2 + 1 < end ? src(i2 + 1) : 0u;
            const uint32_t lit = __ballot_sync(0xffffffffu, c < 128u);
            const int m = lit ? __ffs(lit) - 1 : 32;
            if (m > 0) {
                const bool valid = lane < m;
                const int olen = valid ? (int)c - 127 : 0;
                const int incl = warp_incl_sum(olen, lane);
                const int total = __shfl_sync(0xffffffffu, incl, 31);
                const int o = outp + incl - olen;
                if (__any_sync(0xffffffffu, valid && o + olen > len)) return 1;
                if (runs + m > cap) return 2;
                if (valid) {
                    atomicOr(bm + (o >> 5), 1u << (o & 31));
                    val[runs + lane] = (uint8_t)v;
                }
                runs += m;
                outp += total;
                cur += 2 * m;
                continue;
            }
        }
        const int i = cur + lane;
        const uint32_t b = i < end ? src(i) : 0u;
        const uint32_t b1 = i + 1 < end ? src(i + 1) : 0u;
        int J = lane + (b >= 128u ? 2 : 2 + (int)b);   // next^(2^k), relative to cur
        int pos = 0;                                   // start of token #lane
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            const int y = __shfl_sync(0xffffffffu, J, min(pos, 31));
            if (((lane >> k) & 1) && pos < 32) pos = y;
            if (k < 4) {
                const int z = __shfl_sync(0xffffffffu, J, min(J, 31));
                if (J < 32) J = z;
            }
        }
        const bool valid = pos < min(32, end - cur);
        const int ntok = __popc(__ballot_sync(0xffffffffu, valid));
        const int sl = __shfl_sync(0xffffffffu, pos, ntok);
        const int ps = min(pos, 31);
        const uint32_t tb = __shfl_sync(0xffffffffu, b, ps);
        const uint32_t tv = __shfl_sync(0xffffffffu, b1, ps);
        const bool trep = tb >= 128u;
        const int olen = valid ? (trep ? (int)tb - 127 : (int)tb + 1) : 0;
        const int tnext = pos + (trep ? 2 : 2 + (int)tb);
        const int incl = warp_incl_sum(olen, lane);
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        const int o = outp + incl - olen;
        if (__any_sync(0xffffffffu, valid && (cur + tnext > end || o + olen > len))) return 1;
        const int nr = valid ? (trep ? 1 : olen) : 0;      // runs this token starts
        const int rinc = warp_incl_sum(nr, lane);
        const int rtot = __shfl_sync(0xffffffffu, rinc, 31);
        if (runs + rtot > cap) return 2;
        const int rb = runs + rinc - nr;
        if (valid && trep) {
            atomicOr(bm + (o >> 5), 1u << (o & 31));
            val[rb] = (uint8_t)tv;
        }
        for (uint32_t m = __ballot_sync(0xffffffffu, valid && !trep); m; m &= m - 1u) {
            const int t = __ffs(m) - 1;
            const int oo = __shfl_sync(0xffffffffu, o, t);
            const int ml = __shfl_sync(0xffffffffu, olen, t);
            const int r0 = __shfl_sync(0xffffffffu, rb, t);
            const int s0 = cur + __shfl_sync(0xffffffffu, pos, t) + 1;   // after the control
            for (int k = lane; k < ml; k += 32) {
                atomicOr(bm + ((oo + k) >> 5), 1u << ((oo + k) & 31));
                val[r0 + k] = (uint8_t)src(s0 + k);
            }
        }
        runs += rtot;
        outp += total;
        cur += sl;
    }
    *nruns = runs;
    return outp != len;
}

}  // namespace rlec
}  // namespace ec
