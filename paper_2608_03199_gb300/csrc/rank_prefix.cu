// rank_prefix.cu -- the first ranks of the centroid order alone (Sec. 2.3,
// Sec. 4.1), for a search whose stopping rule visits few of its nprobe ranks.
//
// A search with a window of W visits min(W, nprobe) partitions plus what its
// hits add: about 8 of 256 ranks at W = 8.  So the search ranks a prefix
// first, and only the queries whose stop line passes their prefix get the
// whole ranking (the extension at the end of a round, below).
//
//   k_prefix_scan   one contraction pass on the screen (one fp16 product of
//              the hi halves per score, tiles of two 128-query sub-tiles).
//              Each epilogue thread owns one query and keeps its kL groups of
//              32 centroids with the largest maxima: the maxima sorted in
//              registers, each with its slot in the lowest bits, the 32 scores
//              stored as they are to the slot in global memory.  A group that
//              enters costs no search and no read: the smallest maximum names
//              the slot.  The kL largest scores lie in the kL groups with the
//              largest maxima, and a score of another group is no larger than
//              the smallest of those maxima.  The tile first passes over an
//              eighth of its chunks and keeps only the kL largest group
//              maxima, without a branch: kL groups reach the kL-th, and
//              starting from there about kL (1 + ln 8) groups enter instead
//              of kL (1 + ln(groups / kL)) in a random order.
//   k_prefix_final  one warp per query: of the kept groups' scores the kL best
//              (the scores that reach the smallest kept maximum), scored again
//              in fp32 and sorted by (score desc, id asc).  A centroid that
//              is not among them screens at most u, the largest of the lists'
//              bounds and of what was left out here, so its fp32 score is
//              below u plus the error bounds of both scores; the candidates
//              above that are exactly the first ranks of the order, and their
//              number is the query's limit.  Bound by latency: the scores and
//              the query are loaded before anything depends on them, and the
//              rows of eight candidates are in flight together (1M x 8,192 x
//              256: 4.6 ms with eight lanes a row and four rows at a time, 1.6).
//   k_ext_gather / k_ext_merge  the extension: the listed queries gathered
//              for the full ranking, whose order follows the prefix with the
//              prefix's centroids left out, so that no partition is visited
//              twice should the two disagree on a near-tie.
//
// The scan is bound by the epilogue and the single accumulator per sub-tile it
// holds meanwhile: two fifths of the tensor pipe's cycles are used at 8,192 x
// 256 (issue slots 21% busy: latency).  Against lists of single scores in
// shared memory, searched at each entry: 1M queries x 65,536 x 96 21.7 -> 13.4
// ms, 1M x 8,192 x 256 5.7 -> 4.7 ms; for 1,500 centroids, where two thirds of
// the groups enter, 0.22 ms per 100K both ways, and the final, which reads 2 KB
// a query and not 128 bytes, takes 0.17 ms, not 0.14.
// 12 slots instead of 16 (kL) scan faster (12.5 ms for the first) but extend
// more queries than that saves (the whole search 24.5 -> 25.4 ms).
// Against the full ranking (two contraction passes, ~310 candidates a query
// sorted): 1M queries x 65,536 x 96, nprobe 256, 52.1 -> 15.0 ms; 1M x 8,192 x
// 256, nprobe 128, 17.6 -> 6.3 ms; 100K x 1,500 x 96, nprobe 90, 1.35 -> 0.39 ms;
// 200K x 16,384 x 512, nprobe 128 (against the converter pipeline's three
// products), 16.2 -> 4.1 ms.
#include <cmath>
#include <vector>

#include "rank_select.cuh"
#include "tc_bulk.cuh"

namespace sieve {

struct PrefixArgs {
    const float *Q;
    int64_t nq, nlist;
    int d;
    int *status;
    int wait_limit;      // polls of the epilogue's accumulator wait (0: default)
    const unsigned char *tc_cent;
    int nranges;         // centroid ranges per query tile
    int64_t range_len;   // centroids per range, a multiple of 128
    float *list_s;       // [nq][nranges][kL][32] the kept groups' screened scores (raw: x 2^16) ...
    int2 *list_g;        // [nq][nranges][kL] ... their largest (raw, as bits) and first centroid
    float2 *list_t;      // [nq][nranges] x: what a score left out can be at most (raw; -inf: none
                         // was); y: groups kept, as bits (the last of the kL slots fill first)
};

__device__ int g_prefix_status_sink;

// Scores past fp16's range (|256 x| above 65,504) are not screened soundly, and
// a NaN row is left out by every maximum: with such centroids every prefix is
// empty.  (The scan runs for them all the same: returning at its start on these
// two words took the compiler to other code, 13.4 -> 13.7 ms for 1M queries x
// 65,536 x 96 that have no such centroids.)
constexpr float kScreenMaxNorm = 200.f;
__device__ __forceinline__ float norm_up(unsigned bits) { return __uint_as_float(bits) * (1.f + 0x1p-20f); }
__device__ __forceinline__ bool centroids_screen(unsigned norm, unsigned nan) {
    return nan == 0u && norm_up(norm) < kScreenMaxNorm;
}

// kSubT = 2: centroids in the tensor-core layout, d <= 256.  kSubT = 1: d <= 512,
// A's hi half alone fills 256 columns, and the centroids' hi halves in a layout
// of their own (k_prefix_fill: 16 KB per K-block).
template <int kL, int kNBT, int kSubT>
struct PrefixMode {
    using Args = PrefixArgs;
    static constexpr int kProducts = 1;
    static constexpr int kNB = kNBT;
    static constexpr int kSub = kSubT;
    static constexpr bool kBHasLo = kSubT == 2;
    static constexpr int kRows = kSub * tcp::kM;
    static constexpr bool kSampled = true;
    struct Tile {
        int64_t q0;
        int ni;
        int64_t c0, nb;
        int ns, sstep;   // sample chunks first: chunks 0, sstep, 2 sstep, ...
    };
    __device__ static int num_tiles(const Args &a) { return (int)ceil_div(a.nq, kRows) * a.nranges; }
    __device__ static int *tile_counter(const Args &) { return nullptr; }
    __device__ static int d(const Args &a) { return a.d; }
    __device__ static int *status(const Args &a) { return a.status ? a.status : &g_prefix_status_sink; }
    __device__ static uint32_t epi_wait_polls(const Args &a) { return (uint32_t)a.wait_limit; }
    __device__ static Tile tile(const Args &a, int t) {
        Tile T;
        T.q0 = (int64_t)(t / a.nranges) * kRows;
        T.ni = (int)(a.nq - T.q0 < kRows ? a.nq - T.q0 : kRows);
        T.c0 = (int64_t)(t % a.nranges) * a.range_len;
        T.nb = a.nlist - T.c0 < a.range_len ? a.nlist - T.c0 : a.range_len;
        // an eighth of the whole chunks where there are 16 or more
        const int whole = (int)(T.nb / kNBT);
        T.ns = whole >= 16 ? whole / 8 : 0;
        T.sstep = 8;
        return T;
    }
    __device__ static const float *a_row(const Args &a, const Tile &T, int i) {
        return i < T.ni ? a.Q + (T.q0 + i) * a.d : nullptr;
    }
    __device__ static const unsigned char *b_block(const Args &a, const Tile &T) {
        return a.tc_cent + (T.c0 / kTcRows) * (int64_t)((a.d + 63) / 64) * (kBHasLo ? tcb::kKbBytes : tcb::kKbBytesHi);
    }
    struct Epi {
        float *os;       // this query's kL slots of 32 scores
        int2 *og;
        int64_t at;
        int n;           // groups taken so far
        float floor;     // the sample's threshold (-inf: none; +inf: no query)
        float thr;       // raw units: groups whose maximum is no larger are out
        // the largest first: the sample's group maxima, then those of the kept
        // groups, each with its slot in the lowest bits (2^-18 of the value)
        float top[kL];
        __device__ __forceinline__ void clear() {
#pragma unroll
            for (int j = 0; j < kL; ++j) top[j] = __uint_as_float(0xff7fffe0u | (unsigned)j);   // about -3.4e38
        }
        __device__ void begin(const Args &a, const Tile &T, int slot, unsigned char *) {
            const bool valid = slot < T.ni;
            at = (T.q0 + slot) * a.nranges + T.c0 / a.range_len;
            os = a.list_s + at * (kL * 32);
            og = a.list_g + at * kL;
            n = 0;
            clear();
            floor = valid ? -__int_as_float(0x7f800000) : __int_as_float(0x7f800000);
            thr = fmaxf(floor, top[kL - 1]);
        }
        __device__ __forceinline__ void insert(float x) {   // the smallest leaves
#pragma unroll
            for (int j = 0; j < kL; ++j) {
                const float hi = fmaxf(top[j], x);
                x = fminf(top[j], x);
                top[j] = hi;
            }
        }
        // a sample chunk's scores: the maximum of the 32 into the sorted
        // registers, without a branch (whole chunks only: no column is past
        // the range)
        __device__ __forceinline__ void sample(const float (&v)[32]) { insert(max_of_32(v)); }
        // the sample is through: kL different groups reach top[kL - 1], so
        // only groups from there up are kept (the threshold is the value just
        // below it; the slots then fill)
        __device__ __forceinline__ void seed() {
            const float t = top[kL - 1];
            if (floor < 0.f && t > -3.4e38f && t < 3.4e38f) floor = t - fmaxf(fabsf(t), 1.f) * 0x1p-22f;
            clear();
            thr = fmaxf(floor, top[kL - 1]);
        }
        // a group whose maximum mx passes the threshold takes the slot of the
        // one that leaves
        __device__ __forceinline__ void take(const float (&v)[32], float mx, int32_t id0) {
            const unsigned slot = __float_as_uint(top[kL - 1]) & (unsigned)(kL - 1);
            insert(__uint_as_float((__float_as_uint(mx) & ~(unsigned)(kL - 1)) | slot));
            thr = fmaxf(floor, top[kL - 1]);
            ++n;
            float4 *o = reinterpret_cast<float4 *>(os + slot * 32);
#pragma unroll
            for (int j = 0; j < 8; ++j) o[j] = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            og[slot] = make_int2(__float_as_int(mx), id0);
        }
        // v: the chunk's raw accumulator values (scores x 2^16) of centroids
        // T.c0 + col0 + j, j < ncol (warp-uniform)
        __device__ __forceinline__ void chunk(const Args &, const Tile &T, int64_t col0,
                                              const float (&v)[32], int ncol) {
            if (ncol <= 0) return;
            const int32_t id0 = (int32_t)(T.c0 + col0);
            if (ncol == 32) {
                const float mx = max_of_32(v);
                if (mx > thr) take(v, mx, id0);
            } else {   // the range's last group: -inf past its end
                float w[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) w[j] = j < ncol ? v[j] : -__int_as_float(0x7f800000);
                const float mx = max_of_32(w);
                if (mx > thr) take(w, mx, id0);
            }
            __syncwarp();
        }
        __device__ void end(const Args &a, const Tile &) {
            if (floor > 3.4e38f) return;
            // a group left out had a maximum of thr at most, give or take the slot bits
            const float t = thr + (fabsf(thr) * 0x1p-18f + 0x1p-100f);
            a.list_t[at] = make_float2(n >= kL ? t : -__int_as_float(0x7f800000), __int_as_float(n < kL ? n : kL));
        }
        __device__ void prefetch(const Args &, const Tile &, int) {}
        __device__ void start(const Args &, const Tile &, int) {}
    };
};

template <int kL, int kNBT, int kSubT>
__global__ void __launch_bounds__(tcb::kThreads, 1) k_prefix_scan(PrefixArgs a, int stages) {
    extern __shared__ unsigned char smem_raw[];
    tcb::run_bulk<PrefixMode<kL, kNBT, kSubT>>(a, smem_raw, stages);
}

// The centroids' hi halves in the tensor-core layout's order, for rows wider
// than an index keeps a layout of by default: a thread per (block, K-block,
// row, 16-byte chunk), rows past nlist and columns past d zero.  Bound by
// memory (6d bytes a centroid, once per call).
__global__ void k_prefix_fill(const float *__restrict__ C, int64_t nlist, int d, int nkb,
                              unsigned char *__restrict__ out) {
    const int64_t total = ceil_div(nlist, kTcRows) * nkb * kTcRows * 8;
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < total;
         u += (int64_t)gridDim.x * blockDim.x) {
        const int c = (int)(u & 7), r = (int)((u >> 3) & (kTcRows - 1));
        const int64_t bk = u >> 10, row = bk / nkb * kTcRows + r;
        const int col = (int)(bk % nkb) * 64 + c * 8;
        const float *src = row < nlist ? C + row * d : nullptr;
        const float4 x0 = tcp::load_f4(src, col, d), x1 = tcp::load_f4(src, col + 4, d);
        uint4 h, l;
        tcp::split2(x0.x, x0.y, h.x, l.x);
        tcp::split2(x0.z, x0.w, h.y, l.y);
        tcp::split2(x1.x, x1.y, h.z, l.z);
        tcp::split2(x1.z, x1.w, h.w, l.w);
        *reinterpret_cast<uint4 *>(out + bk * tcb::kKbBytesHi + (int64_t)r * 128 + ((c ^ (r & 7)) << 4)) = h;
    }
}

// The B partial sums of each lane added up over the warp, halving the sums a
// lane holds at each step: the sum of acc[j] ends in lanes j * 32 / B and on.
template <int B>
__device__ __forceinline__ float warp_sum_each(float (&acc)[B]) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int c = B; c > 1; c >>= 1, off >>= 1) {
        const bool hi = lane & off;
#pragma unroll
        for (int i = 0; i < c / 2; ++i) {
            const float keep = hi ? acc[i + c / 2] : acc[i], send = hi ? acc[i] : acc[i + c / 2];
            acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (int o = 16 / B; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
    return acc[0];
}

// One warp per query.  NV: float4 of a row per lane (d <= 128 NV); KPL: kept
// groups per lane (nranges * kL <= 32 KPL).  A scan that gave up on a wait
// leaves lists that an earlier call wrote, or nobody: every id is
// kept below nlist before a row is read, and with the status word set, or
// centroids that are not screened, every prefix is empty.  (Asked at the end,
// where the answer is at hand: 1M queries 1.59 ms; a branch up front 1.76.)
constexpr int kFinalWarps = 8;
template <int kL, int KPL, int NV>
__global__ void __launch_bounds__(kFinalWarps * 32) k_prefix_final(
    const float *__restrict__ Q, int64_t nq, const float *__restrict__ C, int64_t nlist, int d,
    const float *__restrict__ list_s, const int2 *__restrict__ list_g,
    const float2 *__restrict__ list_t, int nranges, int nprobe, const unsigned *__restrict__ cmax,
    const int *__restrict__ status, int32_t *__restrict__ order, float *__restrict__ cscores,
    int *__restrict__ limit) {
    constexpr float kS = 1.f / 65536.f;
    __shared__ int s_id[kFinalWarps][32];
    __shared__ int s_slot[kFinalWarps][kL], s_c0[kFinalWarps][kL];   // the groups taken on: slot, first centroid
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int64_t q = (int64_t)blockIdx.x * kFinalWarps + warp;
    if (q >= nq) return;
    const int M = nranges * kL;
    // one list: its scores and the query's row are on their way at once
    float raw[kL];
    if (M == kL) {
#pragma unroll
        for (int g = 0; g < kL; ++g) raw[g] = __ldg(list_s + (q * kL + g) * 32 + lane);
    }
    float4 x[NV];
#pragma unroll
    for (int t = 0; t < NV; ++t) {
        const int c = 4 * lane + 128 * t;
        x[t] = c < d ? __ldg(reinterpret_cast<const float4 *>(Q + q * d + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    uint32_t un = 0;   // the largest screened score a centroid outside the candidates can have
    for (int r = lane; r < nranges; r += 32) {
        const float t = list_t[q * nranges + r].x;
        if (t > -__int_as_float(0x7f800000)) un = max(un, order_key(t * kS));
    }
    // the kL groups with the largest maxima of all ranges
    uint32_t gkey[KPL];
    int c0[KPL];
#pragma unroll
    for (int j = 0; j < KPL; ++j) {
        const int c = j * 32 + lane;
        gkey[j] = 0u;
        c0[j] = -1;
        if (c < M) {
            const int used = __float_as_int(list_t[q * nranges + c / kL].y);
            const int2 g = list_g[q * M + c];
            if (c % kL >= kL - used && (uint32_t)g.y < (uint64_t)nlist) {
                gkey[j] = order_key(__int_as_float(g.x) * kS);
                c0[j] = g.y;
            }
        }
    }
    uint32_t T = 1u, least = 0xffffffffu;
    int cnt, ng = 0;
    if (M == kL) {
        ng = __popc(__ballot_sync(0xffffffffu, gkey[0] > 0u));
        if (gkey[0] > 0u) least = gkey[0];
        if (lane < kL) s_c0[warp][lane] = c0[0];
    } else {
        warp_threshold(gkey, kL, kL, T, cnt);
        T = max(T, 1u);
#pragma unroll
        for (int j = 0; j < KPL; ++j) {
            const bool sel = gkey[j] >= T;
            const unsigned b = __ballot_sync(0xffffffffu, sel);
            const int p = ng + __popc(b & below);
            if (sel && p < kL) {
                s_slot[warp][p] = j * 32 + lane;
                s_c0[warp][p] = c0[j];
                least = min(least, gkey[j]);
            } else {   // not among them (or one of too many equal ones)
                un = max(un, gkey[j]);
            }
            ng += __popc(b);
        }
        ng = ng < kL ? ng : kL;
        __syncwarp();
#pragma unroll
        for (int g = 0; g < kL; ++g)
            raw[g] = g < ng ? list_s[(q * M + s_slot[warp][g]) * 32 + lane] : 0.f;
    }
    __syncwarp();
    // the kL best of their scores (or a few more), one candidate per lane: the
    // scores that reach the least of the groups' maxima are at least kL, and
    // seldom more than 32 (neighbours in one group): only then a search
    int id = -1, n = 0;
    T = __reduce_min_sync(0xffffffffu, least);
    const float t_raw = key_score(T) * 65536.f;
    int reach = 0;
    if (ng == kL) {
#pragma unroll
        for (int g = 0; g < kL; ++g) reach += __popc(__ballot_sync(0xffffffffu, raw[g] >= t_raw));
    }
    if (ng == kL && reach <= 32) {   // every other score is below T
        un = max(un, T);
#pragma unroll
        for (int g = 0; g < kL; ++g) {
            const bool sel = raw[g] >= t_raw;   // past the centroids the score is -inf
            const unsigned b = __ballot_sync(0xffffffffu, sel);
            if (sel) s_id[warp][n + __popc(b & below)] = (int)min((unsigned)s_c0[warp][g] + lane, (unsigned)nlist - 1u);
            n += __popc(b);
        }
    } else {
        uint32_t key[kL];
#pragma unroll
        for (int g = 0; g < kL; ++g) {
            const int b = M == kL || g < ng ? s_c0[warp][g] : -1;
            key[g] = b >= 0 && b + (int64_t)lane < nlist ? order_key(raw[g] * kS) : 0u;
        }
        warp_threshold(key, kL, 32, T, cnt);
        T = max(T, 1u);
#pragma unroll
        for (int g = 0; g < kL; ++g) {
            const bool sel = key[g] >= T;
            const unsigned b = __ballot_sync(0xffffffffu, sel);
            const int p = n + __popc(b & below);
            if (sel && p < 32)
                s_id[warp][p] = s_c0[warp][g] + lane;
            else
                un = max(un, key[g]);
            n += __popc(b);
        }
    }
    n = n < 32 ? n : 32;
    __syncwarp();
    if (lane < n) id = s_id[warp][lane];
    un = __reduce_max_sync(0xffffffffu, un);
    // fp32 scores: the whole warp on a candidate, the rows of kB of them in
    // flight together
    constexpr int kB = NV == 1 ? 8 : 16 / NV;
    float s[1] = {-__int_as_float(0x7f800000)};
    int cid[1] = {id >= 0 ? id : INT32_MAX};
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += kB) {
        float4 y[kB][NV];
#pragma unroll
        for (int i = 0; i < kB; ++i) {
            // without a branch: past the last candidate the last again, past
            // the row its start (times x = 0)
            const float *row = C + (int64_t)s_id[warp][i0 + i < n ? i0 + i : n - 1] * d;
#pragma unroll
            for (int t = 0; t < NV; ++t) {
                const int c = 4 * lane + 128 * t;
                y[i][t] = __ldg(reinterpret_cast<const float4 *>(row + (c < d ? c : 0)));
            }
        }
        float acc[kB];
#pragma unroll
        for (int i = 0; i < kB; ++i) {
            acc[i] = 0.f;
#pragma unroll
            for (int t = 0; t < NV; ++t) {
                acc[i] = fmaf(x[t].x, y[i][t].x, acc[i]);
                acc[i] = fmaf(x[t].y, y[i][t].y, acc[i]);
                acc[i] = fmaf(x[t].z, y[i][t].z, acc[i]);
                acc[i] = fmaf(x[t].w, y[i][t].w, acc[i]);
            }
        }
        const float sum = warp_sum_each<kB>(acc);
        const float mine = __shfl_sync(0xffffffffu, sum, (lane - i0) * (32 / kB) & 31);
        if (lane >= i0 && lane < i0 + kB && id >= 0) s[0] = mine;
    }
    float qq = 0.f;
#pragma unroll
    for (int t = 0; t < NV; ++t)
        qq = fmaf(x[t].x, x[t].x, fmaf(x[t].y, x[t].y, fmaf(x[t].z, x[t].z, fmaf(x[t].w, x[t].w, qq))));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) qq += __shfl_xor_sync(0xffffffffu, qq, o);
    warp_sort_regs<1>(s, cid);
    // the norms and the margin rounded upward (the bounds of k_rank_threshold:
    // the screen's, and one that covers fp32 sums with room)
    const float qn = __fsqrt_ru(qq) * (1.f + 0x1p-20f);
    const unsigned cmax0 = cmax[0];
    const float cn = norm_up(cmax0);
    const float rd = __fsqrt_ru((float)d);
    const float fp32 = (0x1p-20f + (float)d * 0x1p-22f) * qn * cn + 0x1p-26f * rd * (qn + cn);
    const float scr = (0x1p-10f + 0x1p-12f + (float)d * 0x1p-22f) * qn * cn + 0x1p-26f * rd * (qn + cn);
    const float margin = (scr + fp32) * (1.f + 0x1p-16f);
    const bool usable = (!status || *status == 0) && centroids_screen(cmax0, cmax[1]);
    const bool first = usable && qn < kScreenMaxNorm && cid[0] != INT32_MAX &&
                       (un == 0u || s[0] > __fadd_ru(key_score(un), margin));
    const unsigned b = __ballot_sync(0xffffffffu, first);
    int R = b == 0xffffffffu ? 32 : __ffs(~b) - 1;   // the sorted entries up to the first that may not be
    R = R < nprobe ? R : nprobe;
    if (lane < R) {
        order[q * nprobe + lane] = cid[0];
        if (cscores) cscores[q * nprobe + lane] = s[0];
    }
    if (lane == 0) limit[q] = R;
}

// row i of Qx = query ext[q0 + i] (a warp per row), for the listed queries of
// this chunk; the first chunk of a part (-1: another) counts its run
__global__ void k_ext_gather(const float *__restrict__ Q, int d, const int *__restrict__ ext,
                             Ctl *ctl, int64_t q0, int64_t chunk, float *__restrict__ Qx, int part) {
    const int ext_n = ctl->ext_n;
    if (part >= 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->ext_runs[part] += 1;
        if (part == 0) ctl->tot_ext += (unsigned long long)ext_n;
    }
    const int64_t left = (int64_t)ext_n - q0, n = left < chunk ? left : chunk;
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        const float *src = Q + (int64_t)ext[q0 + i] * d;
        for (int c = 4 * lane; c < d; c += 128)
            *reinterpret_cast<float4 *>(Qx + i * d + c) = *reinterpret_cast<const float4 *>(src + c);
    }
}

// A warp per listed query: ranks limit + 1 .. nprobe of its order become the
// full ranking's centroids, in order, without the limit[q] <= 32 of its prefix.
__global__ void k_ext_merge(const int *__restrict__ ext, const int *__restrict__ ext_n, int64_t q0,
                            int64_t chunk, int nprobe, const int32_t *__restrict__ full,
                            const float *__restrict__ full_s, int32_t *__restrict__ order,
                            float *__restrict__ cscores, int *__restrict__ limit) {
    const int64_t left = (int64_t)*ext_n - q0, n = left < chunk ? left : chunk;
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        const int64_t q = ext[q0 + i];
        const int R = limit[q];
        const int32_t mine = lane < R ? order[q * nprobe + lane] : -1;
        int at = R;
        for (int p0 = 0; p0 < nprobe && at < nprobe; p0 += 32) {
            const int p = p0 + lane;
            const int32_t c = p < nprobe ? full[i * nprobe + p] : -2;
            bool keep = p < nprobe;
            for (int r = 0; r < R; ++r) {   // every lane takes part in each shuffle
                const int32_t pr = __shfl_sync(0xffffffffu, mine, r);
                keep = keep && c != pr;
            }
            const unsigned b = __ballot_sync(0xffffffffu, keep);
            const int o = at + __popc(b & below);
            if (keep && o < nprobe) {
                order[q * nprobe + o] = c;
                if (cscores) cscores[q * nprobe + o] = full_s[i * nprobe + p];
            }
            at += __popc(b);
        }
        __syncwarp();
        if (lane == 0) limit[q] = nprobe;
    }
}

// ---------------------------------------------------------------------------
static bool prefix_wide(int d) { return ceil_div(d, 64) <= 2; }   // 192-centroid chunks, as the screen
static int prefix_sub(int d) { return ceil_div(d, 64) <= 4 ? 2 : 1; }   // sub-tiles of 128 queries per tile
static uint32_t prefix_stage_bytes(int d) {
    return prefix_wide(d) ? tcb::kStageBytesHi / tcb::kN * 192 : tcb::kStageBytesHi;
}

static int prefix_stages(int d) {
    const int nkb = (int)ceil_div(d, 64);
    return tcb::sub_fits(nkb, 1, prefix_sub(d))
               ? tcb::stages_for(nkb, 0, 232448 - 128, prefix_stage_bytes(d), tcb::kStagesMax,
                                 tcb::kMaxKb)
               : 0;
}

// bytes of the centroids' hi halves kept in the scratch (k_prefix_fill)
static int64_t fill_bytes(int64_t nlist, int d) {
    return prefix_sub(d) == 2 ? 0 : ceil_div(nlist, kTcRows) * ceil_div(d, 64) * tcb::kKbBytesHi;
}

// Groups kept per list, and so ranks found: min(W, nprobe) are visited for
// certain, a hit at rank j adds up to rank j + W, and one or two are lost to
// the margin.  16 serve windows up to 10 and 32 up to 24; 0: rank all of nprobe (a
// wider window reads most of the order anyway).
//
// Fewer than L groups of 32 in all are all kept, and nothing is left out: the
// full ranking is as quick or quicker (W 8, tau 0.9, prefix against full:
// 16,384 queries x 64 x 96 313 and 287 us, x 512 x 96 258 and 276, 8,192 x 768 x
// 96 192 and 229; W 20: 8,192 x 512 x 96 279 and 249, 16,384 x 1,500 x 96 411
// and 692).
//
// About 0.15% of the queries go past 13 ranks at W 8 and tau 0.9 on the
// synthetic mixtures, and 6e-5 past 20.  The first of them costs a small batch
// a full ranking's latency (1,024 x 16,384 x 96: about 215 us of 595), so where
// a batch is likely to have one and its time is latency still, 32 groups are
// kept: 1,024 x 16,384 x 96 595 -> 450 us (526 ranked whole), 4,096 925 -> 748
// (822), 4,096 x 1,024 x 256 572 -> 502 (505); where nobody goes past 16 it
// costs 5 to 10% (1,024 x 8,192 x 256 301 -> 317, 4,096 440 -> 485).  From 8,192
// queries the longer lists cost more than they save (easy: 8,192 x 8,192 x 96
// 408 -> 489; mixture: 8,192 x 16,384 x 96 1,071 -> 1,040), below 256 such a
// query is rare (64 x 16,384 x 96 180 -> 197).
constexpr int64_t kLongLists = 256, kLongListsEnd = 8192;
static bool prefix_fits(int64_t nlist, int nprobe, int d, int L) {
    return nlist >= 32 * (int64_t)L && nprobe >= 4 && prefix_stages(d) > 0;
}

int rank_prefix_len(int64_t nq, int64_t nlist, int nprobe, int W, int d) {
    const int need = W < nprobe ? W : nprobe;
    if (need > 24) return 0;
    if ((need > 10 || (nq >= kLongLists && nq < kLongListsEnd)) && prefix_fits(nlist, nprobe, d, 32)) return 32;
    return need <= 10 && prefix_fits(nlist, nprobe, d, 16) ? 16 : 0;
}

// bytes of one (query, range)'s list: the scores, maxima and first centroids of
// L groups, the bound and the count
static int64_t list_bytes(int L) { return (int64_t)L * (32 * 4 + 8) + 8; }

struct PrefixPlan {
    int nranges;
    int64_t range_len;
};

// Ranges: enough tiles to fill the SMs in whole waves.  A tile costs its chunks
// plus about six chunks' time for writing A and filling the lists.
static PrefixPlan prefix_plan(int64_t nq, int64_t nlist, int d, int L) {
    const int64_t tiles = std::max<int64_t>(1, ceil_div(nq, prefix_sub(d) * tcp::kM)), sms = num_sms();
    const int64_t nb = prefix_wide(d) ? 192 : 128;
    const int64_t most = std::min<int64_t>(ceil_div(nlist, kTcRows), std::min<int64_t>(1024 / L, 32));
    PrefixPlan best{1, round_up(nlist, (int64_t)kTcRows)};
    int64_t best_cost = INT64_MAX;
    for (int64_t r = 1; r <= most; ++r) {
        const int64_t len = round_up(ceil_div(nlist, r), (int64_t)kTcRows), nr = ceil_div(nlist, len);
        const int64_t cost = ceil_div(tiles * nr, sms) * (ceil_div(len, nb) + 6);
        if (cost < best_cost) {
            best_cost = cost;
            best = PrefixPlan{(int)nr, len};
        }
        if (tiles * r >= 16 * sms) break;
    }
    return best;
}

// Layout of the ranking scratch of a search with a prefix: the limits and the
// extension list (kept for the whole search), then the lists of a chunk of
// queries (the prefix) or the extension's buffers, which are never live at once.
struct PrefixScratch {
    int64_t limit, ext, rest;      // byte offsets
    int64_t fill, lists;           // the prefix's part: the centroids' hi halves, the lists
    int64_t chunk;                 // queries per prefix pass
    struct Ext {                   // a part of the extension: queries per pass, and byte offsets
        int64_t chunk;             // of its buffers (after its ranking scratch)
        int64_t q, order, s, end;
    } ext_part[kExtParts];
    int64_t total;
};

static PrefixScratch::Ext ext_part(int64_t rest, int64_t x, int64_t nlist, int nprobe, int d) {
    PrefixScratch::Ext E{};
    E.chunk = x;
    E.q = rest + round_up((int64_t)rank_tc_scratch_bytes(x, nlist, nprobe, d), 256);
    E.order = E.q + round_up(x * d * 4, 256);
    E.s = E.order + round_up(x * nprobe * 4, 256);
    E.end = E.s + round_up(x * nprobe * 4, 256);
    return E;
}

// The scratch is what the full ranking takes (plain), or up to kPrefixListBytes
// of lists where that is more; a smaller chunk only means more passes, and a
// chunk past one wave of tiles is a number of whole waves.
constexpr int64_t kPrefixListBytes = int64_t(1) << 30;
static PrefixScratch prefix_scratch(int64_t nq, int64_t nlist, int nprobe, int d, int L) {
    PrefixScratch S{};
    const int64_t plain = (int64_t)rank_tc_scratch_bytes(nq, nlist, nprobe, d);
    S.limit = 0;
    S.ext = round_up(nq * 4, 256);
    S.rest = S.ext + round_up(nq * 4, 256);
    S.total = plain;
    for (int i = 0; ext_part_of(i, nq); ++i) {
        PrefixScratch::Ext &E = S.ext_part[i];
        E = ext_part(S.rest, ext_end(i, nq) - ext_begin(i), nlist, nprobe, d);
        const int64_t least = ext_begin(1);   // more passes before more scratch, down to this many queries
        while (E.end > S.total && E.chunk > least)
            E = ext_part(S.rest, std::max(least, round_up(ceil_div(E.chunk, 2), (int64_t)128)), nlist, nprobe, d);
        S.total = std::max(S.total, E.end);
    }
    const PrefixPlan P = prefix_plan(nq, nlist, d, L);
    const int64_t per = (int64_t)P.nranges * list_bytes(L), least = std::min<int64_t>(nq, 2 * tcp::kM) * per;
    S.fill = S.rest + 256;
    S.lists = S.fill + fill_bytes(nlist, d);
    S.total = std::max(S.total, S.lists + std::max(least, std::min(nq * per, kPrefixListBytes)) + 256);
    S.chunk = (S.total - S.lists - 256) / per;
    if (S.chunk < nq) {
        const int64_t tile = 2 * tcp::kM, wave = tile * num_sms();
        S.chunk = std::max(tile, S.chunk / (S.chunk < wave ? tile : wave) * (S.chunk < wave ? tile : wave));
    }
    S.chunk = std::min(nq, S.chunk);
    return S;
}

// W = 0: for any window
size_t rank_prefix_scratch_bytes(int64_t nq, int64_t nlist, int nprobe, int W, int d) {
    int64_t b = 0;
    for (int L : {16, 32})
        if (nq > 0 && (W == 0 ? prefix_fits(nlist, nprobe, d, L) : rank_prefix_len(nq, nlist, nprobe, W, d) == L))
            b = std::max(b, prefix_scratch(nq, nlist, nprobe, d, L).total);
    return (size_t)b;
}

int *rank_prefix_limit(void *scratch, int64_t nq, int64_t nlist, int nprobe, int W, int d, int **ext) {
    const PrefixScratch S = prefix_scratch(nq, nlist, nprobe, d, rank_prefix_len(nq, nlist, nprobe, W, d));
    unsigned char *w = static_cast<unsigned char *>(scratch);
    *ext = reinterpret_cast<int *>(w + S.ext);
    return reinterpret_cast<int *>(w + S.limit);
}

static size_t scan_smem(int d) {
    return tcb::smem_bytes(prefix_stages(d), 0, prefix_stage_bytes(d));
}

// the scan kernel of this d and list length
using PrefixScan = void (*)(PrefixArgs, int);
static PrefixScan scan_kernel(int d, int L) {
    if (prefix_sub(d) == 1) return L == 16 ? k_prefix_scan<16, 128, 1> : k_prefix_scan<32, 128, 1>;
    if (prefix_wide(d)) return L == 16 ? k_prefix_scan<16, 192, 2> : k_prefix_scan<32, 192, 2>;
    return L == 16 ? k_prefix_scan<16, 128, 2> : k_prefix_scan<32, 128, 2>;
}

cudaError_t prepare_rank_prefix(int64_t nq, int64_t nlist, int nprobe, int W, int d) {
    const int L = rank_prefix_len(nq, nlist, nprobe, W, d);
    return cudaFuncSetAttribute(scan_kernel(d, L), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)scan_smem(d));
}

template <int kL, int KPL>
static void launch_prefix_final(const PrefixArgs &a, const float *C, int nprobe, const unsigned *cmax, int32_t *order, float *cscores, int *limit, cudaStream_t st) {
    const unsigned blocks = (unsigned)ceil_div(a.nq, kFinalWarps);
    auto f = a.d <= 128   ? k_prefix_final<kL, KPL, 1>
             : a.d <= 256 ? k_prefix_final<kL, KPL, 2>
                          : k_prefix_final<kL, KPL, 4>;
    f<<<blocks, kFinalWarps * 32, 0, st>>>(a.Q, a.nq, C, a.nlist, a.d, a.list_s, a.list_g, a.list_t, a.nranges, nprobe,
                                           cmax, a.status, order, cscores, limit);
}

// kernel launches of the prefix ranking of nq queries from q0 on (and its
// contraction launches), for scratch sized for plan_nq
int rank_prefix_launches(int64_t q0, int64_t nq, int64_t plan_nq, int64_t nlist, int nprobe, int W, int d, int *mma) {
    const int L = rank_prefix_len(plan_nq, nlist, nprobe, W, d);
    const PrefixScratch S = prefix_scratch(plan_nq, nlist, nprobe, d, L);
    const int chunks = (int)ceil_div(nq, S.chunk);
    *mma = chunks;
    return 2 * chunks + (q0 > 0 ? 0 : prefix_sub(d) == 1 ? 2 : 1);
}

// The prefix of nq queries q0 .. q0 + nq - 1 of a batch of plan_nq (whose
// scratch this is): order, cscores (nullable) and the scratch's limits.  The
// largest norm and the wide rows' layout are made with the first part (q0 = 0)
// and stay in the scratch for the others, which follow it on the same stream.
cudaError_t enqueue_rank_prefix(const float *Q, int64_t q0, int64_t nq, int64_t plan_nq, const float *C,
                                int64_t nlist, int d, int nprobe, int W, int32_t *order, float *cscores,
                                void *scratch, int *status, const unsigned char *tc_cent, cudaStream_t st,
                                float *mma_ms, int wait_limit) {
    if (nq <= 0) return cudaSuccess;
    const int L = rank_prefix_len(plan_nq, nlist, nprobe, W, d);
    const PrefixScratch S = prefix_scratch(plan_nq, nlist, nprobe, d, L);
    const PrefixPlan P = prefix_plan(plan_nq, nlist, d, L);
    unsigned char *w = static_cast<unsigned char *>(scratch);
    int *limit = reinterpret_cast<int *>(w + S.limit);
    unsigned *cmax = reinterpret_cast<unsigned *>(w + S.rest);
    float *list_s = reinterpret_cast<float *>(w + S.lists);
    const int64_t slots = S.chunk * P.nranges * L;
    int2 *list_g = reinterpret_cast<int2 *>(list_s + slots * 32);
    float2 *list_t = reinterpret_cast<float2 *>(list_g + slots);
    const int stages = prefix_stages(d);
    const size_t smem = scan_smem(d);
    const PrefixScan scan = scan_kernel(d, L);
    struct Events {
        std::vector<cudaEvent_t> v;
        ~Events() {
            for (cudaEvent_t e : v) cudaEventDestroy(e);
        }
    } ev;
    cudaError_t e = q0 == 0 ? launch_cnorm_max(C, nlist, d, cmax, st) : cudaSuccess;
    if (e != cudaSuccess) return e;
    if (prefix_sub(d) == 1) {
        tc_cent = w + S.fill;
        if (q0 == 0) {
            const int64_t pieces = ceil_div(nlist, kTcRows) * ceil_div(d, 64) * kTcRows * 8;
            k_prefix_fill<<<(unsigned)std::min<int64_t>(ceil_div(pieces, 256), 16 * num_sms()), 256, 0, st>>>(
                C, nlist, d, (int)ceil_div(d, 64), w + S.fill);
        }
    }
    for (int64_t b = 0; b < nq; b += S.chunk) {
        const int64_t n = std::min(S.chunk, nq - b);
        const PrefixArgs a{Q + (q0 + b) * d, n, nlist, d, status, wait_limit, tc_cent, P.nranges, P.range_len,
                           list_s, list_g, list_t};
        const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(n, prefix_sub(d) * tcp::kM) * P.nranges, num_sms());
        if (mma_ms) {
            ev.v.resize(ev.v.size() + 2);
            cudaEventCreate(&ev.v[ev.v.size() - 2]);
            cudaEventCreate(&ev.v.back());
            cudaEventRecord(ev.v[ev.v.size() - 2], st);
        }
        scan<<<grid, tcb::kThreads, smem, st>>>(a, stages);
        if (mma_ms) cudaEventRecord(ev.v.back(), st);
        int32_t *o = order + (q0 + b) * nprobe;
        float *cs = cscores ? cscores + (q0 + b) * nprobe : nullptr;
        int *lim = limit + q0 + b;
        const int kpl = (int)ceil_div(P.nranges * L, 32);
#define SIEVE_PREFIX(K)                                                                       \
    if (L == 16) launch_prefix_final<16, K>(a, C, nprobe, cmax, o, cs, lim, st);               \
    else launch_prefix_final<32, K>(a, C, nprobe, cmax, o, cs, lim, st)
        if (kpl <= 1) { SIEVE_PREFIX(1); }
        else if (kpl <= 2) { SIEVE_PREFIX(2); }
        else if (kpl <= 4) { SIEVE_PREFIX(4); }
        else if (kpl <= 8) { SIEVE_PREFIX(8); }
        else if (kpl <= 16) { SIEVE_PREFIX(16); }
        else { SIEVE_PREFIX(32); }
#undef SIEVE_PREFIX
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (mma_ms) {
        e = cudaStreamSynchronize(st);
        for (size_t i = 0; i + 1 < ev.v.size(); i += 2) {
            float t = 0.f;
            if (e == cudaSuccess) e = cudaEventElapsedTime(&t, ev.v[i], ev.v[i + 1]);
            *mma_ms += t;
        }
    }
    return e;
}

// The extension: the full ranking of the queries ext[0 .. *ext_n - 1], behind
// their prefixes, those of one part.  Every pass is launched; passes past
// *ext_n find no work.
cudaError_t enqueue_rank_ext(int part, const float *Q, int64_t nq, const float *C, int64_t nlist, int d,
                             int nprobe, int W, int32_t *order, float *cscores, void *scratch,
                             Ctl *ctl, const unsigned char *tc_cent, cudaStream_t st, float *mma_ms) {
    const PrefixScratch S = prefix_scratch(nq, nlist, nprobe, d, rank_prefix_len(nq, nlist, nprobe, W, d));
    const PrefixScratch::Ext &E = S.ext_part[part];
    unsigned char *w = static_cast<unsigned char *>(scratch);
    int *limit = reinterpret_cast<int *>(w + S.limit);
    const int *ext = reinterpret_cast<const int *>(w + S.ext);
    float *Qx = reinterpret_cast<float *>(w + E.q);
    int32_t *full = reinterpret_cast<int32_t *>(w + E.order);
    float *full_s = cscores ? reinterpret_cast<float *>(w + E.s) : nullptr;
    const int blocks = 4 * num_sms();
    const int64_t hi = ext_end(part, nq);
    for (int64_t b = ext_begin(part); b < hi; b += E.chunk) {
        const int64_t n = std::min(E.chunk, hi - b);
        k_ext_gather<<<blocks, 256, 0, st>>>(Q, d, ext, ctl, b, n, Qx, b == ext_begin(part) ? part : -1);
        cudaError_t e = enqueue_rank_tc(Qx, n, C, nlist, d, nprobe, full, full_s,
                                        reinterpret_cast<float *>(w + S.rest), &ctl->status, st, tc_cent, mma_ms,
                                        E.chunk, &ctl->ext_n, b);
        if (e != cudaSuccess) return e;
        k_ext_merge<<<blocks, 256, 0, st>>>(ext, &ctl->ext_n, b, n, nprobe, full, full_s, order, cscores, limit);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int rank_ext_launches(int part, int64_t nq, int64_t nlist, int nprobe, int W, int d, bool bulk, int *mma) {
    const PrefixScratch S = prefix_scratch(nq, nlist, nprobe, d, rank_prefix_len(nq, nlist, nprobe, W, d));
    const int64_t chunk = S.ext_part[part].chunk;
    int n = 0;
    *mma = 0;
    for (int64_t b = ext_begin(part), hi = ext_end(part, nq); b < hi; b += chunk) {
        const int64_t m = std::min(chunk, hi - b);
        n += 2 + rank_tc_launches(m, nlist, nprobe, d, chunk, bulk);
        *mma += rank_tc_mma_launches(m, nlist, nprobe, d, chunk, bulk);
    }
    return n;
}

}  // namespace sieve
