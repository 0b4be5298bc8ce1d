// Search-by-triplet reconstruction kernels for sm_103a.
//
// Events map to thread blocks, hits and forming tracks to threads (Table 1
// of the paper).  Two kernels per event:
//   1. k_sort: phi16 of every hit and its order by (module, phi16, input
//      index) from one counting pass into (module, coarse phi) buckets and a
//      count inside each bucket, in shared memory (section "Sort by phi"); the
//      sorted hits are written as AoS records (x, y, z, phi16 and input
//      index: float4, or fp16 x, y, z and phi16 with the index beside), with
//      the start of every bucket;
//   2. k_search_*: for every module triplet (s, s+1, s+2): seeding over the unflagged
//      middle hits, then following of every forming track to module s+3 with
//      one-round claims on the hits, flags, and termination after two misses
//      (section "Track seeding and track following"); barriers separate the
//      stages as the paper's flagged-hits dependency requires;
//      then the tracklet filter (section "Tracklet filter") and staging of
//      every track's hit records with its smallest input hit index.
// A device-wide scan and the output kernel then build the CSR output (section
// "Results", data consolidation): canonical ordering of each event's tracks
// by smallest input hit index, their hit lists and the least-squares fit of
// every track, outside the latency-bound search blocks.
//
// Decision arithmetic is fp32 with every operation rounded as written
// (explicit _rn intrinsics, no contraction), so that the result is the
// exact track set of the plain definition.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdint>

#include "sbt_internal.h"

namespace sbt {

constexpr uint16_t kNone = 0xFFFFu;
constexpr uint16_t kDead = 0xFFFEu;

// ------------------------------------------------------------------ phi ---

// 2-argument arctangent: octant reduction and the degree-9 odd polynomial of
// the Hastings form (Abramowitz & Stegun 4.4.49), every operation rounded.
__device__ __forceinline__ float atan2_sbt(float y, float x)
{
    const float a1 = 0.9998660f, a3 = -0.3302995f, a5 = 0.1801410f;
    const float a7 = -0.0851330f, a9 = 0.0208351f;
    float ax = fabsf(x);
    float ay = fabsf(y);
    float mx = ax > ay ? ax : ay;
    float mn = ax > ay ? ay : ax;
    if (mx == 0.0f) return 0.0f;
    float t = __fdiv_rn(mn, mx);
    float t2 = __fmul_rn(t, t);
    float p = a9;
    p = __fadd_rn(__fmul_rn(p, t2), a7);
    p = __fadd_rn(__fmul_rn(p, t2), a5);
    p = __fadd_rn(__fmul_rn(p, t2), a3);
    p = __fadd_rn(__fmul_rn(p, t2), a1);
    p = __fmul_rn(p, t);
    if (ay > ax) p = __fsub_rn(1.5707963267948966f, p);
    if (x < 0.0f) p = __fsub_rn(3.14159265358979323846f, p);
    if (y < 0.0f) p = -p;
    return p;
}

// [-pi, pi] onto the unsigned 16-bit range, modulo 2^16.
__device__ __forceinline__ uint32_t phi16_of(float x, float y)
{
    float a = atan2_sbt(y, x);
    int q = __float2int_rn(__fmul_rn(a, 10430.378350470453f));
    return (uint32_t)q & 0xFFFFu;
}

__device__ __forceinline__ int phi_dist(uint32_t u, uint32_t v)
{
    int d1 = (int)((u - v) & 0xFFFFu);
    int d2 = (int)((v - u) & 0xFFFFu);
    return d1 < d2 ? d1 : d2;
}

__device__ __forceinline__ float3 sub_rn(float4 a, float4 b)
{
    return make_float3(__fsub_rn(a.x, b.x), __fsub_rn(a.y, b.y), __fsub_rn(a.z, b.z));
}

// Straight-line extrapolation to the plane z = zt from the last hit c and its
// difference d from the hit before it.
__device__ __forceinline__ void extrapolate(float3 c, float3 d, float zt, float& xp, float& yp)
{
    float tz = __fdiv_rn(__fsub_rn(zt, c.z), d.z);
    xp = __fadd_rn(c.x, __fmul_rn(d.x, tz));
    yp = __fadd_rn(c.y, __fmul_rn(d.y, tz));
}

__device__ __forceinline__ float scatter_of(float4 B, float xp, float yp)
{
    float dx = __fsub_rn(B.x, xp);
    float dy = __fsub_rn(B.y, yp);
    return __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
}

// Least-squares straight line through n hits (get(i) -> float3 in hit
// order): chi2 = residual sum / sigma^2.
template <class Get>
__device__ __forceinline__ float fit_chi2(int n, Get get, float sigma)
{
    float nf = (float)n;
    float sx = 0.0f, sy = 0.0f, sz = 0.0f;
    for (int i = 0; i < n; i++) {
        float3 h = get(i);
        sx = __fadd_rn(sx, h.x);
        sy = __fadd_rn(sy, h.y);
        sz = __fadd_rn(sz, h.z);
    }
    float xm = __fdiv_rn(sx, nf), ym = __fdiv_rn(sy, nf), zm = __fdiv_rn(sz, nf);
    float szz = 0.0f, szx = 0.0f, szy = 0.0f;
    for (int i = 0; i < n; i++) {
        float3 h = get(i);
        float dz = __fsub_rn(h.z, zm);
        szz = __fadd_rn(szz, __fmul_rn(dz, dz));
        szx = __fadd_rn(szx, __fmul_rn(dz, __fsub_rn(h.x, xm)));
        szy = __fadd_rn(szy, __fmul_rn(dz, __fsub_rn(h.y, ym)));
    }
    float tx = __fdiv_rn(szx, szz);
    float ty = __fdiv_rn(szy, szz);
    float s = 0.0f;
    for (int i = 0; i < n; i++) {
        float3 h = get(i);
        float dz = __fsub_rn(h.z, zm);
        float rx = __fsub_rn(__fsub_rn(h.x, xm), __fmul_rn(tx, dz));
        float ry = __fsub_rn(__fsub_rn(h.y, ym), __fmul_rn(ty, dz));
        s = __fadd_rn(s, __fadd_rn(__fmul_rn(rx, rx), __fmul_rn(ry, ry)));
    }
    return __fdiv_rn(s, __fmul_rn(sigma, sigma));
}

// ------------------------------------------------------- shared layout ---

enum Misc {
    kErr = 0, kNFin = 1, kNTl = 2, kEvent = 3, kCMask = 4, kCnt0 = 5, kCnt1 = 6, kWork = 7, kNew = 8, kList = 9,
    kNOuter = 10, kShift = 11, kMiscN = 12
};
static_assert(kMiscN % 2 == 0, "a pointer follows");

// Per-block shared memory of the search: flag bits, module offsets, counters,
// each sized to what the configuration needs.  Everything sized by the event
// lives in global scratch (L1-resident): shared memory and L1 share one array
// per SM, so every byte a block holds here comes out of the L1 of the resident
// events (about n / 8 + 4 M bytes a block).
struct Smem {
    uint32_t* flag;     // one bit per sorted position
    int* modoff;
    int* misc;
    // first sorted position of each (module, phi16 >> misc[kShift]); here and not
    // in registers, which the windows are short of (calls of 16 quiet events 155
    // -> 153 us, 100 events 338 -> 334, 500 events 482 -> 477)
    const uint16_t** table;
    int* wsum;          // [33]
};

__host__ __device__ inline size_t align16(size_t v) { return (v + 15) & ~(size_t)15; }

struct Plan {
    size_t flag, modoff, misc, table, wsum, total;
};

__host__ __device__ inline Plan make_plan(int nmax, int threads, int M)
{
    Plan p;
    size_t o = 0;
    p.flag = o;     o = align16(o + 4 * (((size_t)nmax + 31) / 32));
    p.modoff = o;   o = align16(o + 4 * ((size_t)M + 1));
    p.misc = o;     o = o + 4 * kMiscN;
    p.table = o;    o = align16(o + sizeof(void*));
    p.wsum = o;     o = align16(o + 4 * ((size_t)threads / 32 + 1));
    p.total = o;
    return p;
}

size_t smem_bytes(int nmax, int threads, int M) { return make_plan(nmax, threads, M).total; }

__device__ inline Smem carve(unsigned char* raw, int nmax, int threads, int M)
{
    Plan p = make_plan(nmax, threads, M);
    Smem S;
    S.flag = (uint32_t*)(raw + p.flag);
    S.modoff = (int*)(raw + p.modoff);
    S.misc = (int*)(raw + p.misc);
    S.table = (const uint16_t**)(raw + p.table);
    S.wsum = (int*)(raw + p.wsum);
    return S;
}

__device__ __forceinline__ bool flagged(const Smem& S, int p) { return (S.flag[p >> 5] >> (p & 31)) & 1u; }
__device__ __forceinline__ void set_flag(const Smem& S, int p) { atomicOr(&S.flag[p >> 5], 1u << (p & 31)); }

// Storage of the sorted hits.  HitsF32: float4 (x, y, z, phi16 << 16 | input
// index as int bits), 16 bytes.  HitsF16: x, y, z rounded to fp16 (nearest
// even) and phi16, 8 bytes (the paper's fp16 AoS storage of hit coordinates),
// the input index in an array of its own, which only the output reads; every
// computation still runs in fp32, on the rounded values.  Either way one load
// gives a window scan the key and the position.
struct HitsF32 {
    using T = float4;
    static constexpr bool kIndexArray = false;
    __device__ __forceinline__ static float round(float v) { return v; }
    // w: phi16 << 16 | anything
    __device__ __forceinline__ static float4 load(const T* p, int i) { return p[i]; }
    __device__ __forceinline__ static void store(T* p, int64_t at, float4 c, uint32_t ph, int i)
    {
        c.w = __int_as_float((int)(ph << 16) | i);
        p[at] = c;
    }
    __device__ __forceinline__ static uint32_t phi(const T* p, int i) { return (uint32_t)__float_as_int(p[i].w) >> 16; }
    __device__ __forceinline__ static int index(float4 c, const uint16_t*, int) { return __float_as_int(c.w) & 0xFFFF; }
};

struct HitsF16 {
    using T = ushort4;
    static constexpr bool kIndexArray = true;
    __device__ __forceinline__ static float round(float v) { return __half2float(__float2half_rn(v)); }
    __device__ __forceinline__ static float4 load(const T* p, int i)
    {
        const ushort4 u = p[i];
        return make_float4(__half2float(__ushort_as_half(u.x)), __half2float(__ushort_as_half(u.y)),
                           __half2float(__ushort_as_half(u.z)), __int_as_float((int)((uint32_t)u.w << 16)));
    }
    __device__ __forceinline__ static void store(T* p, int64_t at, float4 c, uint32_t ph, int)
    {
        p[at] = make_ushort4(__half_as_ushort(__float2half_rn(c.x)), __half_as_ushort(__float2half_rn(c.y)),
                             __half_as_ushort(__float2half_rn(c.z)), (unsigned short)ph);
    }
    __device__ __forceinline__ static uint32_t phi(const T* p, int i) { return p[i].w; }
    __device__ __forceinline__ static int index(float4, const uint16_t* idx, int i) { return idx[i]; }
};

// Sorted hits of one event: hit p as float4, its phi16 and its event-local
// input index (below 2^14).
template <class HS>
struct HitArr {
    const typename HS::T* p;
    const uint16_t* idx;
    __device__ __forceinline__ float4 operator[](int i) const { return HS::load(p, i); }
    __device__ __forceinline__ uint32_t phi(int i) const { return HS::phi(p, i); }
    __device__ __forceinline__ int index(float4 c, int i) const { return HS::index(c, idx, i); }
};

// What one event's search sees: its sorted hits (read-only) and its scratch.
template <class HS>
struct Region {
    HitArr<HS> coords;
    uint32_t* list;
    uint16_t* prev;
    unsigned long long* claim;  // the search's claim of sorted position p is claim[p & cmask]
    unsigned cmask;
    unsigned long long* claim_all;  // by sorted position, for the tracklet filter
    unsigned long long* tracklets;
    uint32_t* tl_q;
    int lcap;
    uint32_t* finals;
    FTrack* ft;         // buffer b starts at ft + b * fstride
    int fstride;
};

template <class HS>
__device__ inline Region<HS> region_of(const Sorted& O, int off, const Work& W, int64_t hb, int64_t r, int cap)
{
    Region<HS> R;
    R.coords = HitArr<HS>{(const typename HS::T*)O.coords + off, O.index + off};
    R.list = W.list + hb;
    R.prev = W.prev + hb;
    R.claim_all = W.claim + hb;
    R.claim = R.claim_all;
    R.cmask = ~0u;
    R.tracklets = W.tracklets + hb + r;
    R.tl_q = W.tl_q + hb + r;
    R.lcap = cap + 1;
    R.finals = W.finals + hb / 3 + r;
    R.ft = W.ft + forming_base(hb, r);
    R.fstride = cap / 12 + 72;
    return R;
}

// Exclusive block scan of one int per thread; returns the prefix, *total the
// sum.  wsum needs NT / 32 + 1 entries.
template <int NT>
__device__ __forceinline__ int block_exclusive_scan(int v, int* wsum, int* total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < NT / 32 ? wsum[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int t = __shfl_up_sync(0xFFFFFFFFu, wi, o);
            if (lane >= o) wi += t;
        }
        if (lane < NT / 32) wsum[lane] = wi - w;
        if (lane == NT / 32 - 1) wsum[NT / 32] = wi;
    }
    __syncthreads();
    int res = wsum[warp] + incl - v;
    *total = wsum[NT / 32];
    __syncthreads();
    return res;
}

// ------------------------------------------------------------- sorting ---

constexpr int kSortThreads = 1024;
constexpr int kSortBuckets = kMaxModules << kBucketBits;

// Bucket of a hit on module m: module and the top 16 - shift bits of phi16.
__device__ __forceinline__ int bucket_of(int m, uint32_t phi16, int shift)
{
    return (int)(((uint32_t)m << 16 | phi16) >> shift);
}

// Hits of buckets up to this size count the smaller keys, above it a warp sorts
// the bucket (12 M hits in buckets of 64: 550 us counted, 583 sorted; of 128:
// 634 sorted either way).
constexpr int kShortBucket = 96;

// Shared memory of the sort kernel: the bucketed entries phi16 << 14 | input
// index (4 B per hit), phi16 by input order (2 B per hit), the bucket counters
// (16 bits, an event's hits fit) and the list of long buckets: 115 KB for events
// of 16384 hits, two blocks an SM with 700 B to spare.
__host__ __device__ inline size_t sort_layout(int nmax, size_t* off_phi, size_t* off_cnt, size_t* off_long)
{
    size_t o = align16(4 * (size_t)nmax);
    *off_phi = o;  o = align16(o + 2 * (size_t)nmax);
    *off_cnt = o;  o = align16(o + 2 * (size_t)kSortBuckets);
    *off_long = o; o = align16(o + 2 * (size_t)(nmax / kShortBucket + 1));
    return o;
}

size_t sort_smem_bytes(int nmax)
{
    size_t a, b, c;
    return sort_layout(nmax, &a, &b, &c);
}

// Ascending sort of a[0, s) by one warp, in place: a bitonic network in the
// form whose comparators all put the smaller key first (a mirrored merge
// step, then half-cleaners), so positions past s behave as +infinity and are
// never touched.
__device__ void warp_bitonic(uint32_t* a, int s)
{
    const int lane = threadIdx.x & 31;
    int P = 1;
    while (P < s) P <<= 1;
    for (int k = 2; k <= P; k <<= 1) {
        const int h = k >> 1;
        for (int i = lane; i < P / 2; i += 32) {
            const int lo = (i / h) * k + (i % h), hi = (i / h) * k + k - 1 - (i % h);
            if (hi < s) {
                const uint32_t u = a[lo], v = a[hi];
                if (u > v) {
                    a[lo] = v;
                    a[hi] = u;
                }
            }
        }
        __syncwarp();
        for (int j = k >> 2; j >= 1; j >>= 1) {
            for (int i = lane; i < P / 2; i += 32) {
                const int lo = (i / j) * 2 * j + (i % j), hi = lo + j;
                if (hi < s) {
                    const uint32_t u = a[lo], v = a[hi];
                    if (u > v) {
                        a[lo] = v;
                        a[hi] = u;
                    }
                }
            }
            __syncwarp();
        }
    }
}

// One block per event: phi16, stable sort by (module, phi16) in shared
// memory, gather of the sorted hits.  A counting pass puts every hit into its
// (module, top bits of phi16) bucket; within it, a hit's place is the number
// of smaller keys phi16 << 14 | input index (unique, so the order is the one
// of a stable sort by (module, phi16)), counted by the hit's own thread: a
// bucket holds about one hit, and nothing has to be moved once the place is
// known (moving entries into order bucket by bucket and inverting the order
// took two more passes: 92 M hits 1280 -> 1190 us).  Long buckets are sorted by
// a warp each, and their hits look their place up.  Status SBT_ERR_ARG for a module id out of
// range or a hit range [offsets[e], offsets[e+1]) that is not inside
// [0, n_hits) (no later kernel reads or writes anything of such an event),
// SBT_ERR_CAPACITY above the configured hit limit.
template <class HS>
__global__ void __launch_bounds__(kSortThreads, 2) k_sort(DevConfig C, Inputs in, Sorted O)
{
    constexpr int NT = kSortThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    size_t ophi, ocnt, olong;
    sort_layout(C.nmax, &ophi, &ocnt, &olong);
    uint32_t* ent = (uint32_t*)smem_raw;
    uint16_t* phi = (uint16_t*)(smem_raw + ophi);
    uint16_t* cnt = (uint16_t*)(smem_raw + ocnt);
    uint32_t* cntw = (uint32_t*)cnt;  // two counters a word
    uint16_t* longb = (uint16_t*)(smem_raw + olong);
    __shared__ int wsum[40];
    __shared__ int err, nlong;
    const int tid = threadIdx.x;
    const int e = blockIdx.x;
    const int off = in.offsets[e];
    const int64_t n64 = (int64_t)in.offsets[e + 1] - off;
    const bool range_bad = off < 0 || n64 < 0 || off + n64 > in.n_hits;
    if (range_bad || n64 > C.nmax || (C.gec > 0 && n64 > C.gec)) {
        if (tid == 0)
            O.status[e] = range_bad ? SBT_ERR_ARG : (C.gec > 0 && n64 > C.gec) ? SBT_EVENT_CUT : SBT_ERR_CAPACITY;
        return;
    }
    const int n = (int)n64;
    const int shift = 16 - bucket_bits(O.tables, n, C.M);
    const int nb = C.M << (16 - shift);
    for (int w = tid; w < (nb + 7) / 8; w += NT) ((uint4*)cnt)[w] = make_uint4(0u, 0u, 0u, 0u);
    if (tid == 0) {
        err = 0;
        nlong = 0;
    }
    __syncthreads();
    // phi16 and bucket counts, two hits per thread per round (loads first)
    for (int i0 = tid; i0 < n; i0 += 2 * NT) {
        float xs[2], ys[2];
        int ms[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int i = i0 + u * NT;
            const bool v = i < n;
            xs[u] = v ? in.x[off + i] : 1.0f;
            ys[u] = v ? in.y[off + i] : 0.0f;
            ms[u] = v ? in.module[off + i] : 0;
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int i = i0 + u * NT;
            if (i >= n) continue;
            int m = ms[u];
            if (m < 0 || m >= C.M) {
                err = SBT_ERR_ARG;
                m = 0;
            }
            const uint32_t ph = phi16_of(HS::round(xs[u]), HS::round(ys[u]));
            phi[i] = (uint16_t)ph;
            const int b = bucket_of(m, ph, shift);
            atomicAdd(&cntw[b >> 1], 1u << (16 * (b & 1)));
        }
    }
    __syncthreads();
    if (err) {
        if (tid == 0) O.status[e] = SBT_ERR_ARG;
        return;
    }
    // bucket starts: exclusive scan, eight consecutive buckets per thread; the
    // search's table of starts, and the long buckets
    {
        static_assert(kSortBuckets <= 8 * NT, "one 16-byte word of counters a thread");
        uint4* mine = (uint4*)cnt + tid;
        const bool any = 8 * tid < nb;
        uint32_t w[4] = {0u, 0u, 0u, 0u};
        if (any) {
            const uint4 v = *mine;
            w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
        }
        int s = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) s += (int)(w[q] & 0xFFFFu) + (int)(w[q] >> 16);
        int total;
        int st = block_exclusive_scan<NT>(s, wsum, &total);
        if (any) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int c0 = (int)(w[q] & 0xFFFFu), c1 = (int)(w[q] >> 16);
                const int b = 8 * tid + 2 * q;
                if (c0 > kShortBucket) longb[atomicAdd(&nlong, 1)] = (uint16_t)b;
                if (c1 > kShortBucket) longb[atomicAdd(&nlong, 1)] = (uint16_t)(b + 1);
                w[q] = (uint32_t)st | ((uint32_t)(st + c0) << 16);
                st += c0 + c1;
            }
            *mine = make_uint4(w[0], w[1], w[2], w[3]);
            ((uint4*)(O.bucket + table_base(O.tables, off, e)))[tid] = *mine;
        }
    }
    __syncthreads();
    // scatter into the buckets (order inside a bucket arbitrary); afterwards
    // cnt[b] is the end of bucket b
    for (int i = tid; i < n; i += NT) {
        const uint32_t ph = phi[i];
        const int b = bucket_of(in.module[off + i], ph, shift);
        const int half = 16 * (b & 1);
        const int p = (int)(atomicAdd(&cntw[b >> 1], 1u << half) >> half) & 0xFFFF;
        ent[p] = (ph << 14) | (uint32_t)i;
    }
    __syncthreads();
    if (tid <= C.M) O.modoff[(int64_t)e * (C.M + 1) + tid] = tid > 0 ? cnt[(tid << (16 - shift)) - 1] : 0;
    if (nlong > 0) {
        for (int q = tid >> 5; q < nlong; q += NT / 32) {
            const int b = longb[q];
            const int lo = b > 0 ? cnt[b - 1] : 0;
            warp_bitonic(ent + lo, cnt[b] - lo);
        }
        __syncthreads();
    }
    // the hits in input order (coalesced loads), each stored at its place; two
    // per thread per round
    for (int i0 = tid; i0 < n; i0 += 2 * NT) {
        float4 c[2];
        int m[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int i = i0 + u * NT;
            if (i < n) {
                m[u] = in.module[off + i];
                c[u] = make_float4(in.x[off + i], in.y[off + i], in.z[off + i], 0.0f);
            }
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int i = i0 + u * NT;
            if (i >= n) continue;
            const uint32_t ph = phi[i], own = (ph << 14) | (uint32_t)i;
            const int b = bucket_of(m[u], ph, shift);
            int lo = b > 0 ? cnt[b - 1] : 0;
            const int hi = cnt[b];
            int q = lo;
            if (hi - lo <= kShortBucket) {
                for (int k = lo; k < hi; k++) q += ent[k] < own;
            } else {
                for (int end = hi; q < end;) {
                    const int mid = (q + end) >> 1;
                    if (ent[mid] < own)
                        q = mid + 1;
                    else
                        end = mid;
                }
            }
            HS::store((typename HS::T*)O.coords, (int64_t)off + q, c[u], ph, i);
            if (HS::kIndexArray) phi[i] = (uint16_t)q;  // read by this thread alone
        }
    }
    if (HS::kIndexArray) {
        // the input indices by place, through the space of the entries, so that
        // they leave coalesced (scattered 2-byte stores: sort of 35 M hits 475 us)
        uint16_t* idx = (uint16_t*)ent;
        __syncthreads();
        for (int i = tid; i < n; i += NT) idx[phi[i]] = (uint16_t)i;
        __syncthreads();
        for (int p = tid; p < n; p += NT) O.index[off + p] = idx[p];
    }
    if (tid == 0) O.status[e] = SBT_OK;
}

// ------------------------------------------------------ seeding, following ---

// phi16 of a window centre.  Only the window bounds use it, and they carry a
// margin of 16 units, so a fast division is enough here.
__device__ __forceinline__ uint32_t phi16_window(float x, float y)
{
    const float a1 = 0.9998660f, a3 = -0.3302995f, a5 = 0.1801410f;
    const float a7 = -0.0851330f, a9 = 0.0208351f;
    float ax = fabsf(x), ay = fabsf(y);
    float mx = fmaxf(ax, ay), mn = fminf(ax, ay);
    const float t = mx > 0.0f ? __fdividef(mn, mx) : 0.0f;
    const float t2 = t * t;
    float p = __fmaf_rn(__fmaf_rn(__fmaf_rn(__fmaf_rn(a9, t2, a7), t2, a5), t2, a3), t2, a1) * t;
    if (ay > ax) p = 1.5707963f - p;
    if (x < 0.0f) p = 3.1415927f - p;
    if (y < 0.0f) p = -p;
    return (uint32_t)__float2int_rn(p * 10430.378f) & 0xFFFFu;
}

// Phi window of a prediction (xp, yp) for a scatter cut: hits outside it
// cannot pass the cut.  A hit within d = sqrt(cut) of the prediction differs
// from it in angle by at most asin(d / r) <= d / sqrt(r^2 - d^2); the
// half-width adds 1/16 of that plus 16 phi16 units for the rounding and
// arctangent error of both phi values and for the approximate arithmetic of
// the bound itself.  Predictions near the axis (r <= 2 d) get no window (the
// whole module is scanned).
__device__ __forceinline__ bool window_of(float xp, float yp, float cut, float sqrt_cut, uint32_t& lo,
                                          uint32_t& width)
{
    const float rp2 = __fmaf_rn(xp, xp, yp * yp);
    if (rp2 < 1.0e30f && rp2 > 4.0f * cut) {
        const float wf = sqrt_cut * rsqrtf(rp2 - cut) * (10430.378f * 1.0625f);
        if (wf < 16000.0f) {
            const uint32_t W = (uint32_t)wf + 16u;
            lo = (phi16_window(xp, yp) - W) & 0xFFFFu;
            width = 2u * W;
            return true;
        }
    }
    lo = 0;
    width = 0xFFFFu;
    return false;
}

// Geometry of the module an extrapolation targets.  PlaneGeo: one plane at
// module_z[m].  PairGeo: a module pair of one-sided planes (the paper's
// method works on module pairs, the two sides of the VELO), hits with
// x >= 0 on the plane at module_z[m] and hits with x < 0 on the plane at
// module_z2[m]; a search visits each plane's hits with the prediction at
// that plane's z, so every candidate is compared at its own plane.
struct PlaneGeo {
    static constexpr int kPlanes = 1;
    __device__ __forceinline__ static float z(const DevConfig& C, int m, int) { return C.module_z[m]; }
    __device__ __forceinline__ static bool on(int, float) { return true; }
};

struct PairGeo {
    static constexpr int kPlanes = 2;
    __device__ __forceinline__ static float z(const DevConfig& C, int m, int p)
    {
        return p ? C.module_z2[m] : C.module_z[m];
    }
    __device__ __forceinline__ static bool on(int p, float x) { return (x < 0.0f) == (p != 0); }
};

// No hit yet: above every (scatter, positions) key.
constexpr unsigned long long kNoHit = ~0ull;

// A straight line (last hit c0, difference d0) extrapolated to module t: the
// least (scatter, position) over the module's unflagged hits under the scatter
// cut; returns scatter bits << 32 | hi << 16 | position, or kNoHit.  Only the
// hits from the bucket that holds the window's lower edge up to its upper edge
// are visited: the bucket table replaces a binary search (seven dependent
// loads a window of a 112-hit module), and hits before the edge in its bucket
// cannot pass the cut, so looking at them changes nothing.  The search is
// bound by the instructions of its longest lane (windows hold 2 to 3 hits on
// average, the longest of a warp about ten), so the loop tests one key, the
// scatter and the end; what concerns the few hits under the best scatter so
// far stands in the branch.  kAhead: each round loads the next hit too (blocks
// of 512, which have the registers: one event 212 -> 206 us; at 32 registers
// it spills).
template <bool kAhead, class G, class HS>
__device__ __forceinline__ unsigned long long best_hit(const DevConfig& C, const Smem& S, const Region<HS>& R,
                                                       int t, float3 c0, float3 d0, float cut, float sqrt_cut,
                                                       uint32_t hi)
{
    const int b0 = S.modoff[t], b1 = S.modoff[t + 1];
    float best = cut;
    int bb = INT_MAX;
    if (b0 < b1) {
        for (int plane = 0; plane < G::kPlanes; plane++) {
            float xp, yp;
            extrapolate(c0, d0, G::z(C, t, plane), xp, yp);
            uint32_t lo, width;
            int b = b0;
            // keys compared as phi16 << 16 | low bits; without a window every hit is inside
            if (window_of(xp, yp, cut, sqrt_cut, lo, width)) {
                const int shift = S.misc[kShift];
                const uint32_t k = (uint32_t)bucket_of(t, lo, shift);
                b = max((*S.table)[k], b0);
                b = b < b1 ? b : b0;
                const uint32_t edge = k << shift << 16;  // the bucket's, above the low bits
                width = ((width + lo) << 16 | 0xFFFFu) - edge;
                lo = edge;
            } else {
                width = ~0u;
            }
            const int end = b;
            auto test = [&](float4 c, int p) {
                const float sc = scatter_of(c, xp, yp);
                if (sc <= best && sc < cut && (sc < best || p < bb) && G::on(plane, c.x) && !flagged(S, p)) {
                    best = sc;
                    bb = p;
                }
            };
            auto outside = [&](float4 c) { return (uint32_t)__float_as_int(c.w) - lo > width; };
            do {
                const float4 c = R.coords[b];
                const int next = b + 1 < b1 ? b + 1 : b0;
                float4 d;
                if (kAhead) d = R.coords[next];
                if (outside(c)) break;
                test(c, b);
                b = next;
                if (kAhead) {
                    if (next == end || outside(d)) break;
                    test(d, next);
                    b = next + 1 < b1 ? next + 1 : b0;
                }
            } while (b != end);
        }
    }
    return bb == INT_MAX ? kNoHit
                         : ((unsigned long long)__float_as_uint(best) << 32) |
                               (unsigned long long)((hi << 16) | (uint32_t)bb);
}

// First index in keys[0, n) whose upper 16 bits are >= v.
__device__ __forceinline__ int lower_bound_hi16(const uint32_t* keys, int n, uint32_t v)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if ((keys[mid] >> 16) < v)
            lo = mid + 1;
        else
            hi = mid;
    }
    return lo;
}

// Lanes that share one middle hit in seeding: each takes one of its
// candidates, so K = 4 (the default) needs one round of extrapolations.  One
// lane per middle hit used 8 to 11 lanes of a warp (the unflagged hits of a
// module) for four extrapolations and scans in a row, the longest chain of a
// step.  With the bucket table, search alone: one event 393 -> 266 us (128
// threads), 16000 uneven events 6.22 -> 5.40 ms, 6000 module-pair events
// 1.66 -> 1.12 ms.
constexpr int kSeedLanes = 4;
constexpr int kSeedGroups = 32 / kSeedLanes;

// Seeding for middle hit c on module s+1 (c < 0: none; phi16 phc) by kSeedLanes lanes:
// the unflagged hits of module s nearest to c in phi (all hits at the K-th
// smallest distance included), each extrapolated through c to module s+2,
// where the unflagged hit of least scatter under the cut is sought; the kept
// triplet minimises (scatter, position of a, position of b).  `outer` lists
// the unflagged hits of module s in sorted order as (phi16 << 16 | position),
// `nu` of them, so the nearest-first walk visits no flagged hit; the lanes
// walk together and take the candidates in turn.  Every lane of the group
// returns the triplet as scatter bits << 32 | a << 16 | b, or kNoHit.
template <bool kAhead, class G, class HS>
__device__ __forceinline__ unsigned long long seed_group(const DevConfig& C, const Smem& S,
                                                         const Region<HS>& R, int s, int c, uint32_t phc,
                                                         const uint32_t* outer, int nu, float sqrt_cut)
{
    unsigned long long best = kNoHit;
    if (c >= 0) {
        const int q = threadIdx.x & (kSeedLanes - 1);
        int up = lower_bound_hi16(outer, nu, phc);
        int dn = up - 1;
        if (up == nu) up = 0;
        if (dn < 0) dn = nu - 1;
        uint32_t ku = outer[up], kd = outer[dn];
        int found = 0, dK = INT_MAX;
        bool more = true;
        while (more) {
            int a = -1;
            for (int r = 0; r < kSeedLanes; r++) {
                const int du = phi_dist(ku >> 16, phc), dd = phi_dist(kd >> 16, phc);
                const bool take_up = du < dd || (du == dd && up <= dn);
                const int d = take_up ? du : dd;
                more = found < C.K || d <= dK;
                if (!more) break;
                if (++found == C.K) dK = d;
                if (r == q) a = (int)((take_up ? ku : kd) & 0xFFFFu);
                more = up != dn;  // else that was the last unflagged hit of the module
                if (!more) break;
                if (take_up) {
                    up = up + 1 < nu ? up + 1 : 0;
                    ku = outer[up];
                } else {
                    dn = dn > 0 ? dn - 1 : nu - 1;
                    kd = outer[dn];
                }
            }
            if (a >= 0) {
                const float4 Cc = R.coords[c];
                const unsigned long long v = best_hit<kAhead, G>(C, S, R, s + 2, make_float3(Cc.x, Cc.y, Cc.z),
                                                         sub_rn(Cc, R.coords[a]), C.S_seed, sqrt_cut, (uint32_t)a);
                best = v < best ? v : best;
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int o = 1; o < kSeedLanes; o <<= 1) {
        const unsigned long long v = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        best = v < best ? v : best;
    }
    return best;
}

__device__ __forceinline__ unsigned long long claim_key(unsigned long long tag, float score, int key)
{
    return tag | ((unsigned long long)__float_as_uint(score) << 16) | (unsigned long long)key;
}

template <class HS>
__device__ __forceinline__ void add_final(const Smem& S, const Region<HS>& R, int last, int nh)
{
    int k = atomicAdd(&S.misc[kNFin], 1);
    R.finals[k] = (uint32_t)last | ((uint32_t)nh << 16);
}

template <class HS>
__device__ __forceinline__ void add_tracklet(const Smem& S, const Region<HS>& R, int h0, int h1, int h2,
                                             int key)
{
    int k = atomicAdd(&S.misc[kNTl], 1);
    if (k < R.lcap)
        R.tracklets[k] = (unsigned long long)h0 | ((unsigned long long)h1 << 16) |
                         ((unsigned long long)h2 << 32) | ((unsigned long long)key << 48);
    else
        S.misc[kErr] = SBT_ERR_CAPACITY;
}

__device__ __forceinline__ FTrack make_track(int h0, int h1, int h2, int key, int nh, int sk)
{
    FTrack T;
    T.h0 = (uint16_t)h0;
    T.h1 = (uint16_t)h1;
    T.h2 = (uint16_t)h2;
    T.key = (uint16_t)key;
    T.nh = (uint8_t)nh;
    T.sk = (uint8_t)sk;
    T.cand = kNone;
    T.sc = 0.0f;
    return T;
}

// Following search of one forming track to module t and its claims: the new
// hit, and for a 3-hit track also its three hits.  A 3-hit track with a
// flagged hit cannot extend any more and is marked dead.
template <bool kAhead, class G, class HS>
__device__ __forceinline__ void follow_and_claim(const DevConfig& C, const Smem& S, const Region<HS>& R,
                                                 int t, unsigned long long tag, float sqrt_cut,
                                                 FTrack& T)
{
    if (T.nh == 3 && (flagged(S, T.h0) || flagged(S, T.h1) || flagged(S, T.h2))) {
        T.cand = kDead;
        return;
    }
    const float4 L = R.coords[T.h2];
    const unsigned long long best = best_hit<kAhead, G>(C, S, R, t, make_float3(L.x, L.y, L.z), sub_rn(L, R.coords[T.h1]),
                                                C.S_follow, sqrt_cut, 0u);
    if (best != kNoHit) {
        const int b = (int)(best & 0xFFFFu);
        T.cand = (uint16_t)b;
        T.sc = __uint_as_float((uint32_t)(best >> 32));
        const unsigned long long k = claim_key(tag, T.sc, T.key);
        atomicMin(&R.claim[b & R.cmask], k);
        if (T.nh == 3) {
            atomicMin(&R.claim[T.h0 & R.cmask], k);
            atomicMin(&R.claim[T.h1 & R.cmask], k);
            atomicMin(&R.claim[T.h2 & R.cmask], k);
        }
    } else {
        T.cand = kNone;
        T.sc = 0.0f;
    }
}

// Iterative seeding and following.  Returns false (uniformly) on overflow.
// Per module triplet (s, s+1, s+2) three phases separated by barriers:
//   P0  work lists: unflagged middle hits of s+1, unflagged hits of s in order,
//       both as phi16 << 16 | position; the last warp walks module s alone (it
//       holds the barrier), the others share module s+1;
//   P1  seeding, kSeedLanes lanes per middle hit, and following of the forming
//       tracks to t = s+3 with claims: a warp keeps its new seeds in its lanes
//       and fills the other lanes with old tracks from a shared counter, so
//       its following rounds are dense; it leaves after the round that found
//       the counter used up (an empty round costs a few hundred clocks);
//   P2  resolution of the claims, flags, termination.
// Claims carry a tag (64 - t) << 48 above (scatter bits, track key), so a
// claim of an earlier step always compares larger than one of the current
// step and the claim words need no reset between steps.
template <int NT, class G, class HS>
__device__ bool search_stage(const DevConfig& C, const Region<HS>& R, const Smem& S, int n)
{
    const int tid = threadIdx.x, lane = tid & 31;
    const int M = C.M;
    int* misc = S.misc;
    const int cap = C.fcap > 0 ? min(C.fcap, forming_capacity(n)) : forming_capacity(n);
    const float sq_seed = sqrtf(C.S_seed), sq_follow = sqrtf(C.S_follow);
    constexpr bool kAhead = NT == 512;
    uint32_t* list = R.list;
    int cur = 0;
    for (int s = 0; s + 2 <= M - 1; ++s) {
        const int nxt = cur ^ 1;
        FTrack* Fc = R.ft + cur * R.fstride;
        FTrack* Fn = R.ft + nxt * R.fstride;
        // P0
        if (tid == 0) {
            misc[kCnt0 + nxt] = 0;
            misc[kNew] = 0;
            misc[kWork] = 0;
        }
        const int c0 = S.modoff[s + 1], c1 = S.modoff[s + 2];
        uint32_t* outer = list + (c1 - c0);
        for (int base = c0 + (tid & ~31); base < c1 && (tid >> 5) < NT / 32 - 1; base += NT - 32) {
            const int c = base + lane;
            const bool ok = c < c1 && !flagged(S, c);
            const unsigned m = __ballot_sync(0xFFFFFFFFu, ok);
            int pos = 0;
            if (lane == 0 && m) pos = atomicAdd(&misc[kList], __popc(m));
            pos = __shfl_sync(0xFFFFFFFFu, pos, 0);
            if (ok) list[pos + __popc(m & ((1u << lane) - 1u))] = (R.coords.phi(c) << 16) | (uint32_t)c;
        }
        if ((tid >> 5) == NT / 32 - 1) {
            const int o0 = S.modoff[s], o1 = S.modoff[s + 1];
            int nu = 0;
            for (int base = o0; base < o1; base += 32) {
                const int a = base + lane;
                const bool ok = a < o1 && !flagged(S, a);
                const unsigned m = __ballot_sync(0xFFFFFFFFu, ok);
                if (ok)
                    outer[nu + __popc(m & ((1u << lane) - 1u))] = (R.coords.phi(a) << 16) | (uint32_t)a;
                nu += __popc(m);
            }
            if (lane == 0) misc[kNOuter] = nu;
        }
        __syncthreads();
        const int nu = misc[kNOuter];
        const int nl = nu > 0 && c1 < S.modoff[s + 3] ? misc[kList] : 0;
        const int nold = misc[kCnt0 + cur];
        const int t = s + 3;
        const bool follow = t <= M - 1;
        const unsigned long long tag = (unsigned long long)(64 - t) << 48;
        // P1
        int na = 0, nc = -1, nb = 0;  // this lane's new seed
        int i0 = (tid >> 5) * kSeedGroups, batch = 0;
        // A warp without middle hits is needed only if the old tracks fill the
        // warps before it that have none.  Otherwise its one round finds nothing
        // and still takes the issue slots of the other blocks' warps: search of
        // 200000 events of 20 hits 7.42 -> 6.25 ms, of 5000 events of 686 hits
        // 549 -> 547 us, of 500 events of 4200 hits 408 us either way.
        const int rank = (tid >> 5) - (nl + kSeedGroups - 1) / kSeedGroups;
        while (i0 < nl || (follow && nold > 32 * rank)) {
            if (i0 < nl) {
                const int i = i0 + lane / kSeedLanes;
                const uint32_t mk = i < nl ? list[i] : 0u;
                const int c = i < nl ? (int)(mk & 0xFFFFu) : -1;
                const unsigned long long best = seed_group<kAhead, G>(C, S, R, s, c, mk >> 16, outer, nu, sq_seed);
                if (best != kNoHit && lane % kSeedLanes == batch) {
                    na = (int)(best >> 16) & 0xFFFF;
                    nc = c;
                    nb = (int)best & 0xFFFF;
                }
                i0 += NT / 32 * kSeedGroups;
                // every lane of a group can hold a seed
                if (++batch < kSeedLanes && i0 < nl) continue;
                batch = 0;
            }
            // following: this warp's new seeds, and old tracks in the other
            // lanes; one atomic instruction numbers both
            const unsigned found = __ballot_sync(0xFFFFFFFFu, nc >= 0);
            int base = 0;
            if (lane < 2 && (lane == 0 ? follow : found != 0))
                base = atomicAdd(&misc[kWork + lane], __popc(lane == 0 ? ~found : found));
            const int taken = follow ? __shfl_sync(0xFFFFFFFFu, base, 0) : nold;
            const int fresh = nold + __shfl_sync(0xFFFFFFFFu, base, 1);
            const unsigned below = (1u << lane) - 1u;
            int slot = nc >= 0 ? fresh + __popc(found & below) : taken + __popc(~found & below);
            FTrack T;
            if (nc >= 0) {
                T = make_track(na, nc, nb, nc, 3, 0);
                if (slot >= cap) {
                    misc[kErr] = SBT_ERR_CAPACITY;
                    slot = -1;
                }
            } else if (slot < nold) {
                T = Fc[slot];
            } else {
                slot = -1;
            }
            if (slot >= 0) {
                if (follow) follow_and_claim<kAhead, G>(C, S, R, t, tag, sq_follow, T);
                Fc[slot] = T;
            }
            nc = -1;
            if (i0 >= nl && taken + 32 - __popc(found) >= nold) break;
        }
        __syncthreads();
        if (misc[kErr]) return false;
        const int nf = nold + misc[kNew];
        if (tid == 0) misc[kList] = 0;
        // P2
        if (follow) {
            for (int f = tid; f < nf; f += NT) {
                const FTrack T = Fc[f];
                if (T.cand == kDead) continue;
                bool won = false;
                if (T.cand != kNone) {
                    const unsigned long long k = claim_key(tag, T.sc, T.key);
                    // all claim words loaded at once (one round trip)
                    const unsigned long long ca = __ldcg(&R.claim[T.cand & R.cmask]);
                    unsigned long long k0 = k, k1 = k, k2 = k;
                    if (T.nh == 3) {
                        k0 = __ldcg(&R.claim[T.h0 & R.cmask]);
                        k1 = __ldcg(&R.claim[T.h1 & R.cmask]);
                        k2 = __ldcg(&R.claim[T.h2 & R.cmask]);
                    }
                    won = ca == k && k0 == k && k1 == k && k2 == k;
                }
                if (won) {
                    set_flag(S, T.cand);
                    if (T.nh == 3) {
                        set_flag(S, T.h0);
                        set_flag(S, T.h1);
                        set_flag(S, T.h2);
                        R.prev[T.h0] = kNone;
                        R.prev[T.h1] = T.h0;
                        R.prev[T.h2] = T.h1;
                    }
                    R.prev[T.cand] = T.h2;
                    const int slot = atomicAdd(&misc[kCnt0 + nxt], 1);
                    Fn[slot] = make_track(T.h1, T.h2, T.cand, T.key, T.nh + 1, 0);
                } else if (T.sk + 1 >= 2) {
                    if (T.nh >= 4)
                        add_final(S, R, T.h2, T.nh);
                    else
                        add_tracklet(S, R, T.h0, T.h1, T.h2, T.key);
                } else {
                    const int slot = atomicAdd(&misc[kCnt0 + nxt], 1);
                    Fn[slot] = make_track(T.h0, T.h1, T.h2, T.key, T.nh, T.sk + 1);
                }
            }
        } else {
            // last iteration: every forming track is finished
            for (int f = tid; f < nf; f += NT) {
                const FTrack T = Fc[f];
                if (T.nh >= 4)
                    add_final(S, R, T.h2, T.nh);
                else
                    add_tracklet(S, R, T.h0, T.h1, T.h2, T.key);
            }
        }
        __syncthreads();
        cur = nxt;
    }
    return misc[kErr] == 0;
}

// Tracklet filter: three unflagged hits and chi2 < C3, then one claim round
// among the survivors (tag 0, below every search tag).
template <int NT, class HS>
__device__ void tracklet_filter(const DevConfig& C, const Region<HS>& R, const Smem& S)
{
    const int tid = threadIdx.x;
    const int ntl = min(S.misc[kNTl], R.lcap);
    // the search kept its claims in a ring; the filter's claims use the whole
    // array, the tracklets' words cleared first
    for (int k = tid; k < ntl; k += NT) {
        const unsigned long long v = R.tracklets[k];
        R.claim_all[v & 0xFFFF] = ~0ull;
        R.claim_all[(v >> 16) & 0xFFFF] = ~0ull;
        R.claim_all[(v >> 32) & 0xFFFF] = ~0ull;
    }
    __syncthreads();
    for (int k = tid; k < ntl; k += NT) {
        unsigned long long v = R.tracklets[k];
        int h[3] = {(int)(v & 0xFFFF), (int)((v >> 16) & 0xFFFF), (int)((v >> 32) & 0xFFFF)};
        int key = (int)(v >> 48);
        uint32_t q = 0xFFFFFFFFu;
        if (!flagged(S, h[0]) && !flagged(S, h[1]) && !flagged(S, h[2])) {
            const float chi2 = fit_chi2(
                3,
                [&](int i) {
                    float4 c = R.coords[h[i]];
                    return make_float3(c.x, c.y, c.z);
                },
                C.sigma);
            if (chi2 < C.C3) {
                q = __float_as_uint(chi2);
                unsigned long long kk = claim_key(0ull, chi2, key);
                atomicMin(&R.claim_all[h[0]], kk);
                atomicMin(&R.claim_all[h[1]], kk);
                atomicMin(&R.claim_all[h[2]], kk);
            }
        }
        R.tl_q[k] = q;
    }
    __syncthreads();
    for (int k = tid; k < ntl; k += NT) {
        uint32_t q = R.tl_q[k];
        if (q == 0xFFFFFFFFu) continue;
        unsigned long long v = R.tracklets[k];
        int h0 = (int)(v & 0xFFFF), h1 = (int)((v >> 16) & 0xFFFF), h2 = (int)((v >> 32) & 0xFFFF);
        unsigned long long kk = claim_key(0ull, __uint_as_float(q), (int)(v >> 48));
        if (__ldcg(&R.claim_all[h0]) == kk && __ldcg(&R.claim_all[h1]) == kk && __ldcg(&R.claim_all[h2]) == kk) {
            R.prev[h0] = kNone;
            R.prev[h1] = (uint16_t)h0;
            R.prev[h2] = (uint16_t)h1;
            add_final(S, R, h2, 3);
        }
    }
    __syncthreads();
}

// Staging of the tracks: each track's linked hit list is walked once, its
// hit records written in traversal order at its found-order place among the
// event's staged hits, with its smallest input index.  Ordering and fits are
// left to the output kernel.
template <int NT, class HS>
__device__ void output_stage(int e, int off, const Region<HS>& R, const Smem& S, const Staging& G,
                             const sbt_tracks& out)
{
    const int tid = threadIdx.x;
    const int T = S.misc[kNFin];
    const int chunk = (T + NT - 1) / NT;
    const int beg = min(T, tid * chunk), end = min(T, beg + chunk);
    int cnt = 0;
    for (int k = beg; k < end; k++) cnt += (int)(R.finals[k] >> 16);
    int H;
    int u = block_exclusive_scan<NT>(cnt, S.wsum, &H);
    const int64_t slot0 = (int64_t)off / 3 + e;
    float4* hits = G.hits + off;
    for (int k = beg; k < end; k++) {
        const uint32_t v = R.finals[k];
        int q = (int)(v & 0xFFFF);
        const int nh = (int)(v >> 16);
        int mn = INT_MAX;
        for (int j = nh - 1; j >= 0; j--) {
            const int nq = R.prev[q];
            const float4 c = R.coords[q];
            const int i = R.coords.index(c, q);
            hits[u + j] = make_float4(c.x, c.y, c.z, __int_as_float(off + i));
            mn = i < mn ? i : mn;
            q = nq;
        }
        G.tkey[slot0 + k] = mn;
        G.tinfo[slot0 + k] = (uint32_t)u | ((uint32_t)nh << 16);
        u += nh;
    }
    if (tid == 0) {
        G.ev_ntracks[e] = T;
        G.ev_nhits[e] = H;
        out.event_status[e] = SBT_OK;
    }
}

__device__ __forceinline__ void fail_event(int e, int code, const Staging& G, const sbt_tracks& out)
{
    if (threadIdx.x == 0) {
        G.ev_ntracks[e] = 0;
        G.ev_nhits[e] = 0;
        out.event_status[e] = code;
    }
}

// Search of one sorted event by the whole block.
template <int NT, class HS, class GEO>
__device__ void run_event(const DevConfig& C, const Inputs& in, const Sorted& O, const Work& W,
                          const Staging& G, const sbt_tracks& out, int e, int64_t hb, int64_t r,
                          int cap, const Smem& S)
{
    const int tid = threadIdx.x;
    const int off = in.offsets[e];
    const int n = in.offsets[e + 1] - off;
    const int st = O.status[e];
    if (st != SBT_OK || n > cap) {
        fail_event(e, st != SBT_OK ? st : SBT_ERR_CAPACITY, G, out);
        return;
    }
    Region<HS> R = region_of<HS>(O, off, W, hb, r, cap);
    for (int m = tid; m <= C.M; m += NT) S.modoff[m] = O.modoff[(int64_t)e * (C.M + 1) + m];
    for (int w = tid; w < (n + 31) / 32; w += NT) S.flag[w] = 0u;
    __syncthreads();
    // Claims are live only on the modules s-1 .. s+3 of step s (a 3-hit track
    // has its hits on s-1 or later, a new hit lies on s+3), so the search keeps
    // them in a ring of the smallest power of two that covers every such span:
    // live positions never share a slot, and the ring stays in cache.  Without
    // such a power of two within the region's capacity, no ring.
    if (tid < 32) {
        int w = 0;
        for (int s = tid; s + 2 <= C.M - 1; s += 32)
            w = max(w, S.modoff[min(s + 4, C.M)] - S.modoff[max(s - 1, 0)]);
        w = __reduce_max_sync(0xFFFFFFFFu, w);
        const int p2 = w > 1 ? 1 << (32 - __clz(w - 1)) : 1;
        if (tid == 0) S.misc[kCMask] = p2 <= cap ? p2 - 1 : -1;
        if (tid == 0) {
            S.misc[kShift] = 16 - bucket_bits(O.tables, n, C.M);
            *S.table = O.bucket + table_base(O.tables, off, e);
        }
        if (tid < kMiscN && tid != kCMask && tid != kEvent && tid != kShift) S.misc[tid] = 0;
    }
    __syncthreads();
    // the ring starts empty; older claims lose against newer ones by their tag
    R.cmask = (unsigned)S.misc[kCMask];
    const int ring = R.cmask == ~0u ? n : min(n, (int)R.cmask + 1);
    for (int p = tid; p < ring; p += NT) R.claim[p] = ~0ull;
    __syncthreads();
    if (!search_stage<NT, GEO>(C, R, S, n)) {
        fail_event(e, SBT_ERR_CAPACITY, G, out);
        __syncthreads();
        return;
    }
    tracklet_filter<NT>(C, R, S);
    output_stage<NT>(e, off, R, S, G, out);
    __syncthreads();
}

// ------------------------------------------------------------- kernels ---

// Residency of the search: the kernel waits on load latency, so throughput
// follows the number of resident events; the compiler is asked for a
// register count that lets 2048 threads share an SM (16 blocks of 128, 16000
// uneven events: 4.99 ms; 1536 threads 5.34, 1024 threads 6.07).  Blocks of 512
// run calls of a few events, where a step's length counts: 64 registers, no
// spills (one event 226 us at 256 threads and 32 registers, 204 at 64; 200 us at
// 512).
constexpr int search_blocks_per_sm(int threads) { return (threads == 512 ? 1024 : 2048) / threads; }

// One block per event.
template <int NT, class HS, class GEO>
__global__ void __launch_bounds__(NT, search_blocks_per_sm(NT)) k_search_plain(DevConfig C, Inputs in, Sorted O, Work W,
                                                      Staging G, sbt_tracks out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem S = carve(smem_raw, C.nmax, NT, C.M);
    const int e = blockIdx.x;
    const int off = in.offsets[e];
    const int n = in.offsets[e + 1] - off;
    run_event<NT, HS, GEO>(C, in, O, W, G, out, e, off, e, max(n, 0), S);
}

// Persistent: each resident block takes events from the work queue, sizes
// alternating from both ends of G.order (largest first), and reuses its own
// scratch region.
template <int NT, class HS, class GEO>
__global__ void __launch_bounds__(NT, search_blocks_per_sm(NT)) k_search_persistent(DevConfig C, Inputs in, Sorted O, Work W,
                                                           Staging G, sbt_tracks out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Smem S = carve(smem_raw, C.nmax, NT, C.M);
    const int64_t hb = (int64_t)blockIdx.x * C.nmax;
    for (;;) {
        if (threadIdx.x == 0) S.misc[kEvent] = atomicAdd(&G.queue[0], 1);
        __syncthreads();
        const int q = S.misc[kEvent];
        __syncthreads();
        if (q >= in.n_events) break;
        // alternately the largest and the smallest event not yet taken, so
        // the resident events' hits and scratch stay near the average size
        // (the largest-first order alone fills L2 with the heaviest events at
        // the start); the last 2 x blocks events, from the middle of the size
        // order, are taken largest first, which keeps the tail short
        const int q0 = max(0, in.n_events - 2 * (int)gridDim.x) & ~1;
        const int qi = q >= q0 ? (q0 >> 1) + (q - q0) : (q & 1) ? in.n_events - 1 - (q >> 1) : (q >> 1);
        run_event<NT, HS, GEO>(C, in, O, W, G, out, G.order[qi], hb, blockIdx.x, C.nmax, S);
    }
}

// Processing order, largest events first (counting sort on size classes).
__global__ void __launch_bounds__(1024) k_order(Inputs in, Staging G)
{
    __shared__ int hist[1024];
    __shared__ int wsum[33];
    const int tid = threadIdx.x;
    const int E = in.n_events;
    hist[tid] = 0;
    __syncthreads();
    for (int e = tid; e < E; e += 1024) {
        int n = in.offsets[e + 1] - in.offsets[e];
        int b = 1023 - min(max(n, 0) >> 4, 1023);
        atomicAdd(&hist[b], 1);
    }
    __syncthreads();
    int v = hist[tid];
    int total;
    int ex = block_exclusive_scan<1024>(v, wsum, &total);
    hist[tid] = ex;
    __syncthreads();
    for (int e = tid; e < E; e += 1024) {
        int n = in.offsets[e + 1] - in.offsets[e];
        int b = 1023 - min(max(n, 0) >> 4, 1023);
        G.order[atomicAdd(&hist[b], 1)] = e;
    }
}

// Device-wide exclusive scan of the per-event track and hit counts, with the
// capacity check.  One block; each thread owns a contiguous run of events.
__global__ void __launch_bounds__(1024) k_scan(Inputs in, Staging G, sbt_tracks out)
{
    __shared__ int wsum[33];
    __shared__ int first_over;
    const int tid = threadIdx.x;
    const int E = in.n_events;
    if (tid == 0) first_over = INT_MAX;
    const int chunk = (E + 1023) / 1024;
    const int beg = min(E, tid * chunk), end = min(E, beg + chunk);
    int t = 0, h = 0, f = 0;
    for (int e = beg; e < end; e++) {
        t += G.ev_ntracks[e];
        h += G.ev_nhits[e];
        f += out.event_status[e] != SBT_OK && out.event_status[e] != SBT_EVENT_CUT;
    }
    int T, H, F;
    int bt = block_exclusive_scan<1024>(t, wsum, &T);
    int bh = block_exclusive_scan<1024>(h, wsum, &H);
    block_exclusive_scan<1024>(f, wsum, &F);
    for (int e = beg; e < end; e++) {
        G.track_base[e] = bt;
        G.hit_base[e] = bh;
        out.track_offsets[e] = bt;
        // the output kernel skips the events past the capacities: a suffix
        if ((int64_t)bt + G.ev_ntracks[e] > out.cap_tracks || (int64_t)bh + G.ev_nhits[e] > out.cap_hits)
            atomicMin(&first_over, bt);
        bt += G.ev_ntracks[e];
        bh += G.ev_nhits[e];
    }
    __syncthreads();
    if (tid == 0) {
        G.queue[1] = min(first_over, T);
        out.track_offsets[E] = T;
        bool ok = T <= out.cap_tracks && H <= out.cap_hits;
        if (ok) out.hit_offsets[T] = H;
        out.counts[0] = T;
        out.counts[1] = H;
        out.counts[2] = ok ? SBT_OK : SBT_ERR_CAPACITY;
        out.counts[3] = F;
    }
}

// Output (section "Results", data consolidation), one block per event: the
// canonical order of the event's T tracks by smallest input hit index and
// their CSR starts, from batch track tb and hit hbase on; the hit lists and
// fits follow in fit_tracks.  A track's rank is the number of tracks with a
// smaller smallest index: one bit per input index marks the tracks' smallest
// indices (shared memory, `bits` and `wpre` a word per 32 hits), and a prefix
// of the words' bit counts gives every rank.
constexpr int kOutputThreads = 256;

__device__ __forceinline__ void order_tracks(const Inputs& in, const Staging& G, const sbt_tracks& out, int e, int T,
                                             int tb, int hbase, uint32_t* bits, int* wpre, int* wsum)
{
    constexpr int NT = kOutputThreads;
    const int tid = threadIdx.x;
    const int off = in.offsets[e];
    const int n = in.offsets[e + 1] - off;
    const int64_t slot0 = (int64_t)off / 3 + e;
    const int nw = (n + 31) / 32;
    for (int w = tid; w < nw; w += NT) bits[w] = 0u;
    __syncthreads();
    for (int k = tid; k < T; k += NT) {
        const int mn = G.tkey[slot0 + k];
        atomicOr(&bits[mn >> 5], 1u << (mn & 31));
    }
    __syncthreads();
    {
        const int wc = (nw + NT - 1) / NT;
        const int wb = min(nw, tid * wc), we = min(nw, wb + wc);
        int c = 0;
        for (int w = wb; w < we; w++) c += __popc(bits[w]);
        int tot;
        int st = block_exclusive_scan<NT>(c, wsum, &tot);
        for (int w = wb; w < we; w++) {
            wpre[w] = st;
            st += __popc(bits[w]);
        }
    }
    __syncthreads();
    for (int k = tid; k < T; k += NT) {
        const int mn = G.tkey[slot0 + k];
        const int r = wpre[mn >> 5] + __popc(bits[mn >> 5] & ((1u << (mn & 31)) - 1u));
        G.rinfo[slot0 + r] = G.tinfo[slot0 + k];
    }
    __syncthreads();
    // canonical starts: each thread takes a contiguous run of ranks
    const int chunk = (T + NT - 1) / NT;
    const int beg = min(T, tid * chunk), end = min(T, beg + chunk);
    int c = 0;
    for (int r = beg; r < end; r++) c += (int)(G.rinfo[slot0 + r] >> 16);
    int Ht;
    int cs = block_exclusive_scan<NT>(c, wsum, &Ht);
    for (int r = beg; r < end; r++) {
        const uint32_t ri = G.rinfo[slot0 + r];
        const int nh = (int)(ri >> 16);
        const int64_t g = (int64_t)tb + r;
        out.hit_offsets[g] = hbase + cs;
        G.tfit[g] = make_uint2((uint32_t)(off + (int)(ri & 0xFFFFu)), (uint32_t)nh);
        cs += nh;
    }
}

// Batches above kFinishEvents: order per event, then all tracks' fits.
__global__ void __launch_bounds__(kOutputThreads) k_output(DevConfig C, Inputs in, Staging G,
                                                          sbt_tracks out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nwmax = (C.nmax + 31) / 32;
    uint32_t* bits = (uint32_t*)smem_raw;
    __shared__ int wsum[40];
    const int e = blockIdx.x;
    const int T = G.ev_ntracks[e];
    if (T == 0) return;
    const int tb = G.track_base[e], hbase = G.hit_base[e];
    if ((int64_t)tb + T > out.cap_tracks || (int64_t)hbase + G.ev_nhits[e] > out.cap_hits) return;
    order_tracks(in, G, out, e, T, tb, hbase, bits, (int*)(bits + nwmax), wsum);
}

// Hit lists and least-squares fits of canonical tracks [g0, g0 + 32) below T by
// one warp, a lane per track (a warp's hit lists and parameters are contiguous
// in the output).  The warp first copies its tracks, half a warp per track,
// eight tracks in flight: the staged records come in coalesced, the hit lists
// go out coalesced, and the coordinates of the first kFitRows hits land in
// shared memory, one column per track, where every lane then reads its own
// without conflicts (33 words a row).  With each lane
// loading its own track's records and storing its own hit list, every lane was
// an L1 wavefront of its own (two a hit, the LSU data pipe 74% busy).  The sums
// run in hit order, every operation rounded as in fit_chi2.
constexpr int kFitThreads = 128;
constexpr int kFitRows = 16;
constexpr int kFitAhead = 4;
// Six blocks an SM (80 registers, 25 KB a block) hold enough loads in flight:
// output step of 16000 uneven events 798 -> 660 us; at four blocks with 24 rows
// 744, five with 20 rows 687, eight (64 registers) 893; half as many tracks in
// flight 960.
constexpr int kFitBlocksPerSM = 6;

struct FitColumns {
    float v[3][kFitRows][33];
};

__device__ __forceinline__ void fit_tracks(const DevConfig& C, const Staging& G, const sbt_tracks& out,
                                           FitColumns& cols, int64_t g0, int T)
{
    const int lane = threadIdx.x & 31;
    float(*col)[kFitRows][33] = cols.v;
    const bool wide = ((uintptr_t)out.params & 15) == 0;
    const int64_t g = g0 + lane;
    const uint2 f = g < T ? G.tfit[g] : make_uint2(0u, 0u);
    const int n = (int)f.y;
    const int to = g < T ? out.hit_offsets[g] : 0;
    // half a warp per track: hits 0-15 of two tracks, then 16-31 where there are any
    const int half = lane >> 4, j0 = lane & 15;
    for (int k0 = 0; k0 < 32; k0 += 2 * kFitAhead) {
        float4 v[kFitAhead], w[kFitAhead];
        int nk[kFitAhead], tk[kFitAhead];
#pragma unroll
        for (int u = 0; u < kFitAhead; u++) {
            const int k = k0 + 2 * u + half;
            nk[u] = __shfl_sync(0xFFFFFFFFu, n, k);
            tk[u] = __shfl_sync(0xFFFFFFFFu, to, k);
            const float4* sk = G.hits + (__shfl_sync(0xFFFFFFFFu, f.x, k) + (uint32_t)j0);
            if (j0 < nk[u]) v[u] = sk[0];
            if (j0 + 16 < nk[u]) w[u] = sk[16];
        }
        auto keep = [&](float4 c, int j, int u) {
            out.track_hits[tk[u] + j] = __float_as_int(c.w);
            if (j < kFitRows) {
                const int k = k0 + 2 * u + half;
                col[0][j][k] = c.x;
                col[1][j][k] = c.y;
                col[2][j][k] = c.z;
            }
        };
#pragma unroll
        for (int u = 0; u < kFitAhead; u++) {
            if (j0 < nk[u]) keep(v[u], j0, u);
            if (j0 + 16 < nk[u]) keep(w[u], j0 + 16, u);
        }
    }
    __syncwarp();
    // hits past the rows, and hit lists past a warp's lanes
    const float4* src = G.hits + f.x;
    for (int j = 32; j < n; j++) out.track_hits[to + j] = __float_as_int(src[j].w);
    const int ns = min(n, kFitRows);
    auto each = [&](auto use) {
#pragma unroll 4
        for (int j = 0; j < ns; j++) use(col[0][j][lane], col[1][j][lane], col[2][j][lane]);
        for (int j = kFitRows; j < n; j++) {
            const float4 q = src[j];
            use(q.x, q.y, q.z);
        }
    };
    if (n > 0) {
        float sx = 0.0f, sy = 0.0f, sz = 0.0f;
        each([&](float x, float y, float z) {
            sx = __fadd_rn(sx, x);
            sy = __fadd_rn(sy, y);
            sz = __fadd_rn(sz, z);
        });
        const float nf = (float)n;
        const float xm = __fdiv_rn(sx, nf), ym = __fdiv_rn(sy, nf), zm = __fdiv_rn(sz, nf);
        float szz = 0.0f, szx = 0.0f, szy = 0.0f;
        each([&](float x, float y, float z) {
            const float dz = __fsub_rn(z, zm);
            szz = __fadd_rn(szz, __fmul_rn(dz, dz));
            szx = __fadd_rn(szx, __fmul_rn(dz, __fsub_rn(x, xm)));
            szy = __fadd_rn(szy, __fmul_rn(dz, __fsub_rn(y, ym)));
        });
        const float tx = __fdiv_rn(szx, szz);
        const float ty = __fdiv_rn(szy, szz);
        float s = 0.0f;
        each([&](float x, float y, float z) {
            const float dz = __fsub_rn(z, zm);
            const float rx = __fsub_rn(__fsub_rn(x, xm), __fmul_rn(tx, dz));
            const float ry = __fsub_rn(__fsub_rn(y, ym), __fmul_rn(ty, dz));
            s = __fadd_rn(s, __fadd_rn(__fmul_rn(rx, rx), __fmul_rn(ry, ry)));
        });
        const float4 p = make_float4(__fsub_rn(xm, __fmul_rn(tx, zm)), __fsub_rn(ym, __fmul_rn(ty, zm)), tx, ty);
        if (wide) {
            ((float4*)out.params)[g] = p;
        } else {
            out.params[4 * g + 0] = p.x;
            out.params[4 * g + 1] = p.y;
            out.params[4 * g + 2] = p.z;
            out.params[4 * g + 3] = p.w;
        }
        out.chi2[g] = __fdiv_rn(s, __fmul_rn(C.sigma, C.sigma));
        out.ndof[g] = 2 * n - 4;
    }
    __syncwarp();
}

// All tracks of the events that k_output wrote, G.queue[1] of them.
__global__ void __launch_bounds__(kFitThreads, kFitBlocksPerSM) k_fit(DevConfig C, Staging G, sbt_tracks out)
{
    __shared__ FitColumns cols[kFitThreads / 32];
    const int T = G.queue[1];
    for (int64_t g0 = (int64_t)blockIdx.x * kFitThreads + (threadIdx.x & ~31); g0 < T;
         g0 += (int64_t)gridDim.x * kFitThreads)
        fit_tracks(C, G, out, cols[threadIdx.x >> 5], g0, T);
}

// Scan, order and fits of a small batch in one launch, one block per event:
// every block sums the counts of the events before its own (at most
// kFinishEvents of them), then orders and fits its tracks; the last block
// writes the totals.  Launch latencies are what the three kernels of a large
// batch cost here.
__global__ void __launch_bounds__(kOutputThreads) k_finish(DevConfig C, Inputs in, Staging G, sbt_tracks out)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FitColumns* cols = (FitColumns*)smem_raw;  // [kOutputThreads / 32]
    const int nwmax = (C.nmax + 31) / 32;
    uint32_t* bits = (uint32_t*)(cols + kOutputThreads / 32);
    __shared__ int wsum[40];
    __shared__ int sums[3];  // tracks and hits before this event; failed events of the batch
    const int e = blockIdx.x, E = in.n_events, tid = threadIdx.x;
    const bool last = e == E - 1;
    if (tid < 3) sums[tid] = 0;
    __syncthreads();
    int t = 0, h = 0, f = 0;
    for (int k = tid; k < E; k += kOutputThreads) {
        if (k < e) {
            t += G.ev_ntracks[k];
            h += G.ev_nhits[k];
        }
        if (last) f += out.event_status[k] != SBT_OK && out.event_status[k] != SBT_EVENT_CUT;
    }
    t = __reduce_add_sync(0xFFFFFFFFu, t);
    h = __reduce_add_sync(0xFFFFFFFFu, h);
    f = __reduce_add_sync(0xFFFFFFFFu, f);
    if ((tid & 31) == 0) {
        atomicAdd(&sums[0], t);
        atomicAdd(&sums[1], h);
        atomicAdd(&sums[2], f);
    }
    const int T = G.ev_ntracks[e], H = G.ev_nhits[e];
    __syncthreads();
    const int tb = sums[0], hbase = sums[1];
    if (tid == 0) {
        out.track_offsets[e] = tb;
        if (last) {
            const bool ok = tb + T <= out.cap_tracks && hbase + H <= out.cap_hits;
            out.track_offsets[E] = tb + T;
            if (ok) out.hit_offsets[tb + T] = hbase + H;
            out.counts[0] = tb + T;
            out.counts[1] = hbase + H;
            out.counts[2] = ok ? SBT_OK : SBT_ERR_CAPACITY;
            out.counts[3] = sums[2];
        }
    }
    // events past the capacities are a suffix
    if (T == 0 || (int64_t)tb + T > out.cap_tracks || (int64_t)hbase + H > out.cap_hits) return;
    order_tracks(in, G, out, e, T, tb, hbase, bits, (int*)(bits + nwmax), wsum);
    __syncthreads();
    for (int64_t g0 = tb + (tid & ~31); g0 < tb + T; g0 += kOutputThreads)
        fit_tracks(C, G, out, cols[tid >> 5], g0, tb + T);
}

size_t output_smem_bytes(int nmax) { return 8 * (size_t)((nmax + 31) / 32); }
size_t finish_smem_bytes(int nmax) { return sizeof(FitColumns) * (kOutputThreads / 32) + output_smem_bytes(nmax); }

// Chunked host pipeline: adds the totals of the earlier chunks to one chunk's
// CSR offsets (track_offsets [n_events + 1], hit_offsets [counts[0] + 1]) and
// advances the running totals (running[0] tracks, running[1] hits).
// Chunk offsets made global: running[0..1] hold the tracks and track hits of
// the earlier chunks (read by every block), running[2..3] receive the totals
// including this chunk (written by block 0 only).
__global__ void __launch_bounds__(256) k_offset_fixup(int32_t* track_offsets, int32_t n_events,
                                                      int32_t* hit_offsets, const int32_t* counts,
                                                      int64_t* running)
{
    const int64_t bt = running[0], bh = running[1];
    const int T = counts[0];
    const bool ok = counts[2] == SBT_OK;
    const int stride = gridDim.x * blockDim.x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n_events; i += stride)
        track_offsets[i] += (int32_t)bt;
    if (ok)
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t <= T; t += stride)
            hit_offsets[t] += (int32_t)bh;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        running[2] = bt + T;
        running[3] = bh + counts[1];
    }
}

// Sort stage output copied out, for stage-level checks.
template <class HS>
__global__ void k_debug_sort_copy(DevConfig C, Inputs in, Sorted O, uint16_t* phi16, int32_t* perm,
                                  int32_t* modoff)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < in.n_hits) {
        const HitArr<HS> hits{(const typename HS::T*)O.coords, O.index};
        phi16[i] = (uint16_t)hits.phi((int)i);
        perm[i] = hits.index(hits[(int)i], (int)i);
    }
    if (i < (int64_t)in.n_events * (C.M + 1)) modoff[i] = O.modoff[i];
}

__global__ void k_debug_phi16(const float* x, const float* y, int32_t n, uint16_t* out)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (uint16_t)phi16_of(x[i], y[i]);
}

// ------------------------------------------------------------ launchers ---

cudaError_t launch_sort(const DevConfig& C, const Inputs& in, const Sorted& O, cudaStream_t st)
{
    size_t sm = sort_smem_bytes(C.nmax);
    auto kern = C.h16 ? k_sort<HitsF16> : k_sort<HitsF32>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    if (in.n_events > 0) kern<<<in.n_events, kSortThreads, sm, st>>>(C, in, O);
    return cudaGetLastError();
}

template <int NT, class HS, class GEO>
static cudaError_t plain_ntg(const DevConfig& C, const Inputs& in, const Sorted& O, const Work& W,
                             const Staging& G, const sbt_tracks& out, cudaStream_t st)
{
    size_t sm = smem_bytes(C.nmax, NT, C.M);
    cudaError_t err = cudaFuncSetAttribute(k_search_plain<NT, HS, GEO>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    if (in.n_events > 0) k_search_plain<NT, HS, GEO><<<in.n_events, NT, sm, st>>>(C, in, O, W, G, out);
    return cudaGetLastError();
}

template <int NT, class HS>
static cudaError_t plain_nt(const DevConfig& C, const Inputs& in, const Sorted& O, const Work& W,
                            const Staging& G, const sbt_tracks& out, cudaStream_t st)
{
    return C.pairs ? plain_ntg<NT, HS, PairGeo>(C, in, O, W, G, out, st)
                   : plain_ntg<NT, HS, PlaneGeo>(C, in, O, W, G, out, st);
}

cudaError_t launch_plain(const DevConfig& C, const Inputs& in, const Sorted& O, const Work& W,
                         const Staging& S, const sbt_tracks& out, int threads, cudaStream_t stream)
{
    switch (threads) {
        case 64: return C.h16 ? plain_nt<64, HitsF16>(C, in, O, W, S, out, stream) : plain_nt<64, HitsF32>(C, in, O, W, S, out, stream);
        case 128: return C.h16 ? plain_nt<128, HitsF16>(C, in, O, W, S, out, stream) : plain_nt<128, HitsF32>(C, in, O, W, S, out, stream);
        case 256: return C.h16 ? plain_nt<256, HitsF16>(C, in, O, W, S, out, stream) : plain_nt<256, HitsF32>(C, in, O, W, S, out, stream);
        case 512: return C.h16 ? plain_nt<512, HitsF16>(C, in, O, W, S, out, stream) : plain_nt<512, HitsF32>(C, in, O, W, S, out, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_order(const Inputs& in, const Staging& S, cudaStream_t stream)
{
    k_order<<<1, 1024, 0, stream>>>(in, S);
    return cudaGetLastError();
}

template <int NT, class HS, class GEO>
static int occupancy_ntg(const DevConfig& C)
{
    size_t sm = smem_bytes(C.nmax, NT, C.M);
    if (cudaFuncSetAttribute(k_search_persistent<NT, HS, GEO>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sm) != cudaSuccess)
        return 0;
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_search_persistent<NT, HS, GEO>, NT, sm) !=
        cudaSuccess)
        return 0;
    return blocks;
}

template <int NT, class HS>
static int occupancy_nt(const DevConfig& C)
{
    return C.pairs ? occupancy_ntg<NT, HS, PairGeo>(C) : occupancy_ntg<NT, HS, PlaneGeo>(C);
}

int persistent_blocks_per_sm(const DevConfig& C, int threads)
{
    switch (threads) {
        case 64: return C.h16 ? occupancy_nt<64, HitsF16>(C) : occupancy_nt<64, HitsF32>(C);
        case 128: return C.h16 ? occupancy_nt<128, HitsF16>(C) : occupancy_nt<128, HitsF32>(C);
        case 256: return C.h16 ? occupancy_nt<256, HitsF16>(C) : occupancy_nt<256, HitsF32>(C);
        case 512: return C.h16 ? occupancy_nt<512, HitsF16>(C) : occupancy_nt<512, HitsF32>(C);
        default: return 0;
    }
}

template <int NT, class HS, class GEO>
static cudaError_t persistent_ntg(const DevConfig& C, const Inputs& in, const Sorted& O, const Work& W,
                                  const Staging& G, const sbt_tracks& out, int blocks,
                                  cudaStream_t st)
{
    size_t sm = smem_bytes(C.nmax, NT, C.M);
    cudaError_t err = cudaFuncSetAttribute(k_search_persistent<NT, HS, GEO>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    if (blocks > 0) k_search_persistent<NT, HS, GEO><<<blocks, NT, sm, st>>>(C, in, O, W, G, out);
    return cudaGetLastError();
}

template <int NT, class HS>
static cudaError_t persistent_nt(const DevConfig& C, const Inputs& in, const Sorted& O, const Work& W,
                                 const Staging& G, const sbt_tracks& out, int blocks,
                                 cudaStream_t st)
{
    return C.pairs ? persistent_ntg<NT, HS, PairGeo>(C, in, O, W, G, out, blocks, st)
                   : persistent_ntg<NT, HS, PlaneGeo>(C, in, O, W, G, out, blocks, st);
}

cudaError_t launch_persistent(const DevConfig& C, const Inputs& in, const Sorted& O, const Work& W,
                              const Staging& S, const sbt_tracks& out, int threads, int blocks,
                              cudaStream_t stream)
{
    switch (threads) {
        case 64: return C.h16 ? persistent_nt<64, HitsF16>(C, in, O, W, S, out, blocks, stream) : persistent_nt<64, HitsF32>(C, in, O, W, S, out, blocks, stream);
        case 128: return C.h16 ? persistent_nt<128, HitsF16>(C, in, O, W, S, out, blocks, stream) : persistent_nt<128, HitsF32>(C, in, O, W, S, out, blocks, stream);
        case 256: return C.h16 ? persistent_nt<256, HitsF16>(C, in, O, W, S, out, blocks, stream) : persistent_nt<256, HitsF32>(C, in, O, W, S, out, blocks, stream);
        case 512: return C.h16 ? persistent_nt<512, HitsF16>(C, in, O, W, S, out, blocks, stream) : persistent_nt<512, HitsF32>(C, in, O, W, S, out, blocks, stream);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_scan(const Inputs& in, const Staging& S, const sbt_tracks& out,
                        cudaStream_t stream)
{
    k_scan<<<1, 1024, 0, stream>>>(in, S, out);
    return cudaGetLastError();
}

cudaError_t launch_output(const DevConfig& C, const Inputs& in, const Staging& S,
                          const sbt_tracks& out, cudaStream_t stream)
{
    const size_t sm = output_smem_bytes(C.nmax);
    cudaError_t err = cudaFuncSetAttribute(k_output, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    if (in.n_events > 0) k_output<<<in.n_events, kOutputThreads, sm, stream>>>(C, in, S, out);
    err = cudaGetLastError();
    if (err != cudaSuccess || in.n_events == 0) return err;
    // k_fit: one resident wave over the device, a grid-stride loop over the tracks
    int dev = 0, sms = 0, per_sm = 0;
    err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err == cudaSuccess) err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fit, kFitThreads, 0);
    if (err != cudaSuccess) return err;
    k_fit<<<sms * std::max(per_sm, 1), kFitThreads, 0, stream>>>(C, S, out);
    return cudaGetLastError();
}

// One launch up to here: 16 quiet events 152 -> 144 us a call, one event 243 ->
// 238; from 100 events on (363 -> 365 us, 500 events 484 -> 490) three kernels
// pack the tracks of all events better than a block per event does.
constexpr int kFinishEvents = 64;
int finish_launches(int n_events) { return n_events <= kFinishEvents ? 1 : 3; }

cudaError_t launch_finish(const DevConfig& C, const Inputs& in, const Staging& S,
                          const sbt_tracks& out, cudaStream_t stream)
{
    if (in.n_events > 0 && in.n_events <= kFinishEvents) {
        const size_t sm = finish_smem_bytes(C.nmax);
        cudaError_t err = cudaFuncSetAttribute(k_finish, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        if (err != cudaSuccess) return err;
        k_finish<<<in.n_events, kOutputThreads, sm, stream>>>(C, in, S, out);
        return cudaGetLastError();
    }
    cudaError_t e = launch_scan(in, S, out, stream);
    if (e == cudaSuccess) e = launch_output(C, in, S, out, stream);
    return e;
}

cudaError_t launch_debug_sort_copy(const DevConfig& C, const Inputs& in, const Sorted& O,
                                   uint16_t* phi16, int32_t* perm, int32_t* module_offsets,
                                   cudaStream_t stream)
{
    const int64_t n = std::max<int64_t>(in.n_hits, (int64_t)in.n_events * (C.M + 1));
    if (n > 0)
        (C.h16 ? k_debug_sort_copy<HitsF16> : k_debug_sort_copy<HitsF32>)<<<(unsigned)((n + 255) / 256), 256, 0,
                                                                          stream>>>(C, in, O, phi16, perm,
                                                                                    module_offsets);
    return cudaGetLastError();
}

cudaError_t launch_offset_fixup(int32_t* track_offsets, int32_t n_events, int32_t* hit_offsets,
                                const int32_t* counts, int64_t* running, cudaStream_t stream)
{
    k_offset_fixup<<<kFixupBlocks, 256, 0, stream>>>(track_offsets, n_events, hit_offsets, counts, running);
    return cudaGetLastError();
}

cudaError_t launch_debug_phi16(const float* x, const float* y, int32_t n, uint16_t* out,
                               cudaStream_t stream)
{
    if (n > 0) k_debug_phi16<<<(n + 255) / 256, 256, 0, stream>>>(x, y, n, out);
    return cudaGetLastError();
}

}  // namespace sbt
