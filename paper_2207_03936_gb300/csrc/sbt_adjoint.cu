// Adjoint of the consolidation fit with respect to per-module alignment.
//
// Objective: sum over tracks of the least-squares residual sum / sigma^2 of
// the straight-line fit (section "Tracklet filter": least-squares fit; the
// same fit is applied to every consolidated track), evaluated on aligned hits
//     h' = Rz(g) Ry(b) Rx(a) (h - c_m) + c_m + (dx, dy, dz),  c_m = (0, 0, z_m).
// At the least-squares optimum the derivative with respect to a hit is the
// partial derivative at fixed line parameters (the parameters are stationary),
//     d chi2 / d h' = 2 / sigma^2 (rx, ry, -(rx tx + ry ty)) = g,
// chained through d h' / d(align_m): g itself for the translations, and
// g . (w x q) = w . (q x g) for a rotation angle, q = R_m (h - c_m) and w the
// axis that the angle turns about: e_z for g, Rz e_y for b, Rz Ry e_x for a
// (dR_m/d angle = [w]x R_m).  So the kernel accumulates per module the force g
// and the torque q x g, and the axes are applied once per module at the end.
//
// Arithmetic is fp64 (the hits are fp32), and the fp64 pipe is the bound: it
// takes two lanes a clock and SM on this GPU, 16 clocks a warp instruction
// whether its lanes are used or not, while 64 other warp instructions issue.
// So every fp64 operation runs on full warps: a block takes tiles of
// consecutive tracks and changes the assignment of threads between phases,
//   hits    one thread per hit: aligned position p and q;
//   tracks  one thread per track, tracks of a tile in order of length: the
//           line, from the positions in shared memory;
//   hits    one thread per hit: residuals, force and torque, stored in order of
//           module (a stable counting sort of the tile's hits, integer work);
//   modules one thread per (module, component): sums into a register that lives
//           over all tiles.
// 62 fp64 warp instructions per 32 hits; one warp per track with its lanes over
// the hits took about 220 (20 of 32 lanes used, shuffled sums, five divisions
// per track).  2.1 M tracks of 20 hits: 17.5 -> 5.4 ms, the fp64 pipe busy 77%
// of the time; three hits a thread and tile (smaller tiles) 11% slower.
//
// A track may have any number of hits and several hits on one module (tracks
// above kTileTrack hits go through a warp each); a track without a
// straight-line fit (fewer than two hits or modules) or with an index out of
// range contributes nothing and is counted as skipped.  Every sum has a fixed
// order (hits of a module in tile order, tiles of a block, blocks), so the
// result is bitwise reproducible.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "sbt_internal.h"

namespace sbt {

constexpr int kAdjThreads = 384;
constexpr int kAdjWarps = kAdjThreads / 32;
constexpr int kAdjPerThread = 4;
constexpr int kTileHits = kAdjThreads * kAdjPerThread;
constexpr int kTileTracks = 128;  // 1536 hits are 77 tracks of average length
constexpr int kTileTrack = 64;    // longest track of a tile (one hit per module at most, of 64)
constexpr int kAdjPerModule = 6;  // force and torque
constexpr int kAdjBlocksPerSM = 2;
static_assert(kAdjPerModule * kMaxModules <= kAdjThreads, "one thread per accumulated component");
static_assert(kTileTracks <= 256 && kMaxModules < 255 && kTileTrack <= kTileHits, "tile indices are bytes");

// Accumulated entries: per module force and torque, then chi2 and the
// skipped-track count.
__host__ __device__ inline int adjoint_entries(int M) { return kAdjPerModule * M + 2; }

// Words per module of the angles' axes, after the blocks' entries.
constexpr int kAdjAxes = 5;

// Blocks of a launch: two per SM, fewer when there are fewer than 32 tracks
// for each (a block's start, the rotation matrices, costs as much as 100
// tracks).
int adjoint_blocks(int sm_count, int n_tracks)
{
    return std::max(1, std::min(kAdjBlocksPerSM * std::max(sm_count, 1), n_tracks / 32 + 1));
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Rotation of a module: R = Rz(g) Ry(b) Rx(a) in R[0..8], then the translation
// with the plane's z added to its last component, sin g and cos g.
constexpr int kAdjMat = 14;

__device__ __forceinline__ void rotation(const double* th, double zc, double* R)
{
    double sa, ca, sb, cb, sg, cg;
    sincos(th[3], &sa, &ca);
    sincos(th[4], &sb, &cb);
    sincos(th[5], &sg, &cg);
    R[0] = cg * cb;
    R[1] = cg * sb * sa - sg * ca;
    R[2] = cg * sb * ca + sg * sa;
    R[3] = sg * cb;
    R[4] = sg * sb * sa + cg * ca;
    R[5] = sg * sb * ca - cg * sa;
    R[6] = -sb;
    R[7] = cb * sa;
    R[8] = cb * ca;
    R[9] = th[0];
    R[10] = th[1];
    R[11] = zc + th[2];
    R[12] = sg;
    R[13] = cg;
}

// Aligned hit: q = R (h - c), p = q + c + t.
struct AHit {
    double px, py, pz, qx, qy, qz;
};

__device__ __forceinline__ AHit aligned_hit(const double* A, double zc, float x, float y, float z)
{
    const double vx = (double)x, vy = (double)y, vz = (double)z - zc;
    AHit a;
    a.qx = A[0] * vx + A[1] * vy + A[2] * vz;
    a.qy = A[3] * vx + A[4] * vy + A[5] * vz;
    a.qz = A[6] * vx + A[7] * vy + A[8] * vz;
    a.px = a.qx + A[9];
    a.py = a.qy + A[10];
    a.pz = a.qz + A[11];
    return a;
}

struct Line {
    double xm, ym, zm, tx, ty;
};

// Squared residual of an aligned hit, and with kGrad its force and torque over
// 2 / sigma^2.
template <bool kGrad>
__device__ __forceinline__ double force_torque(const AHit& a, const Line& l, double* f)
{
    const double dz = a.pz - l.zm;
    const double rx = (a.px - l.xm) - l.tx * dz;
    const double ry = (a.py - l.ym) - l.ty * dz;
    if (!kGrad) return rx * rx + ry * ry;
    const double w = rx * l.tx + ry * l.ty;
    f[0] = rx;
    f[1] = ry;
    f[2] = -w;
    f[3] = -(a.qy * w) - a.qz * ry;
    f[4] = a.qz * rx + a.qx * w;
    f[5] = a.qx * ry - a.qy * rx;
    return rx * rx + ry * ry;
}

struct AdjSmem {
    double tile[6 * kTileHits];   // p and q by hit (six arrays), then forces and torques by module order
    double mats[kAdjMat * kMaxModules];
    double zc[kMaxModules];
    Line line[kTileTracks];
    double warp_chi2[kAdjWarps];
    int first[kTileTracks + 1];   // first tile hit of each track of the tile
    int src[kTileTracks];         // first entry of track_hits of each track
    int start[kMaxModules + 1];   // first hit of each module in module order
    int skipped, n_tile, tile_end, has_long;
    uint16_t before[kTileHits / 32 * kMaxModules];  // hits of a module in the earlier groups of 32
    uint8_t count[kTileHits / 32 * kMaxModules];    // hits of a module in each group of 32
    uint8_t module[kTileHits];    // by tile hit; 255: an index out of range
    uint8_t order[kTileTracks];   // tracks by length
    uint8_t skip[kTileTracks];
    int bins[kTileTrack + 1];
};
static_assert(sizeof(double) * kAdjWarps * kAdjPerModule * kMaxModules <= sizeof(AdjSmem::tile),
              "the long tracks' accumulators fit the tile");

// One track above kTileTrack hits by one warp, lanes over its hits in rounds of
// 32, positions recomputed in each pass; `my`: the warp's accumulators [6 M].
template <bool kGrad>
__device__ void long_track(const Inputs& in, const AdjSmem& S, int M, const int32_t* hits, int n, double* my,
                           double& chi2, int& skipped)
{
    const int lane = threadIdx.x & 31;
    auto hit_at = [&](int j, int& m) {
        const int h = hits[j];
        m = in.module[h];
        return aligned_hit(S.mats + kAdjMat * m, S.zc[m], in.x[h], in.y[h], in.z[h]);
    };
    bool bad = false;
    int mlo = INT32_MAX, mhi = -1;
    for (int j = lane; j < n; j += 32) {
        const int h = hits[j];
        const int m = h >= 0 && h < in.n_hits ? in.module[h] : -1;
        bad |= m < 0 || m >= M;
        mlo = min(mlo, m);
        mhi = max(mhi, m);
    }
    bad = __any_sync(0xFFFFFFFFu, bad);
    mlo = __reduce_min_sync(0xFFFFFFFFu, mlo);
    mhi = __reduce_max_sync(0xFFFFFFFFu, mhi);
    if (bad || mlo == mhi) {
        if (lane == 0) skipped++;
        return;
    }
    int m;
    double sx = 0, sy = 0, sz = 0;
    for (int j = lane; j < n; j += 32) {
        const AHit a = hit_at(j, m);
        sx += a.px;
        sy += a.py;
        sz += a.pz;
    }
    Line l;
    l.xm = warp_sum(sx) / n;
    l.ym = warp_sum(sy) / n;
    l.zm = warp_sum(sz) / n;
    double szz = 0, szx = 0, szy = 0;
    for (int j = lane; j < n; j += 32) {
        const AHit a = hit_at(j, m);
        const double dz = a.pz - l.zm;
        szz += dz * dz;
        szx += dz * (a.px - l.xm);
        szy += dz * (a.py - l.ym);
    }
    szz = warp_sum(szz);
    l.tx = warp_sum(szx) / szz;
    l.ty = warp_sum(szy) / szz;
    for (int base = 0; base < n; base += 32) {
        const int j = base + lane;
        double f[kAdjPerModule];
        m = -1 - lane;  // distinct for inactive lanes
        if (j < n) chi2 += force_torque<kGrad>(hit_at(j, m), l, f);
        if (!kGrad) continue;
        // lanes that share a module add in lane order: each in the turn of its
        // rank among them (a turn for every lane: 20000 tracks of 160 hits with
        // eight hits a module 1638 us, now 636)
        const int rank = __popc(__match_any_sync(0xFFFFFFFFu, m) & ((1u << lane) - 1u));
        const int turns = __reduce_max_sync(0xFFFFFFFFu, rank) + 1;
        for (int turn = 0; turn < turns; turn++) {
            if (j < n && turn == rank)
                for (int k = 0; k < kAdjPerModule; k++) my[kAdjPerModule * m + k] += f[k];
            __syncwarp();
        }
    }
}

// kGrad false: the value alone, without forces, torques and their order by module
// (2 M tracks of 20 hits 4.76 ms, 3.42 without; 20000 tracks of 160 hits 636 and
// 500 us).
template <bool kGrad>
__global__ void __launch_bounds__(kAdjThreads, kAdjBlocksPerSM)
k_adjoint(DevConfig C, Inputs in, const int32_t* hit_offsets, const int32_t* track_hits, int32_t n_tracks,
          const double* align, double* partial)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AdjSmem& S = *(AdjSmem*)smem_raw;
    const int M = C.M;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < M) {
        double* A = S.mats + kAdjMat * tid;
        S.zc[tid] = (double)C.module_z[tid];
        rotation(align + 6 * tid, S.zc[tid], A);
        if (kGrad && blockIdx.x == 0) {  // the axes of the angles, for the reduction
            double* x = partial + (int64_t)gridDim.x * adjoint_entries(M) + kAdjAxes * tid;
            x[0] = A[0];  // Rz Ry e_x: the first column of R
            x[1] = A[3];
            x[2] = A[6];
            x[3] = -A[12];  // Rz e_y = (-sin g, cos g, 0)
            x[4] = A[13];
        }
    }
    if (tid == 0) {
        S.skipped = 0;
        S.has_long = 0;
    }
    __syncthreads();
    const int64_t end = n_tracks > 0 ? hit_offsets[n_tracks] : 0;
    const int tbeg = (int)((int64_t)n_tracks * blockIdx.x / gridDim.x);
    const int tend = (int)((int64_t)n_tracks * (blockIdx.x + 1) / gridDim.x);
    double acc = 0.0, chi2 = 0.0;  // this thread's (module, component), and its hits' squared residuals
    int skipped = 0;
    int t0 = tbeg;
    while (t0 < tend) {
        // the tile: the next tracks whose hits fit, at most kTileTracks of
        // them (scan over four warps); skipped and long ones take no room
        if (tid < kTileTracks) {
            const int t = t0 + tid;
            int n = 0, h0 = 0;
            if (t < tend) {
                h0 = hit_offsets[t];
                n = hit_offsets[t + 1] - h0;
                const bool bad = n < 2 || h0 < 0 || (int64_t)h0 + n > end;
                if (!bad && n > kTileTrack) S.has_long = 1;
                if (bad || n > kTileTrack) n = bad ? -1 : 0;
            }
            S.skip[tid] = n < 0;
            n = max(n, 0);
            S.src[tid] = h0;
            int incl = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += v;
            }
            S.first[tid + 1] = incl;
        }
        if (tid <= kTileTrack) S.bins[tid] = 0;
        __syncthreads();
        int before = 0;
        if (tid < kTileTracks)
            for (int w = 0; w < warp; w++) before += S.first[32 * w + 32];
        __syncthreads();
        if (tid < kTileTracks) {
            const int e = S.first[tid + 1] + before;
            const int b = __shfl_up_sync(0xFFFFFFFFu, e, 1);
            const int s = lane > 0 ? b : before;
            // tracks that fit form a prefix
            S.first[tid + 1] = e;
            if (t0 + tid < tend && e <= kTileHits) {
                atomicAdd(&S.bins[kTileTrack - (e - s)], 1);
                if (S.skip[tid]) skipped++;
            }
            if (tid == 0) S.first[0] = 0;
        }
        __syncthreads();
        if (tid < kTileTracks) {
            const bool fits = t0 + tid < tend && S.first[tid + 1] <= kTileHits;
            const bool next = tid + 1 < kTileTracks && t0 + tid + 1 < tend && S.first[min(tid + 2, kTileTracks)] <= kTileHits;
            if (fits && !next) {
                S.n_tile = tid + 1;
                S.tile_end = S.first[tid + 1];
            }
        }
        if (tid == 0)  // longest tracks first
            for (int k = 0, s = 0; k <= kTileTrack; k++) {
                const int c = S.bins[k];
                S.bins[k] = s;
                s += c;
            }
        if (kGrad)
            for (int k = tid; k < kTileHits / 32 * M; k += kAdjThreads) S.count[k] = 0;
        __syncthreads();
        const int nt = S.n_tile, nh = S.tile_end;
        if (tid < nt) S.order[atomicAdd(&S.bins[kTileTrack - (S.first[tid + 1] - S.first[tid])], 1)] = (uint8_t)tid;
        // hits: track, module, aligned position, rank within the module's hits
        // of this group of 32
        uint32_t mine[kAdjPerThread];  // module | track << 8 | rank << 16; module 255: no hit
#pragma unroll
        for (int u = 0; u < kAdjPerThread; u++) {
            const int h = tid + u * kAdjThreads;
            int m = 255, tr = 0;
            if (h < nh) {
                int hi = nt;  // last track that starts at or before h and is not empty
                while (hi - tr > 1) {
                    const int mid = (tr + hi) >> 1;
                    if (S.first[mid] <= h)
                        tr = mid;
                    else
                        hi = mid;
                }
                const int i = track_hits[S.src[tr] + (h - S.first[tr])];
                if (i >= 0 && i < in.n_hits) {
                    const int mm = in.module[i];
                    if (mm >= 0 && mm < M) m = mm;
                }
                S.module[h] = (uint8_t)m;
                if (m != 255) {
                    const AHit a = aligned_hit(S.mats + kAdjMat * m, S.zc[m], in.x[i], in.y[i], in.z[i]);
                    S.tile[0 * kTileHits + h] = a.px;
                    S.tile[1 * kTileHits + h] = a.py;
                    S.tile[2 * kTileHits + h] = a.pz;
                    if (kGrad) {
                        S.tile[3 * kTileHits + h] = a.qx;
                        S.tile[4 * kTileHits + h] = a.qy;
                        S.tile[5 * kTileHits + h] = a.qz;
                    }
                }
            }
            int rank = 0;
            if (kGrad) {
                const unsigned same = __match_any_sync(0xFFFFFFFFu, m);
                rank = __popc(same & ((1u << lane) - 1u));
                if (m != 255 && rank == 0) S.count[(h >> 5) * M + m] = (uint8_t)__popc(same);
            }
            mine[u] = (uint32_t)m | ((uint32_t)tr << 8) | ((uint32_t)rank << 16);
        }
        __syncthreads();
        // tracks: the line (tid < nt); modules: hits before each group (the
        // last warps, integer work beside the fp64 of the first)
        if (tid < nt) {
            const int tr = S.order[tid];
            const int b = S.first[tr], n = S.first[tr + 1] - b;
            bool bad = false, one = true;
            const double* P = S.tile + b;
            // Moments about a point near the mean, their mean part taken out at
            // the end: the fp32 mean is that point (any point gives the same
            // line), so the fp64 pipe takes no sums of positions, and the means
            // carry the rounding of micrometres instead of that of metres.
            // Gradient error against 128-bit sums, over that of a tree of sums:
            // 0.92 / 0.94 / 0.98 / 0.99 at 1 / 8 / 60 / 400 events, 1.00 at 2000
            // and 10000 (the rounding of the rotations, common to both); sums of
            // positions in fp64, by fours, 1.09 / 1.07 / 1.03 / 1.01 (10000
            // events 5154 us, here 5363), their means corrected by the sums of
            // differences 0.92 / 0.93 / 0.98 / 0.99 (5517 us).
            float sx = 0, sy = 0, sz = 0;
#pragma unroll 4
            for (int j = 0; j < n; j++) {
                bad |= S.module[b + j] == 255;
                one &= S.module[b + j] == S.module[b];
                sx += (float)P[0 * kTileHits + j];
                sy += (float)P[1 * kTileHits + j];
                sz += (float)P[2 * kTileHits + j];
            }
            if (n > 0 && (bad || one)) {
                S.skip[tr] = 1;
                skipped++;
            } else if (n > 0) {
                Line l;
                const float inv = 1.0f / (float)n;
                const auto near_mean = [&](float sum, const double* v) {
                    if (isfinite(sum)) return (double)(sum * inv);
                    double s = 0;  // beyond fp32, or not finite: as it is in fp64
                    for (int j = 0; j < n; j++) s += v[j];
                    return s / n;
                };
                l.xm = near_mean(sx, P);
                l.ym = near_mean(sy, P + kTileHits);
                l.zm = near_mean(sz, P + 2 * kTileHits);
                double szz = 0, szx = 0, szy = 0, cx = 0, cy = 0, cz = 0;
                for (int j = 0; j < n; j += 4) {
                    double zz = 0, zx = 0, zy = 0;
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        if (j + u < n) {
                            const double dz = P[2 * kTileHits + j + u] - l.zm;
                            const double dx = P[0 * kTileHits + j + u] - l.xm;
                            const double dy = P[1 * kTileHits + j + u] - l.ym;
                            zz += dz * dz;
                            zx += dz * dx;
                            zy += dz * dy;
                            cx += dx;
                            cy += dy;
                            cz += dz;
                        }
                    szz += zz;
                    szx += zx;
                    szy += zy;
                }
                cx /= n;
                cy /= n;
                cz /= n;
                const double szc = cz * n;
                szz -= szc * cz;
                szx -= szc * cx;
                szy -= szc * cy;
                l.tx = szx / szz;
                l.ty = szy / szz;
                l.xm += cx;
                l.ym += cy;
                l.zm += cz;
                S.line[tr] = l;
            }
        }
        if (kGrad && tid >= kAdjThreads - 64 && tid - (kAdjThreads - 64) < M) {
            const int m = tid - (kAdjThreads - 64);
            int s = 0;
#pragma unroll 8
            for (int g = 0; g < kTileHits / 32; g++) {
                S.before[g * M + m] = (uint16_t)s;
                s += S.count[g * M + m];
            }
            S.start[m + 1] = s;
        }
        __syncthreads();
        if (kGrad && warp == 0) {  // module starts, two modules a lane
            const int a = 2 * lane < M ? S.start[2 * lane + 1] : 0, b = 2 * lane + 1 < M ? S.start[2 * lane + 2] : 0;
            int incl = a + b;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= o) incl += v;
            }
            if (2 * lane < M) S.start[2 * lane + 1] = incl - b;
            if (2 * lane + 1 < M) S.start[2 * lane + 2] = incl;
            if (lane == 0) S.start[0] = 0;
        }
        // hits: forces and torques, kept in registers until every position is
        // read, then stored in module order over the positions
        double f[kAdjPerThread][kAdjPerModule];
#pragma unroll
        for (int u = 0; u < kAdjPerThread; u++) {
            const int h = tid + u * kAdjThreads;
            const int tr = (int)(mine[u] >> 8) & 0xFF;
#pragma unroll
            for (int k = 0; k < kAdjPerModule; k++) f[u][k] = 0.0;
            if ((mine[u] & 0xFFu) != 255u && !S.skip[tr]) {
                AHit a;
                a.px = S.tile[0 * kTileHits + h];
                a.py = S.tile[1 * kTileHits + h];
                a.pz = S.tile[2 * kTileHits + h];
                if (kGrad) {
                    a.qx = S.tile[3 * kTileHits + h];
                    a.qy = S.tile[4 * kTileHits + h];
                    a.qz = S.tile[5 * kTileHits + h];
                }
                chi2 += force_torque<kGrad>(a, S.line[tr], f[u]);
            }
        }
        if (kGrad) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kAdjPerThread; u++) {
                const int h = tid + u * kAdjThreads;
                const int m = (int)(mine[u] & 0xFFu);
                if (m != 255) {
                    const int s = S.start[m] + S.before[(h >> 5) * M + m] + (int)(mine[u] >> 16);
#pragma unroll
                    for (int k = 0; k < kAdjPerModule; k++) S.tile[kAdjPerModule * s + k] = f[u][k];
                }
            }
            __syncthreads();
            if (tid < kAdjPerModule * M) {
                const int m = tid / kAdjPerModule, k = tid % kAdjPerModule;
                const int e = S.start[m + 1];
                for (int s = S.start[m]; s < e; s++) acc += S.tile[kAdjPerModule * s + k];
            }
        }
        t0 += nt;
        __syncthreads();
    }
    if (S.has_long) {
        if (kGrad)
            for (int k = tid; k < kAdjWarps * kAdjPerModule * M; k += kAdjThreads) S.tile[k] = 0.0;
        __syncthreads();
        for (int t = tbeg + warp; t < tend; t += kAdjWarps) {
            const int h0 = hit_offsets[t], n = hit_offsets[t + 1] - h0;
            if (n > kTileTrack && h0 >= 0 && (int64_t)h0 + n <= end)
                long_track<kGrad>(in, S, M, track_hits + h0, n, S.tile + warp * kAdjPerModule * M, chi2, skipped);
        }
        __syncthreads();
        if (kGrad && tid < kAdjPerModule * M)
            for (int w = 0; w < kAdjWarps; w++) acc += S.tile[w * kAdjPerModule * M + tid];
    }
    // the block's entries
    const int P = adjoint_entries(M);
    if (skipped) atomicAdd(&S.skipped, skipped);
    chi2 = warp_sum(chi2);
    if (lane == 0) S.warp_chi2[warp] = chi2;
    __syncthreads();
    double* out = partial + (int64_t)blockIdx.x * P;
    const double s2 = (double)C.sigma * (double)C.sigma;
    if (kGrad && tid < kAdjPerModule * M) out[tid] = acc * (2.0 / s2);
    if (tid == 0) {
        double c = 0.0;
        for (int w = 0; w < kAdjWarps; w++) c += S.warp_chi2[w];
        out[P - 2] = c / s2;
        out[P - 1] = (double)S.skipped;
    }
}

// Sum of the blocks' entries in a fixed order, one block for chi2 and the skipped
// count and, with a gradient, one per module: 64 threads per entry over the blocks, then
// a tree.  The translation gradient is the summed force, each rotation
// gradient the torque along the angle's axis.
constexpr int kAdjRows = 64;

__global__ void __launch_bounds__(8 * kAdjRows)
k_adjoint_reduce(int M, int blocks, const double* partial, double* chi2_sum, double* grad, int32_t* skipped)
{
    __shared__ double s[kAdjRows][8];
    const int P = adjoint_entries(M);
    const int m = blockIdx.x == 0 ? M : blockIdx.x - 1, k = threadIdx.x & 7, row = threadIdx.x >> 3;
    const int n = m < M ? kAdjPerModule : 2;
    double v = 0.0;
    if (k < n)
        for (int b = row; b < blocks; b += kAdjRows) v += partial[(int64_t)b * P + kAdjPerModule * m + k];
    s[row][k] = v;
    __syncthreads();
    for (int o = kAdjRows / 2; o > 0; o >>= 1) {
        if (row < o) s[row][k] += s[row + o][k];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    const double* a = s[0];
    if (m == M) {
        *chi2_sum = a[0];
        if (skipped) *skipped = (int32_t)a[1];
    } else {
        double* g = grad + 6 * m;
        g[0] = a[0];
        g[1] = a[1];
        g[2] = a[2];
        const double* x = partial + (int64_t)blocks * P + kAdjAxes * m;
        g[3] = x[0] * a[3] + x[1] * a[4] + x[2] * a[5];
        g[4] = x[3] * a[3] + x[4] * a[4];
        g[5] = a[5];  // e_z
    }
}

size_t adjoint_partial_entries(int M, int blocks)
{
    return (size_t)blocks * (size_t)adjoint_entries(M) + (size_t)kAdjAxes * M;
}

cudaError_t launch_adjoint(const DevConfig& C, const Inputs& in, const int32_t* hit_offsets,
                           const int32_t* track_hits, int32_t n_tracks, const double* align,
                           double* chi2_sum, double* grad, int32_t* skipped, const AdjointWork& W,
                           cudaStream_t stream)
{
    auto kern = grad ? k_adjoint<true> : k_adjoint<false>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(AdjSmem));
    if (err != cudaSuccess) return err;
    kern<<<W.blocks, kAdjThreads, sizeof(AdjSmem), stream>>>(C, in, hit_offsets, track_hits, n_tracks, align,
                                                             W.partial);
    k_adjoint_reduce<<<grad ? C.M + 1 : 1, 8 * kAdjRows, 0, stream>>>(C.M, W.blocks, W.partial, chi2_sum, grad, skipped);
    return cudaGetLastError();
}

}  // namespace sbt
