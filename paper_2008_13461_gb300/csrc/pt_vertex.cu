// Pixel vertices (Sec. 3.6): clusters of tracks in z0, the z of each
// track's point of closest approach to the beam line.
//
// Tracks are eligible when kept by the ambiguity resolution, with at least
// min_hits hits, pT > pt_min, 0 < ez0 < ez0_max and a finite z0.  Two tracks
// i, j of an event are compatible when dz = z0_i - z0_j satisfies
// |dz| < dz_cut and dz^2 < chi2_max (ez0_i^2 + ez0_j^2).  A track's density
// rho is 1 + the number of tracks compatible with it; each track links to the
// nearest compatible track (smallest |dz|, then smaller z0, then smaller
// index) of higher rank (larger rho, or equal rho and smaller z0, or equal
// rho and z0 and smaller index: ties go by z0 first, so the result does not
// depend on the order of the tracks unless two share a z0); the links end at roots
// (ranks grow along them, so there are no cycles), and a root with rho > 1
// seeds a candidate made of every track whose links lead to it.  Candidates
// with at least min_tracks tracks become vertices: z the mean of z0 weighted
// by 1/ez0^2, ez = 1/sqrt(sum of weights), chi2 = sum w (z0 - z)^2, ndf =
// n - 1.  A vertex with chi2/ndf > split_chi2 is split by 2-means in z
// (centres from the tracks below / at-or-above z, each track to the nearer
// centre, ties to the lower one, until no assignment changes, at most 20
// rounds) when both parts keep min_tracks tracks.  The vertices of an event
// are ordered by the sum of pT^2 of their tracks, largest first.
//
// Cuts compare float32 values rounded as written (no contraction); sums and
// the vertex quantities are float64, converted to float32 on output.
//
// GPU form: a counting sort groups the eligible tracks by event; one block of
// 1024 threads per event then sorts its tracks by (z0, index) in shared
// memory, so that every track's compatible tracks lie in a window around it;
// densities and links come from window scans (two threads per track, one to
// each side), roots from pointer jumping, candidates from a counting sort of
// the tracks by root.  With few tracks per event that block does all of it
// (k_vtx_group); with many on average the window scans of all events run
// over every SM in between (k_vtx_sort, k_vtx_density, k_vtx_link,
// k_vtx_roots).  The sort by z0 is a counting sort too (by z0 tile, a
// tile's few entries ranked by comparing them with each other); where a tile
// is crowded a bitonic sort takes over.  The candidates' fits and 2-means splits, the
// float64 part, then run one warp per candidate over the candidates of all
// events at once (shuffle reductions), so that every SM takes part; a last
// block per event orders its vertices and labels their tracks.
#include "pt_common.cuh"
#include "pt_kernels.cuh"

namespace ptk {
namespace {

constexpr int kVtxMax = PT_VTX_MAX_TRACKS;   // eligible tracks per event (sorted in shared memory)
constexpr int kPosBits = 14;                 // bits of a sorted position
constexpr int kPosMask = kVtxMax - 1;
constexpr int kSideBit = 30;                 // 2-means side of a member, kept in its key
constexpr int kVtxCap = PT_VTX_MAX_VERTICES; // vertex candidates / vertices per event
constexpr int kVtxThreads = 1024;
constexpr int kZTiles = 4096;                // z0 tiles of the counting sort, over +-kZHalf
constexpr float kZHalf = 24.0f;              //   (beyond, the outermost tiles)
constexpr int kVtxSplit = 10000;             // tracks per event from which the windows run over all SMs
constexpr int kCrowd = 256;                  // entries of a tile that are still ranked pairwise
constexpr size_t kVtxDynSmem = sizeof(int32_t) * (3 * kVtxMax + kZTiles);
constexpr int kKmeansRounds = 20;
constexpr unsigned kFull = 0xffffffffu;

static_assert((1 << kPosBits) == kVtxMax, "sorted positions must fit their key field");

struct VtxArgs {
    int32_t n_tracks, n_events, max_vertices;
    pt_vertex_tracks in;
    pt_vertex_cuts cuts;
    // scratch; arrays "by sorted position" hold each event's tracks at its ev_off
    int32_t *ev_off, *ev_cur, *order, *rho, *root;   // order: key before its groups are put
                                                     //   in order, then ~vertex of each member
    float4 *rec;                     // (z0, ez0, track index as int bits, -), grouped by event
    double2 *wz;                     // (1 / ez0^2, z0) in float64 by sorted position (in rec's place: each
                                     //   event's records are used up when its first weight is written)
    float2 *ze;                      // (z0, ez0) by sorted position
    int32_t *key;                    // sorted positions grouped by root; the members of the candidates
    int32_t *sid;                    // track index by sorted position
    int32_t *nc, *nv;                // per event: candidates, provisional vertices
    int32_t *cq, *cn;                // per event and candidate (kVtxCap each): first key, members
    double *vz, *vsp;                // per event and provisional vertex (kVtxCap each): z, sum of pT^2
    float *vez, *vc2;                //   its error and chi2
    int32_t *vnt, *vkey;             //   its tracks and (2 * first key + part)
    pt_vertices out;
};

__device__ __forceinline__ bool eligible(const VtxArgs &a, int i) {
    const float e = a.in.ez0[i], z = a.in.z0[i];
    const int ev = a.in.ev[i];
    return (!a.in.keep || a.in.keep[i]) && (int)a.in.nhits[i] >= a.cuts.min_hits && a.in.pt[i] > a.cuts.pt_min &&
           e > 0.f && e < a.cuts.ez0_max && fabsf(z) <= 3.402823466e38f && ev >= 0 && ev < a.n_events;
}

__device__ __forceinline__ void set_status(const VtxArgs &a, int bit) { atomicOr(a.out.status, bit); }

// Tracks of one event are mostly consecutive, so the per-event atomics are
// aggregated over the lanes of a warp that share an event.
__global__ void __launch_bounds__(kThreads) k_vtx_count(VtxArgs a) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < a.n_tracks; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + lane;
        const bool ok = i < a.n_tracks && eligible(a, i);
        if (i < a.n_tracks) a.out.track_vertex[i] = -1;
        const int e = ok ? a.in.ev[i] : -1;
        const unsigned grp = __match_any_sync(kFull, e);
        if (ok && lane == __ffs(grp) - 1) atomicAdd(a.ev_off + e, __popc(grp));
    }
}

__global__ void __launch_bounds__(kThreads) k_vtx_fill(VtxArgs a) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    for (int i0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < a.n_tracks; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + lane;
        const bool ok = i < a.n_tracks && eligible(a, i);
        const int e = ok ? a.in.ev[i] : -1;
        const unsigned grp = __match_any_sync(kFull, e);
        const int leader = __ffs(grp) - 1;
        int slot = 0;
        if (ok && lane == leader) slot = atomicAdd(a.ev_cur + e, __popc(grp));
        slot = __shfl_sync(kFull, slot, leader) + __popc(grp & ((1u << lane) - 1u));
        if (ok) a.rec[a.ev_off[e] + slot] = make_float4(a.in.z0[i], a.in.ez0[i], __int_as_float(i), 0.f);
    }
}

// the chi2 half of the compatibility of a track (squared error ep2) with a
// track of error eq at distance dz: dz^2 < chi2_max (ep2 + eq^2)
__device__ __forceinline__ bool chi2_ok(float dz, float ep2, float eq, float c2m) {
    return __fmul_rn(dz, dz) < __fmul_rn(c2m, __fadd_rn(ep2, __fmul_rn(eq, eq)));
}

// Warp-wide sums (every lane ends with the same bits).  The float64 pipe
// takes ~19 cycles for one instruction of a warp, so four sums share their
// additions: after each of the first two exchanges a lane carries on half of
// them, in the same pairing of lanes as a butterfly for each alone.
__device__ __forceinline__ int warp_sum(int v) { return __reduce_add_sync(kFull, v); }

__device__ __forceinline__ void warp_sum4(double &a, double &b, double &c, double &d) {
    const int lane = threadIdx.x & 31;
    const bool h16 = lane & 16, h8 = lane & 8;
    // lanes with bit 16 clear keep a, b; the others c, d
    double x = (h16 ? c : a) + __shfl_xor_sync(kFull, h16 ? a : c, 16);
    double y = (h16 ? d : b) + __shfl_xor_sync(kFull, h16 ? b : d, 16);
    // bit 8 clear: the first of the two; set: the second
    double v = (h8 ? y : x) + __shfl_xor_sync(kFull, h8 ? x : y, 8);
    for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    a = __shfl_sync(kFull, v, 0);
    b = __shfl_sync(kFull, v, 8);
    c = __shfl_sync(kFull, v, 16);
    d = __shfl_sync(kFull, v, 24);
}

__device__ __forceinline__ void warp_sum2(double &a, double &b) {
    const bool h16 = threadIdx.x & 16;
    double v = (h16 ? b : a) + __shfl_xor_sync(kFull, h16 ? a : b, 16);
    for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    a = __shfl_sync(kFull, v, 0);
    b = __shfl_sync(kFull, v, 16);
}

// a / b and c / d in one division's instructions
__device__ __forceinline__ void warp_div2(double a, double b, double c, double d, double &q0, double &q1) {
    const bool h16 = threadIdx.x & 16;
    const double q = (h16 ? c : a) / (h16 ? d : b);
    q0 = __shfl_sync(kFull, q, 0);
    q1 = __shfl_sync(kFull, q, 16);
}

// The members of a candidate, lane k mod 32 holding member k: weight and z0
// (wz: in float64 by sorted position, computed once per track) and the side
// of a partition.  Up to 32 kMemCache of them stay in registers, so that
// the rounds of a 2-means split wait for no loads; in a larger candidate
// they are read again each time and the sides are kept in the keys' side
// bits (mk).
constexpr int kMemCache = 8;

struct Sides {
    double sw0, swz0, sw1, swz1;
    int n1;
};

struct Members {
    int32_t *mk;
    const double2 *wz;
    int n;
    bool cached;
    double2 v[kMemCache];
    unsigned side;

    // f(member, weight and z0, side) -> side, for every member of the lane
    template <class F>
    __device__ __forceinline__ void each(F f) {
        const int lane = threadIdx.x & 31;
        if (cached) {
#pragma unroll
            for (int i = 0; i < kMemCache; i++) {
                if (32 * i >= n) break;
                if (lane + 32 * i < n) {
                    const unsigned u = f(lane + 32 * i, v[i], (int)((side >> i) & 1));
                    side = (side & ~(1u << i)) | u << i;
                }
            }
        } else {
            for (int k = lane; k < n; k += 32) {
                const int32_t kk = mk[k];
                const int u = f(k, wz[kk & kPosMask], (kk >> kSideBit) & 1);
                mk[k] = (kk & ~(1 << kSideBit)) | (u << kSideBit);
            }
        }
    }

    __device__ __forceinline__ Sides sums() {
        Sides s = {0.0, 0.0, 0.0, 0.0, 0};
        each([&](int, const double2 &m, int u) {
            if (u) {
                s.sw1 += m.x;
                s.swz1 += m.x * m.y;
                s.n1++;
            } else {
                s.sw0 += m.x;
                s.swz0 += m.x * m.y;
            }
            return u;
        });
        warp_sum4(s.sw0, s.swz0, s.sw1, s.swz1);
        s.n1 = warp_sum(s.n1);
        return s;
    }

    // chi2 of the members on side sel about z, and the sum of their pT^2
    // (pt(k): member k's pT); sel < 0: every member
    template <class Pt>
    __device__ __forceinline__ void chi2_pt2(int sel, double z, Pt pt, double &chi2, double &pt2) {
        double c = 0.0, p = 0.0;
        each([&](int k, const double2 &m, int u) {
            if (sel < 0 || u == sel) {
                const double d = m.y - z, t = pt(k);
                c += m.x * d * d;
                p += t * t;
            }
            return u;
        });
        warp_sum2(c, p);
        chi2 = c;
        pt2 = p;
    }
};

// sort element: z0 and record, in order of (z0, track index)
struct ZRec {
    float z;
    int rec;
};
__device__ __forceinline__ int track_of(const float4 *rec, int r) { return r < kVtxMax ? __float_as_int(rec[r].z) : r; }
__device__ __forceinline__ bool elem_gt(const ZRec &a, const ZRec &b, const float4 *rec) {
    return a.z > b.z || (a.z == b.z && track_of(rec, a.rec) > track_of(rec, b.rec));
}

// z0 tile: monotone in z0 (the track's place among equal tiles is found by
// comparing the values)
__device__ __forceinline__ int z_tile(float z) {
    return min(max((int)((z + kZHalf) * (kZTiles / (2.0f * kZHalf))), 0), kZTiles - 1);
}

// Exclusive prefix sums of a[0, n) in place (the whole block), and whether
// any entry was above kCrowd.  warp: 32 ints.
__device__ __forceinline__ bool block_starts(int32_t *a, int n, int32_t *warp) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, per = (n + kVtxThreads - 1) / kVtxThreads;
    const int i0 = min((int)threadIdx.x * per, n), i1 = min(i0 + per, n);
    int sum = 0;
    bool crowded = false;
    for (int i = i0; i < i1; i++) {
        sum += a[i];
        crowded |= a[i] > kCrowd;
    }
    int incl = sum;
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += t;
    }
    if (lane == 31) warp[w] = incl;
    __syncthreads();
    if (w == 0) {
        const int v = warp[lane];
        int x = v;
        for (int d = 1; d < 32; d <<= 1) {
            const int t = __shfl_up_sync(kFull, x, d);
            if (lane >= d) x += t;
        }
        warp[lane] = x - v;
    }
    __syncthreads();
    int run = warp[w] + incl - sum;
    for (int i = i0; i < i1; i++) {
        const int v = a[i];
        a[i] = run;
        run += v;
    }
    return __syncthreads_or(crowded) != 0;
}

// Ascending bitonic sort of P entries (P a power of two, at least 32; the
// block a multiple of 32 threads); padding entries have records from kVtxMax
// on and an infinite z0.  Position p is handled by thread p mod
// blockDim, so the partners of the stages at distance 16 or less are lanes
// of one warp: those stages of each merge run in registers with shuffles,
// one barrier per merge instead of one per stage.
__device__ __forceinline__ void bitonic(int P, float *sz, int32_t *srec, const float4 *rec) {
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j >= 32; j >>= 1) {
            for (int p = threadIdx.x; p < P; p += blockDim.x) {
                const int q = p ^ j;
                if (q > p) {
                    const ZRec a = {sz[p], srec[p]}, b = {sz[q], srec[q]};
                    if (elem_gt(a, b, rec) == ((p & k) == 0)) {
                        sz[p] = b.z;
                        srec[p] = b.rec;
                        sz[q] = a.z;
                        srec[q] = a.rec;
                    }
                }
            }
            __syncthreads();
        }
        // whole warps take part: P and blockDim are multiples of 32
        for (int p = threadIdx.x; p < P; p += blockDim.x) {
            ZRec e = {sz[p], srec[p]};
            const bool up = (p & k) == 0;
            for (int j = min(k >> 1, 16); j > 0; j >>= 1) {
                const ZRec o = {__shfl_xor_sync(kFull, e.z, j), __shfl_xor_sync(kFull, e.rec, j)};
                // the lower of a pair keeps the smaller entry in an ascending
                // run and the larger in a descending one
                if (((p & j) == 0) == up ? elem_gt(e, o, rec) : elem_gt(o, e, rec)) e = o;
            }
            sz[p] = e.z;
            srec[p] = e.rec;
        }
        __syncthreads();
    }
}

// Densities: the compatible tracks of the track at position p of an event's
// sorted tracks [0, cnt) lie in the window |z0 - z0_p| < dz_cut (rounded
// differences are monotonic along the sorted order); those on one side.
template <class Z, class Ez>
__device__ __forceinline__ int side_density(int p, int dir, int cnt, Z z, Ez ez, float dzc, float c2m) {
    const float zp = z(p), ep = ez(p), ep2 = __fmul_rn(ep, ep);
    int r = 0;
    for (int q = p + dir; q >= 0 && q < cnt; q += dir) {
        const float dz = __fsub_rn(zp, z(q));
        if (!(fabsf(dz) < dzc)) break;
        r += chi2_ok(dz, ep2, ez(q), c2m);
    }
    return r;
}

// Links: the nearest compatible track of higher rank on one side (-1: none)
// and its distance; the sorted position orders equal densities and equal
// distances by (z0, index).
template <class Z, class Ez, class Rho>
__device__ __forceinline__ int side_link(int p, int dir, int cnt, Z z, Ez ez, Rho rho, float dzc, float c2m, float &bd) {
    const float zp = z(p), ep = ez(p), ep2 = __fmul_rn(ep, ep);
    const int rp = rho(p);
    int best = -1;
    bd = __int_as_float(0x7f800000);
    for (int q = p + dir; q >= 0 && q < cnt; q += dir) {
        const float dz = __fsub_rn(zp, z(q)), ad = fabsf(dz);
        // distances do not shrink along the window, so nothing nearer
        // follows; at an equal one the smaller position wins
        if (!(ad < dzc) || ad > bd) break;
        const int rq = rho(q);
        if (!(rq > rp || (rq == rp && q < p))) continue;
        if (!chi2_ok(dz, ep2, ez(q), c2m)) continue;
        if (best < 0 || q < best) best = q;
        bd = ad;
    }
    return best;
}

// the nearer of the two sides' links of a track, whose lanes are neighbours
__device__ __forceinline__ int join_sides(int best, float bd) {
    const int ob = __shfl_xor_sync(kFull, best, 1);
    const float od = __shfl_xor_sync(kFull, bd, 1);
    return ob >= 0 && (best < 0 || od < bd || (od == bd && ob < best)) ? ob : best;
}

__device__ __forceinline__ double2 weight_and_z(float2 ze) {
    const double e = ze.y;
    return make_double2(1.0 / (e * e), (double)ze.x);
}

// Densities (kLinks = false; and the fits' weights) or links (true) of the
// sorted tracks of all events, over every SM: two neighbouring lanes take a
// track, one to each side.
template <bool kLinks>
__global__ void __launch_bounds__(kThreads) k_vtx_window(VtxArgs a) {
    pdl_enter();
    const int total = a.ev_off[a.n_events];
    const float dzc = a.cuts.dz_cut, c2m = a.cuts.chi2_max;
    const int64_t items = (2 * (int64_t)total + 31) & ~31;
    for (int64_t it = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; it < items; it += (int64_t)gridDim.x * blockDim.x) {
        const int g = (int)(it >> 1), dir = (it & 1) ? 1 : -1;
        bool ok = g < total;
        int base = 0, cnt = 0;
        if (ok) {
            int lo = 0, hi = a.n_events - 1;                 // the event of position g
            while (lo < hi) {
                const int m = (lo + hi + 1) >> 1;
                if (__ldg(a.ev_off + m) <= g) lo = m;
                else hi = m - 1;
            }
            base = __ldg(a.ev_off + lo);
            cnt = __ldg(a.ev_off + lo + 1) - base;
            ok = cnt <= kVtxMax;                             // (a larger one was not sorted)
        }
        const float2 *ze = a.ze + base;
        int *rho = a.rho + base;
        const auto z = [&](int q) { return ze[q].x; };
        const auto ez = [&](int q) { return ze[q].y; };
        if (!kLinks) {
            int r = ok ? side_density(g - base, dir, cnt, z, ez, dzc, c2m) : 0;
            r += __shfl_xor_sync(kFull, r, 1);
            if (ok && dir > 0) rho[g - base] = 1 + r;
            if (ok && dir < 0) a.wz[g] = weight_and_z(ze[g - base]);
        } else {
            float bd = 0.f;
            int best = ok ? side_link(g - base, dir, cnt, z, ez, [&](int q) { return rho[q]; }, dzc, c2m, bd) : -1;
            best = join_sides(best, bd);
            if (ok && dir > 0) a.root[g] = best < 0 ? g - base : best;
        }
    }
}

// Per event (one block): sort, densities, links, roots, candidates
// (kVtxAll), or only the sort (kVtxSort) or only the roots and candidates
// (kVtxRoots), the windows in between run by k_vtx_window over every SM.
//
// One SM works on an event, so the length of its chain of phases counts:
// with two bitonic sorts and one thread per track and window, 24 PU200 events
// of 4950 eligible tracks took 381 us and one PU50 event of 449 took 31 us;
// with the counting sorts and two lanes per track 225 and 17 us, and the
// first 106 us with the windows over every SM.
enum VtxPart { kVtxAll, kVtxSort, kVtxRoots };

template <VtxPart kPart>
__global__ void __launch_bounds__(kVtxThreads, 1) k_vtx_group(VtxArgs a) {
    pdl_enter();
    extern __shared__ __align__(16) unsigned char vsm[];
    float *sz = reinterpret_cast<float *>(vsm);                   // z0 by sorted position
    int32_t *sid = reinterpret_cast<int32_t *>(sz + kVtxMax);     // track index by sorted position, then rho
    int32_t *key = sid + kVtxMax;                                 // z0 errors, then roots, then keys
    int32_t *tile = key + kVtxMax;
    __shared__ int s_nc;
    __shared__ int32_t s_warp[32];

    const int e = blockIdx.x, tid = threadIdx.x;
    const int base = a.ev_off[e], cnt = a.ev_off[e + 1] - base;
    if (kPart != kVtxSort && tid == 0) {
        a.nc[e] = 0;
        a.nv[e] = 0;
        s_nc = 0;
    }
    if (cnt > kVtxMax) {                                          // uniform over the block
        if (kPart != kVtxSort && tid == 0) set_status(a, PT_VTX_EVENT_TOO_LARGE);
        return;
    }
    int32_t *gsid = a.sid + base, *root = a.root + base;
    float2 *ze = a.ze + base;
    if constexpr (kPart != kVtxRoots) {
        const float4 *rec = a.rec + base;
        for (int t = tid; t < kZTiles; t += blockDim.x) tile[t] = 0;
        __syncthreads();
        // four records of a thread in flight at a time
        for (int p0 = tid; p0 < cnt; p0 += 4 * kVtxThreads) {
            float z[4];
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (p0 + i * kVtxThreads < cnt) z[i] = rec[p0 + i * kVtxThreads].x;
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (p0 + i * kVtxThreads < cnt) atomicAdd(&tile[z_tile(z[i])], 1);
        }
        __syncthreads();
        auto put = [&](int at, int r) {
            const float4 v = rec[r];
            ze[at] = make_float2(v.x, v.y);
            gsid[at] = __float_as_int(v.z);
        };
        if (!block_starts(tile, kZTiles, s_warp)) {
            // by tile, any order inside (tile[] becomes each tile's end), then
            // every entry's place among its tile's
            for (int p0 = tid; p0 < cnt; p0 += 4 * kVtxThreads) {
                float z[4];
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (p0 + i * kVtxThreads < cnt) z[i] = rec[p0 + i * kVtxThreads].x;
#pragma unroll
                for (int i = 0; i < 4; i++)
                    if (p0 + i * kVtxThreads < cnt) {
                        const int q = atomicAdd(&tile[z_tile(z[i])], 1);
                        sz[q] = z[i];
                        sid[q] = p0 + i * kVtxThreads;
                    }
            }
            __syncthreads();
            for (int p = tid; p < cnt; p += blockDim.x) {
                const ZRec me = {sz[p], sid[p]};
                const int t = z_tile(me.z), q0 = t > 0 ? tile[t - 1] : 0, q1 = tile[t];
                int at = q0;
                for (int q = q0; q < q1; q++) at += elem_gt(me, ZRec{sz[q], sid[q]}, rec);
                put(at, me.rec);
            }
        } else {
            int P = 32;
            while (P < cnt) P <<= 1;
            for (int p = tid; p < P; p += blockDim.x) {
                sz[p] = p < cnt ? rec[p].x : __int_as_float(0x7f800000);
                sid[p] = p < cnt ? p : kVtxMax + p;
            }
            __syncthreads();
            bitonic(P, sz, sid, rec);
            for (int p = tid; p < cnt; p += blockDim.x) put(p, sid[p]);
        }
        if constexpr (kPart == kVtxSort) return;
        __syncthreads();
    }
    int32_t *rho = a.rho + base;
    if constexpr (kPart == kVtxAll) {
        // z0, its error (in the key array until the roots are known) and the
        // densities by sorted position
        const float dzc = a.cuts.dz_cut, c2m = a.cuts.chi2_max;
        float *sez = reinterpret_cast<float *>(key);
        rho = sid;
        for (int p = tid; p < cnt; p += blockDim.x) {
            const float2 v = ze[p];
            sz[p] = v.x;
            sez[p] = v.y;
            a.wz[base + p] = weight_and_z(v);
        }
        __syncthreads();
        const auto z = [&](int q) { return sz[q]; };
        const auto ez = [&](int q) { return sez[q]; };
        const int items = (2 * cnt + 31) & ~31;                   // whole warps
        for (int it = tid; it < items; it += blockDim.x) {
            const int p = it >> 1, dir = (it & 1) ? 1 : -1;
            int r = p < cnt ? side_density(p, dir, cnt, z, ez, dzc, c2m) : 0;
            r += __shfl_xor_sync(kFull, r, 1);
            if (p < cnt && dir > 0) rho[p] = 1 + r;
        }
        __syncthreads();
        for (int it = tid; it < items; it += blockDim.x) {
            const int p = it >> 1, dir = (it & 1) ? 1 : -1;
            float bd = 0.f;
            int best = p < cnt ? side_link(p, dir, cnt, z, ez, [&](int q) { return rho[q]; }, dzc, c2m, bd) : -1;
            best = join_sides(best, bd);
            if (p < cnt && dir > 0) root[p] = best < 0 ? p : best;
        }
        __syncthreads();
    }
    for (int p = tid; p < cnt; p += blockDim.x) key[p] = root[p];
    int32_t *start = reinterpret_cast<int32_t *>(sz);             // by root: count, start, then end of its group
    for (int p = tid; p < cnt; p += blockDim.x) start[p] = 0;
    __syncthreads();
    // roots by pointer jumping; a racing read sees an old or a new value, both
    // ancestors, so the iteration still converges (path lengths halve)
    bool done = false;
    for (int it = 0; it < 2 * kPosBits + 4 && !done; it++) {
        bool ch = false;
        for (int p = tid; p < cnt; p += blockDim.x) {
            const int r = key[p], rr = key[r];
            if (rr != r) {
                key[p] = rr;
                ch = true;
            }
        }
        done = !__syncthreads_or(ch);
    }
    if (!done) {                                                  // uniform over the block
        if (tid == 0) set_status(a, PT_VTX_INTERNAL);
        return;
    }
    // group the tracks by root (k_vtx_fit puts a group's members in order of
    // position); a group whose root has rho > 1 and at least min_tracks
    // tracks is a candidate
    for (int p = tid; p < cnt; p += blockDim.x) {
        const int r = key[p];
        atomicAdd(&start[r], 1);
        root[p] = r;
    }
    __syncthreads();
    block_starts(start, cnt, s_warp);
    for (int p = tid; p < cnt; p += blockDim.x) {
        if (key[p] != p) continue;
        const int q = start[p], n = (p + 1 < cnt ? start[p + 1] : cnt) - q;
        if (rho[p] <= 1 || n < a.cuts.min_tracks) continue;
        const int c = atomicAdd(&s_nc, 1);
        if (c < kVtxCap) {
            a.cq[e * kVtxCap + c] = q;
            a.cn[e * kVtxCap + c] = n;
        } else {
            set_status(a, PT_VTX_TOO_MANY);
        }
    }
    __syncthreads();
    int32_t *order = a.order + base;
    for (int p = tid; p < cnt; p += blockDim.x) order[atomicAdd(&start[key[p]], 1)] = p;
    __syncthreads();
    if (tid == 0) a.nc[e] = min(s_nc, kVtxCap);
}

// The candidates of all events, one warp each: members in order, fit,
// 2-means split, provisional vertices (grid: candidates / warps per block x
// events).  What bounds it is the float64 pipe and the longest split: with a
// butterfly per sum, a division per centre, the members read again in every
// round and the outputs summed anew, 24 PU200 events (194 vertices of 25
// tracks each, up to 192) took 122 us; 70 us now.
constexpr int kFitWarps = 8;

__global__ void __launch_bounds__(32 * kFitWarps) k_vtx_fit(VtxArgs a) {
    pdl_enter();
    const int e = blockIdx.y, c = blockIdx.x * kFitWarps + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (c >= a.nc[e]) return;                                     // uniform over the warp
    const int base = a.ev_off[e], cnt = a.ev_off[e + 1] - base;
    const int32_t *sid = a.sid + base;
    const double2 *wz = a.wz + base;
    const int q = a.cq[e * kVtxCap + c], n = a.cn[e * kVtxCap + c];
    int32_t *mk = a.key + base + q;
    // the members in order of position: by comparing them with each other,
    // or, where that is more work, by a pass over the event's roots
    const int32_t *un = a.order + base + q;
    if ((int64_t)n * n <= 2 * (int64_t)cnt) {
        for (int k = lane; k < n; k += 32) {
            const int p = un[k];
            int at = 0;
            for (int j = 0; j < n; j++) at += un[j] < p;
            mk[at] = p;
        }
    } else {
        const int32_t *root = a.root + base;
        const int r = root[un[0]];
        int at = 0;
        for (int p0 = lane; p0 - lane < cnt; p0 += 256) {
            int v[8];                                             // eight loads in flight
#pragma unroll
            for (int i = 0; i < 8; i++) v[i] = p0 + 32 * i < cnt ? root[p0 + 32 * i] : -1;
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const unsigned m = __ballot_sync(kFull, v[i] == r);
                if (v[i] == r) mk[at + __popc(m & ((1u << lane) - 1u))] = p0 + 32 * i;
                at += __popc(m);
            }
        }
    }
    __syncwarp();
    Members m;
    m.mk = mk;
    m.wz = wz;
    m.n = n;
    m.cached = n <= 32 * kMemCache;
    m.side = 0;
    if (m.cached) {
#pragma unroll
        for (int i = 0; i < kMemCache; i++)
            if (lane + 32 * i < n) m.v[i] = wz[mk[lane + 32 * i]];
    }
    const auto pt = [&](int k) { return (double)a.in.pt[sid[mk[k] & kPosMask]]; };
    const Sides all = m.sums();                                   // (all on side 0 yet)
    const double z = all.swz0 / all.sw0;
    double chi2, pt2;
    m.chi2_pt2(-1, z, pt, chi2, pt2);
    // chi2 / (n - 1) > split_chi2, the quotient taken only near the cut
    const double lim = (double)a.cuts.split_chi2 * (double)(n - 1);
    bool split = false;
    if (n > 1 && (chi2 > lim * (1.0 + 1e-12) ||
                  (!(chi2 < lim * (1.0 - 1e-12)) && chi2 / (double)(n - 1) > (double)a.cuts.split_chi2))) {
        int hi = 0;
        m.each([&](int, const double2 &v, int) {
            const int u = v.y >= z;
            hi += u;
            return u;
        });
        hi = warp_sum(hi);
        if (hi > 0 && hi < n) {
            Sides s = m.sums();
            double c0, c1;
            warp_div2(s.swz0, s.sw0, s.swz1, s.sw1, c0, c1);
            int up = 0;
            bool have = false;
            for (int round = 0; round < kKmeansRounds; round++) {
                bool diff = false;
                up = 0;
                m.each([&](int, const double2 &v, int was) {
                    const int u = fabs(v.y - c1) < fabs(v.y - c0);          // ties: the lower centre
                    diff |= u != was;
                    up += u;
                    return u;
                });
                up = warp_sum(up);
                diff = __any_sync(kFull, diff);
                if (have && !diff) break;
                have = true;
                if (up == 0 || up == n) break;
                s = m.sums();
                warp_div2(s.swz0, s.sw0, s.swz1, s.sw1, c0, c1);
            }
            split = up >= a.cuts.min_tracks && n - up >= a.cuts.min_tracks;
        }
    }
    Sides s = all;
    double z0 = z, z1 = 0.0;
    if (split) {
        s = m.sums();
        warp_div2(s.swz0, s.sw0, s.swz1, s.sw1, z0, z1);
    }
    int vtx[2] = {0, 0};
    for (int part = 0; part < (split ? 2 : 1); part++) {
        const double zv = part ? z1 : z0, sw = part ? s.sw1 : s.sw0;
        if (split) m.chi2_pt2(part, zv, pt, chi2, pt2);
        int v = 0;
        if (lane == 0) {
            v = atomicAdd(a.nv + e, 1);
            if (v < kVtxCap) {
                const int o = e * kVtxCap + v;
                a.vz[o] = zv;
                a.vez[o] = (float)(1.0 / sqrt(sw));
                a.vc2[o] = (float)chi2;
                a.vnt[o] = split ? (part ? s.n1 : n - s.n1) : n;
                a.vsp[o] = pt2;
                a.vkey[o] = 2 * q + part;
            } else {
                set_status(a, PT_VTX_TOO_MANY);
            }
        }
        vtx[part] = __shfl_sync(kFull, v, 0);
    }
    // the vertex of every member, as its complement (members of no candidate
    // keep their position there, which is not negative)
    int32_t *mv = a.order + base + q;
    m.each([&](int k, const double2 &, int u) {
        mv[k] = ~(split && u ? vtx[1] : vtx[0]);
        return u;
    });
}

// Per event: the vertices by sum of pT^2 (then z, then the key), their
// outputs and the vertex of every member track (one block).
constexpr int kOrderThreads = 1024;

__global__ void __launch_bounds__(kOrderThreads) k_vtx_order(VtxArgs a) {
    pdl_enter();
    __shared__ double s_z[kVtxCap], s_sp[kVtxCap];
    __shared__ int s_vkey[kVtxCap], s_rank[kVtxCap];
    const int e = blockIdx.x, tid = threadIdx.x;
    const int base = a.ev_off[e], cnt = a.nv[e] > 0 ? a.ev_off[e + 1] - base : 0;     // (none if not clustered)
    const int nv = min(a.nv[e], kVtxCap);
    const int32_t *key = a.key + base, *sid = a.sid + base;
    for (int v = tid; v < nv; v += blockDim.x) {
        s_z[v] = a.vz[e * kVtxCap + v];
        s_sp[v] = a.vsp[e * kVtxCap + v];
        s_vkey[v] = a.vkey[e * kVtxCap + v];
    }
    __syncthreads();
    for (int v = tid; v < nv; v += blockDim.x) {
        // sums of pT^2 are not negative, so their bits order like them: the
        // float64 pipe stays out of this loop over all vertices
        const double sv = s_sp[v], zv = s_z[v];
        const long long bv = __double_as_longlong(sv);
        const int kv = s_vkey[v];
        int r = 0;
        for (int u = 0; u < nv; u++) {
            const long long bu = __double_as_longlong(s_sp[u]);
            r += bu > bv || (bu == bv && (s_z[u] < zv || (s_z[u] == zv && s_vkey[u] < kv)));
        }
        s_rank[v] = r;
        if (r < a.max_vertices) {
            const int64_t o = (int64_t)e * a.max_vertices + r;
            a.out.z[o] = (float)zv;
            a.out.ez[o] = a.vez[e * kVtxCap + v];
            a.out.chi2[o] = a.vc2[e * kVtxCap + v];
            a.out.ndf[o] = a.vnt[e * kVtxCap + v] - 1;
            a.out.ntracks[o] = a.vnt[e * kVtxCap + v];
            a.out.sumpt2[o] = (float)sv;
        }
    }
    if (tid == 0) {
        a.out.n[e] = min(nv, a.max_vertices);
        if (nv > a.max_vertices) set_status(a, PT_VTX_TOO_MANY);
    }
    __syncthreads();
    const int32_t *mv = a.order + base;
    for (int j = tid; j < cnt; j += blockDim.x) {
        const int v = ~mv[j];
        if (v >= 0 && v < nv && s_rank[v] < a.max_vertices)
            a.out.track_vertex[sid[key[j] & kPosMask]] = s_rank[v];
    }
}

__global__ void __launch_bounds__(kThreads) k_track_summary(int32_t n_tracks, const int32_t *hits, const uint8_t *tn,
                                                            const float *params, const float *cov,
                                                            const int32_t *tuple, const int32_t *ev_off,
                                                            int32_t n_events, float pt_of_kappa, int32_t *ev,
                                                            float *z0, float *ez0, float *pt, uint8_t *nh) {
    pdl_enter();
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_tracks; k += gridDim.x * blockDim.x) {
        const int t = tuple[k];
        const int h = hits[(int64_t)t * PT_NMAX];
        int lo = 0, hi = n_events;                       // the last e with ev_off[e] <= h
        while (hi - lo > 1) {
            const int m = (lo + hi) >> 1;
            if (ev_off[m] <= h) lo = m;
            else hi = m;
        }
        ev[k] = lo;
        z0[k] = params[(int64_t)k * 5 + 4];
        ez0[k] = sqrtf(cov[(int64_t)k * 15 + 14]);
        pt[k] = pt_of_kappa / fabsf(params[(int64_t)k * 5]);
        nh[k] = tn[t];
    }
}

}  // namespace

// Scratch layout (byte offsets, each array 16-byte aligned).
struct VtxLayout {
    size_t ev_off, ev_cur, part, order, rho, root, wz, ze, key, sid, nc, nv, cq, cn, vz, vsp, vez, vc2, vnt,
        vkey, total;
};

VtxLayout vertex_layout(int32_t n_tracks, int32_t n_events) {
    VtxLayout L;
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o = (o + bytes + 15) & ~(size_t)15;
        return at;
    };
    const size_t nt = (size_t)n_tracks + 1, ne = (size_t)n_events + 1, ncap = (size_t)n_events * kVtxCap + 1;
    L.ev_off = take(4 * ne);
    L.ev_cur = take(4 * ne);
    L.part = take(4 * ((size_t)n_events / kScanItems + 2));
    L.order = take(4 * nt);
    L.rho = take(4 * nt);
    L.root = take(4 * nt);
    L.wz = take(16 * nt);
    L.ze = take(8 * nt);
    L.key = take(4 * nt);
    L.sid = take(4 * nt);
    L.nc = take(4 * ne);
    L.nv = take(4 * ne);
    L.cq = take(4 * ncap);
    L.cn = take(4 * ncap);
    L.vz = take(8 * ncap);
    L.vsp = take(8 * ncap);
    L.vez = take(4 * ncap);
    L.vc2 = take(4 * ncap);
    L.vnt = take(4 * ncap);
    L.vkey = take(4 * ncap);
    L.total = o;
    return L;
}

size_t vertex_scratch_bytes(int32_t n_tracks, int32_t n_events) { return vertex_layout(n_tracks, n_events).total; }

pt_status launch_vertices(const pt_vertex_tracks &in, int32_t n_tracks, int32_t n_events,
                          const pt_vertex_cuts &cuts, int32_t max_vertices, void *scratch, const pt_vertices &out,
                          int grid, cudaStream_t s) {
    VtxArgs a;
    a.n_tracks = n_tracks;
    a.n_events = n_events;
    a.max_vertices = max_vertices;
    a.in = in;
    a.cuts = cuts;
    const VtxLayout L = vertex_layout(n_tracks, n_events);
    char *w = (char *)scratch;
    a.ev_off = (int32_t *)(w + L.ev_off);
    a.ev_cur = (int32_t *)(w + L.ev_cur);
    int32_t *part = (int32_t *)(w + L.part);
    a.order = (int32_t *)(w + L.order);
    a.rho = (int32_t *)(w + L.rho);
    a.root = (int32_t *)(w + L.root);
    a.wz = (double2 *)(w + L.wz);
    a.rec = (float4 *)(w + L.wz);
    a.ze = (float2 *)(w + L.ze);
    a.key = (int32_t *)(w + L.key);
    a.sid = (int32_t *)(w + L.sid);
    a.nc = (int32_t *)(w + L.nc);
    a.nv = (int32_t *)(w + L.nv);
    a.cq = (int32_t *)(w + L.cq);
    a.cn = (int32_t *)(w + L.cn);
    a.vz = (double *)(w + L.vz);
    a.vsp = (double *)(w + L.vsp);
    a.vez = (float *)(w + L.vez);
    a.vc2 = (float *)(w + L.vc2);
    a.vnt = (int32_t *)(w + L.vnt);
    a.vkey = (int32_t *)(w + L.vkey);
    a.out = out;
    // Windows in kernels of their own where the events are large: for track
    // summaries of which a third are eligible, one block against four kernels
    // measured 35 / 49 us at 3400 tracks per event, 50 / 57 us at 5100 and
    // 67 / 62 us at 6800; for fitted PU200 events (48,600 tracks, a tenth
    // eligible) 225 / 106 us.  For events of like size the line lies where
    // either costs at most ~15 us more than the other.  The host knows only the
    // mean: one large event among many small ones is left to its block, at up
    // to the 225 us above.
    const bool split = n_tracks / n_events > kVtxSplit;
    // per device and call (cheap; no shared state between threads or devices)
    auto big_smem = [](void (*k)(VtxArgs)) {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kVtxDynSmem) == cudaSuccess;
    };
    if (!(split ? big_smem(k_vtx_group<kVtxSort>) && big_smem(k_vtx_group<kVtxRoots>) : big_smem(k_vtx_group<kVtxAll>)))
        return PT_ERR_CUDA;
    // (ev_off and ev_cur are neighbours in the scratch)
    if (cudaMemsetAsync(a.ev_off, 0, L.part - L.ev_off, s) != cudaSuccess ||
        cudaMemsetAsync(out.status, 0, sizeof(int32_t), s) != cudaSuccess)
        return PT_ERR_CUDA;
    {
        KernelTimer t("k_vtx_count", s);
        launch_pdl(k_vtx_count, grid, kThreads, 0, s, a);
    }
    launch_scan(a.ev_off, n_events, part, s);
    {
        KernelTimer t("k_vtx_fill", s);
        launch_pdl(k_vtx_fill, grid, kThreads, 0, s, a);
    }
    if (split) {
        {
            KernelTimer t("k_vtx_sort", s);
            launch_pdl(k_vtx_group<kVtxSort>, n_events, kVtxThreads, kVtxDynSmem, s, a);
        }
        {
            KernelTimer t("k_vtx_density", s);
            launch_pdl(k_vtx_window<false>, 2 * grid, kThreads, 0, s, a);
        }
        {
            KernelTimer t("k_vtx_link", s);
            launch_pdl(k_vtx_window<true>, 2 * grid, kThreads, 0, s, a);
        }
        KernelTimer t("k_vtx_roots", s);
        launch_pdl(k_vtx_group<kVtxRoots>, n_events, kVtxThreads, kVtxDynSmem, s, a);
    } else {
        KernelTimer t("k_vtx_group", s);
        launch_pdl(k_vtx_group<kVtxAll>, n_events, kVtxThreads, kVtxDynSmem, s, a);
    }
    {
        KernelTimer t("k_vtx_fit", s);
        launch_pdl(k_vtx_fit, dim3(kVtxCap / kFitWarps, n_events), 32 * kFitWarps, 0, s, a);
    }
    KernelTimer t("k_vtx_order", s);
    launch_pdl(k_vtx_order, n_events, kOrderThreads, 0, s, a);
    return PT_OK;
}

void launch_track_summary(int32_t n_tracks, const int32_t *hits, const uint8_t *tn, const float *params,
                          const float *cov, const int32_t *tuple, const int32_t *ev_off, int32_t n_events, float bz,
                          int32_t *ev, float *z0, float *ez0, float *pt, uint8_t *nhits, int grid, cudaStream_t s) {
    // pT [GeV] = 0.299792458 B[T] R[m], R = 1 / (100 |kappa|) with kappa in 1/cm
    const float pt_of_kappa = 0.299792458e-2f * bz;
    KernelTimer t("k_track_summary", s);
    launch_pdl(k_track_summary, grid, kThreads, 0, s, n_tracks, hits, tn, params, cov, tuple, ev_off, n_events, pt_of_kappa,
                                             ev, z0, ez0, pt, nhits);
}

}  // namespace ptk
