// Step a2: the Fishbone (Sec. 3.3), and the per-cell data the CA connection
// needs from it.
//
// Cells sharing an outer hit o whose inner hits lie on one layer and are
// aligned as seen from o form a fishbone; every cell of it dies except the
// shortest (equal lengths: the smaller input index of the inner hit wins).
//
// A team of one or more warps per outer hit.  It keeps, per cell, the difference vector
// u = h_inner - h_o in shared memory; hits are multiples of 2^-14 below 64 in
// magnitude, so u is exact in float32 and the alignment test and the squared
// length (an integer in grid units) are evaluated from it with no further
// memory traffic.  Alignment within eps implies that the unit directions of
// two siblings differ by at most du = eps pi/2 (plus float32 slack), hence
// so does any 1-Lipschitz key of them (u^_z for a barrel o, the radial
// component for a disk o).  The siblings are counting-sorted into one or two
// key buckets each, and each cell is compared only with the later cells
// of its own bucket and of the next K buckets, K covering a key difference
// of du: a superset of its aligned siblings, so the result is exact at
// ~O(k) work per outer hit.
//
// The same pass prepares the CA connection: it writes the cells of o ordered
// by a bucket of their R-z slope key relative to o (with the inner hit, -1
// for a dead cell, and the cell index; the bucket is monotone in the key,
// about one cell per bucket, free order inside), the ends of those buckets, the bucket parameters, and
// per hit the bounds the slope window needs (over all cells of o).  Both sorts
// are done at once: their counters share 32-bit words, so one clearing, one
// scan and one loop over the cells each for counting and placing serve both.
//
// What bounds it is the work in shared memory and the instructions around
// it.  For 64 PU200 events the hits of up to 184 cells took 2.84 ms; with the
// scan's 16-byte accesses (its entries met in a few banks: half of the
// kernel's shared-memory cycles) 2.69; with both sorts at once and
// up to two direction buckets per cell 2.19.  A dead cell is marked with a byte
// store: the same with an atomicOr of a bit, in a branch that single lanes
// take, costs 0.77 ms; so does a list of the close pairs for later, 0.2 ms; so do
// the pairs laid end to end with full warps of them (0.2 to 0.3 ms: a pair per
// lane has to find its two cells, which costs what the idle lanes cost).
//
// The cells of an outer hit sit in shared memory while its team works on them,
// so the shared memory per hit bounds how many hits an SM holds, and
// the warps per hit how many warps hide the gathers' latency and how long a
// hit takes.  Most outer hits have few cells, so three launches share the
// work: one warp per hit up to 128 cells (256 buckets, 40 warps per SM),
// taking chunks of outer hits from a queue and listing the others for two
// warps (up to 288 cells, 42 warps per SM) and four warps per hit (up to 512,
// 44); an exact pass of eight takes the rest (undecided tests, more
// cells), sorted in shared memory like the others up to 1024 cells, which
// pT > 0.3 GeV events reach (0.2% of their hits), with a pairwise loop over
// global memory beyond.  With one warp per hit throughout (up to 184, 320 and
// 512 cells; 32, 24 and 12 warps per SM) the four kernels took 2.25 + 0.79 +
// 0.05 + 0.04 ms for 64 PU200 events, now 1.20 + 1.38 + 0.05 + 0.02; 0.68 + 0.93
// + 0.36 + 0.07 for 24 events with pT > 0.3 GeV, now 0.42 + 0.75 + 0.35 + 0.02;
// 62 + 57 + 42 + 17 us for one PU200 event, whose few large hits are a wait for
// the slowest team, now 47 + 48 + 19 + 13; 158 us for 32 PU50 events, now 146.
// Limits of 64 or 96 cells for one warp take 8% and 3% longer in all; 256 or 320
// cells for two warps 2% (more hits of 257 or more for four; fewer hits per SM).
#include "pt_common.cuh"
#include "pt_kernels.cuh"

namespace ptk {

// Per team: the cells of one outer hit (up to M) and NB bucket counters, whose
// low halves count the cells by direction key and whose high halves by
// R-z slope key, so that one scan serves both sorts.
template <int M, int NB>
struct __align__(16) FbCells {
    float4 rec[M];                   // u = h_inner - h_o (exact), 1/|u| in w
    uint32_t pos[NB];                // counts, then starts, then ends
    float ck[M];                     // R-z slope key
    uint32_t meta[M];                // slot; then direction bucket and, in the high half, slope bucket and then place
    uint16_t idx[M];                 // cells sorted by direction bucket
    uint8_t dead[M];
};

// pair_slot in shared memory: a lane-wise index into the kernel's parameters
// would serialise
__device__ __forceinline__ void load_slots(const Params &p, uint8_t *slot) {
    if (threadIdx.x < PT_MAX_PAIRS) slot[threadIdx.x] = (uint8_t)p.pair_slot[threadIdx.x];
    __syncthreads();
}

// Bucket key of a record: u^_z (barrel o) or the radial component of u^
// (disk o; (rx, ry) is o's radial direction).  Explicit roundings, so every
// evaluation gives the same bits.
__device__ __forceinline__ float fb_key(const float4 &r, bool disk, float rx, float ry) {
    const float k = disk ? __fmul_rn(__fmaf_rn(r.x, rx, __fmul_rn(r.y, ry)), r.w) : __fmul_rn(r.z, r.w);
    return k == k ? k : 0.f;
}

// squared length of a difference vector, in grid units (exact)
__device__ __forceinline__ long long len2u(float ux, float uy, float uz) {
    const int x = __float2int_rn(ux * 16384.0f), y = __float2int_rn(uy * 16384.0f), z = __float2int_rn(uz * 16384.0f);
    return (long long)x * x + (long long)y * y + (long long)z * z;     // |x| < 2^21: 32x32 -> 64-bit products
}

__device__ __forceinline__ int cell_layer(const Params &p, int64_t c) { return p.pair[p.cell_pair[c]].inner; }

// Warp-wide minimum, maximum and sum with one redux instruction each.  The
// float map keeps their order (non-negative floats keep their bits,
// negative ones have the magnitude bits flipped; no NaN reaches it), and a
// minimum or maximum is one of the inputs, so nothing is rounded.
__device__ __forceinline__ int ford(float f) {
    const int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float fval(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }
__device__ __forceinline__ float warp_min(float f) { return fval(__reduce_min_sync(0xffffffffu, ford(f))); }
__device__ __forceinline__ float warp_max(float f) { return fval(__reduce_max_sync(0xffffffffu, ford(f))); }
__device__ __forceinline__ int warp_sum(int v) { return __reduce_add_sync(0xffffffffu, v); }

// The T warps that work on one outer hit: a warp of a block of several, or
// (T > 1) a block.
template <int T>
__device__ __forceinline__ void team_sync() {
    if (T == 1) __syncwarp();
    else __syncthreads();
}

// The direction key's and the slope key's ranges and bounds, reduced over a
// team (part: shared, for T > 1).
struct FbRange {
    float bmin, bmax, smin, smax, k2max, gmin;
};

template <int T>
__device__ __forceinline__ FbRange team_range(FbRange v, bool starts, FbRange *part) {
    v.bmin = warp_min(v.bmin);
    v.bmax = warp_max(v.bmax);
    if (starts) {
        v.k2max = warp_max(v.k2max);
        v.gmin = warp_min(v.gmin);
        v.smin = warp_min(v.smin);
        v.smax = warp_max(v.smax);
    }
    if (T > 1) {
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < T; w++) {
            const FbRange q = part[w];
            v.bmin = fminf(v.bmin, q.bmin);
            v.bmax = fmaxf(v.bmax, q.bmax);
            v.smin = fminf(v.smin, q.smin);
            v.smax = fmaxf(v.smax, q.smax);
            v.k2max = fmaxf(v.k2max, q.k2max);
            v.gmin = fminf(v.gmin, q.gmin);
        }
    }
    return v;
}

// exclusive prefix sums of both halves of a[0, nb) in place (nb a power of two >= 32; one
// team): 128 entries at a time, four per lane in one 16-byte access.  (Entries
// lane * nb / 32 + q, one after the other, met in 2 to 4 banks: half of the
// kernel's shared-memory cycles were those conflicts.)  Each warp of a team
// adds up the entries before its share first.
template <int T>
__device__ __forceinline__ void team_exclusive_scan(uint32_t *a, int nb, int lane) {
    int q0 = 0, q1 = nb;
    uint32_t carry = 0;
    if (T > 1) {
        const int w = threadIdx.x >> 5, share = max(128, nb / T);
        q0 = min(w * share, nb);
        q1 = min(q0 + share, nb);
        for (int q = 4 * lane; q < q0; q += 128) {
            const uint4 v = *reinterpret_cast<const uint4 *>(a + q);
            carry += (v.x + v.y) + (v.z + v.w);
        }
        carry = __reduce_add_sync(0xffffffffu, carry);     // (halves below 2^16: no more than the cells)
        __syncthreads();
    }
    for (int q = q0 + 4 * lane; q - 4 * lane < q1; q += 128) {
        uint4 v = q < q1 ? *reinterpret_cast<const uint4 *>(a + q) : make_uint4(0, 0, 0, 0);
        const uint32_t sum = (v.x + v.y) + (v.z + v.w);
        uint32_t incl = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += t;
        }
        const uint32_t e = carry + incl - sum;
        carry += __shfl_sync(0xffffffffu, incl, 31);
        v = make_uint4(e, e + v.x, e + v.x + v.y, e + v.x + v.y + v.z);
        if (q < q1) *reinterpret_cast<uint4 *>(a + q) = v;
    }
}

// Verdicts of the n <= M cells of outer hit o (one team; t: thread of it); returns the
// thread's count of live cells.  kExact = false (float32 filters only): returns -1,
// having written no verdict, when an alignment test is undecided.
template <int T, int M, int NB, bool kExact>
__device__ __forceinline__ int fishbone_hit(const Params &p, int o, int n, int64_t b, int t, float unit_thr,
                                            float du, FbCells<M, NB> &sm, FbRange *part, const uint8_t *slot) {
    // NB: at least the buckets of M cells (sk_buckets)
    static_assert(M <= kSkEnds, "the connection expects the ends of the buckets");
    static_assert(NB >= 32 && NB >= M && (NB & (NB - 1)) == 0, "bucket array too small");
    const float4 ho = __ldg(p.bh + o);
    const int Lo = p.blayer[o];
    const bool disk = p.layer[Lo].kind == PT_LAYER_DISK;
    const float irr = rsqrtf(ho.x * ho.x + ho.y * ho.y);
    const float rx = ho.x * irr, ry = ho.y * irr;
    // a hit on a layer that is the inner layer of no pair starts no cell:
    // the connection never reads the slope keys of the cells ending on it
    const bool starts = p.layer_is_inner[Lo] != 0;
    // pass 1: records, direction keys' range, and the R-z slope keys (barrel
    // o: (z_o - z_a)/(r_o - r_a); disk o: (r_o - r_a)/(z_o - z_a)) with the
    // per-hit bounds and their range
    const float inf = __int_as_float(0x7f800000);
    FbRange rg = {3.0f, -3.0f, inf, -inf, 0.f, 3.0e38f};
    for (int j = t; j < n; j += 32 * T) {
        const float4 a = __ldg(p.bh + p.cell_inner[b + j]);
        sm.meta[j] = slot[p.cell_pair[b + j]];
        sm.dead[j] = 0;
        if (starts) {
            const float dr = ho.w - a.w, dz = ho.z - a.z;
            const float num = disk ? dr : dz, den = disk ? dz : dr;
            // the key only places the cell in the connection's search window,
            // whose margins (1e-5 relative) are far above the 2 ulp of this quotient
            const float ck = den != 0.f ? __fdividef(num, den) : __int_as_float(0x7f800000);
            rg.k2max = fmaxf(rg.k2max, ck * ck);
            rg.gmin = fminf(rg.gmin, fabsf(den));
            sm.ck[j] = ck;
            if (fabsf(ck) <= 3.4e38f) {
                rg.smin = fminf(rg.smin, ck);
                rg.smax = fmaxf(rg.smax, ck);
            }
        }
        const float ux = a.x - ho.x, uy = a.y - ho.y, uz = a.z - ho.z;
        const float4 r = make_float4(ux, uy, uz, rsqrtf(ux * ux + uy * uy + uz * uz));
        sm.rec[j] = r;
        const float key = fb_key(r, disk, rx, ry);
        rg.bmin = fminf(rg.bmin, key);
        rg.bmax = fmaxf(rg.bmax, key);
    }
    rg = team_range<T>(rg, starts, part);
    const float bmin = rg.bmin, bmax = rg.bmax, smin = rg.smin, smax = rg.smax;
    // Direction buckets: each inner layer of o has its own aligned range of
    // nbr buckets (one or two buckets per cell), so a cell meets only siblings
    // on its own layer.  Two keys within du lie at most K buckets apart (K
    // bounds du / width plus the rounding of the bucket coordinates, below
    // 6e-4 for up to 2048 buckets).  Slope buckets: about one per cell.
    const int nbs = sk_buckets(n), nb = min(NB, 2 * nbs);
    const int nbr = nb >> p.fb_slot_shift[Lo];
    const float span = fmaxf(bmax - bmin, fmaxf(fabsf(bmin), fabsf(bmax)) * 1e-6f);
    const float iw = span > 0.f ? (float)nbr / span : 0.f;
    const int K = (int)fminf(du * iw + 6e-4f, (float)nbr) + 1;
    float siw = 0.f;
    if (starts) {
        const float sspan = fmaxf(smax - smin, fmaxf(fabsf(smin), fabsf(smax)) * 1e-6f);
        siw = sspan > 0.f && sspan <= 3.4e38f ? (float)nbs / sspan : 0.f;
        // bound of sqrt(1 + key^2), smallest gap, lowest key, inverse width
        if (t == 0) p.hk[o] = make_float4(sqrtf(1.0f + rg.k2max), rg.gmin, smin, siw);
    }
    for (int q = t; q < nb; q += 32 * T) sm.pos[q] = 0;
    team_sync<T>();
    for (int j = t; j < n; j += 32 * T) {
        const float key = fb_key(sm.rec[j], disk, rx, ry);
        uint32_t m = sm.meta[j] * nbr + min(max((int)((key - bmin) * iw), 0), nbr - 1);
        atomicAdd(&sm.pos[m], 1u);
        if (starts) {
            const uint32_t bs = sk_bucket(sm.ck[j], smin, siw, nbs);
            atomicAdd(&sm.pos[bs], 1u << 16);
            m |= bs << 16;
        }
        sm.meta[j] = m;
    }
    team_sync<T>();
    team_exclusive_scan<T>(sm.pos, nb, t & 31);
    team_sync<T>();
    for (int j = t; j < n; j += 32 * T) {
        const uint32_t m = sm.meta[j];
        sm.idx[atomicAdd(&sm.pos[m & 0xffffu], 1u) & 0xffffu] = (uint16_t)j;
        if (starts)
            sm.meta[j] = (m & 0xffffu) | (atomicAdd(&sm.pos[m >> 16], 1u << 16) & 0xffff0000u);
    }
    team_sync<T>();
    // sm.pos[bk] now holds the ends of bucket bk.  Each pair once: every cell
    // against the cells after it in its own bucket and the next K buckets of
    // its layer (a superset of its siblings within du of its key); of an
    // aligned pair the longer cell dies (equal lengths: the larger input
    // index of the inner hit).
    bool und = false;
    for (int q0 = t; q0 < n; q0 += 32 * T) {
        const int j = sm.idx[q0];
        const float4 r1 = sm.rec[j];
        const float3 v1 = make_float3(r1.x * r1.w, r1.y * r1.w, r1.z * r1.w);
        const int bk1 = sm.meta[j] & 0xffffu;
        const int qend = sm.pos[min(bk1 + K, bk1 | (nbr - 1))] & 0xffffu;
        for (int q = q0 + 1; q < qend; q++) {
            const int d = sm.idx[q];
            const float4 r2 = sm.rec[d];
            const float dx = v1.x - r2.x * r2.w, dy = v1.y - r2.y * r2.w, dz = v1.z - r2.z * r2.w;
            if (dx * dx + dy * dy + dz * dz > unit_thr) continue;
            const int v = pred_fb_d<kExact>(r1.x, r1.y, r1.z, r2.x, r2.y, r2.z, p.fishbone_eps2, p.counters);
            if (v == 2) und = true;
            if (v != 1) continue;
            const long long l1 = len2u(r1.x, r1.y, r1.z), l2 = len2u(r2.x, r2.y, r2.z);
            const bool j_wins = l1 < l2 || (l1 == l2 && p.perm[p.cell_inner[b + j]] < p.perm[p.cell_inner[b + d]]);
            sm.dead[j_wins ? d : j] = 1;
        }
    }
    if (T == 1) {
        __syncwarp();
        und = __any_sync(0xffffffffu, und);
    } else {
        und = __syncthreads_or(und);
    }
    if (!kExact && und) return -1;

    // pass 2: the verdicts, and the cells grouped by slope-key bucket for the
    // CA connection, a dead one with the inner hit -1 (any order inside a
    // bucket: the connection searches by bucket)
    int alive = 0;
    for (int j = t; j < n; j += 32 * T) {
        const bool dead = sm.dead[j];
        if (dead) p.cell_alive[b + j] = 0;
        else alive++;
        if (starts) {
            const int64_t q = b + (sm.meta[j] >> 16);
            p.sk[q] = make_float2(sm.ck[j], __int_as_float(dead ? -1 : p.cell_inner[b + j]));
            p.sci[q] = (int32_t)(b + j);
        }
    }
    // where the connection starts and ends its searches
    if (starts) {
        const int sh = sk_end_shift(n);
        for (int e = t; e < sk_ends(n); e += 32 * T) p.sk_end[b + e] = sm.pos[((e + 1) << sh) - 1] >> 16;
    }
    if (t == 0) p.in_live[o] = n;       // (never all dead: the shortest of them lives)
    team_sync<T>();
    return alive;
}

// The same for any n with a pairwise loop over global memory and ranks by
// direct comparison (outer hits with more cells than a team holds: sorted
// keys, so sorted buckets too).
template <int T>
__device__ __noinline__ int fishbone_pairwise(const Params &p, int o, int n, int64_t b, int t, FbRange *part) {
    const float4 ho = __ldg(p.bh + o);
    const bool disk = p.layer[p.blayer[o]].kind == PT_LAYER_DISK;
    const bool starts = p.layer_is_inner[p.blayer[o]] != 0;
    const GHit gh = ghit(ho.x, ho.y, ho.z, ho.w);
    const FHit h = {ho.x, ho.y, ho.z, ho.w};
    const float inf = __int_as_float(0x7f800000);
    FbRange rg = {3.0f, -3.0f, inf, -inf, 0.f, 3.0e38f};
    for (int j = t; j < n; j += 32 * T) {
        const int i1 = p.cell_inner[b + j];
        const int L1 = cell_layer(p, b + j);
        const FHit h1 = load_hit(p.bh, i1);
        if (starts) {
            const float dr = ho.w - h1.r, dz = ho.z - h1.z;
            const float num = disk ? dr : dz, den = disk ? dz : dr;
            const float ck = den != 0.f ? __fdividef(num, den) : __int_as_float(0x7f800000);
            rg.k2max = fmaxf(rg.k2max, ck * ck);
            rg.gmin = fminf(rg.gmin, fabsf(den));
            p.ck[b + j] = ck;
            if (fabsf(ck) <= 3.4e38f) {
                rg.smin = fminf(rg.smin, ck);
                rg.smax = fmaxf(rg.smax, ck);
            }
        }
        const GHit g1 = ghit(h1.x, h1.y, h1.z, h1.r);
        const long long l1 = (g1.x - gh.x) * (g1.x - gh.x) + (g1.y - gh.y) * (g1.y - gh.y) +
                             (g1.z - gh.z) * (g1.z - gh.z);
        bool dead = false;
        for (int d = 0; d < n && !dead; d++) {
            if (d == j || cell_layer(p, b + d) != L1) continue;
            const int i2 = p.cell_inner[b + d];
            const FHit h2 = load_hit(p.bh, i2);
            if (!pred_fb(h1, h2, h, p.fishbone_eps2, p.counters)) continue;
            const GHit g2 = ghit(h2.x, h2.y, h2.z, h2.r);
            const long long l2 = (g2.x - gh.x) * (g2.x - gh.x) + (g2.y - gh.y) * (g2.y - gh.y) +
                                 (g2.z - gh.z) * (g2.z - gh.z);
            dead = l2 < l1 || (l2 == l1 && p.perm[i2] < p.perm[i1]);
        }
        if (dead) p.cell_alive[b + j] = 0;
    }
    if (starts) {
        rg = team_range<T>(rg, true, part);
        const float span = fmaxf(rg.smax - rg.smin, fmaxf(fabsf(rg.smin), fabsf(rg.smax)) * 1e-6f);
        const float iw = span > 0.f && span <= 3.4e38f ? (float)sk_buckets(n) / span : 0.f;
        if (t == 0) p.hk[o] = make_float4(sqrtf(1.0f + rg.k2max), rg.gmin, rg.smin, iw);
    }
    team_sync<T>();
    int alive = 0;
    for (int j = t; j < n; j += 32 * T) {
        const bool dead = p.cell_alive[b + j] == 0;
        alive += !dead;
        if (!starts) continue;
        const float key = p.ck[b + j];
        int rank = 0;
        for (int i = 0; i < n; i++) {
            const float ki = p.ck[b + i];
            rank += ki < key || (ki == key && i < j);
        }
        p.sk[b + rank] = make_float2(key, __int_as_float(dead ? -1 : p.cell_inner[b + j]));
        p.sci[b + rank] = (int32_t)(b + j);
    }
    if (t == 0) p.in_live[o] = n;
    team_sync<T>();
    return alive;
}

// an outer hit left to the exact pass (listed in hit_bin, free once the
// hits are binned and the doublets' exact pass has run)
__device__ __forceinline__ void list_pending(const Params &p, int o, int lane) {
    if (lane == 0) p.hit_bin[atomicAdd(p.counters + C_FB_PENDING, 1)] = o;
}

__device__ __forceinline__ void add_alive(const Params &p, int v) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(p.counters + C_ALIVE_CELLS, v);
}

// Small warps: take chunks of consecutive binned hits from a queue, load
// their cell counts together, work through those with 1..M cells and list
// the ones with more: up to kFbMidMax cells from the front of the list
// array, more from its back.  A warp walks its chunk's hits in turn, so a
// chunk is 32 hits only where that leaves every resident warp several chunks:
// with 32 whatever the size, one PU200 event (30.8 k hits) kept 962 of 4864
// warps busy (454 -> 75 us with chunks by size; a PU50 event 158 -> 19 us, a
// batch of 32 of them 279 -> 194 us).
constexpr int kFbSmallMax = 128, kFbSmallBlocks = 5;
constexpr int kFbMidMax = 288, kFbMidWarps = 2, kFbMidBlocks = 21;
constexpr int kFbMaxWarps = 4, kFbMaxBlocks = 11;
constexpr int kFbExactWarps = 8;

template <int W, int M, int NB, int kMinBlocks>
__global__ void __launch_bounds__(32 * W, kMinBlocks) k_fishbone_small(Params p, float unit_thr, float du,
                                                                    int chunk_log2) {
    pdl_enter();
    __shared__ FbCells<M, NB> sm[W];
    __shared__ uint8_t s_slot[PT_MAX_PAIRS];
    if (upstream_overflow(p, PT_FLAG_CELLS)) return;
    load_slots(p, s_slot);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    int my_alive = 0;
    const int n_binned = p.bin_cnt[p.n_bins];
    const int n_chunks = (n_binned + (1 << chunk_log2) - 1) >> chunk_log2;
    for (;;) {
        int ch = 0;
        if (lane == 0) ch = atomicAdd(p.counters + C_FB_NEXT, 1);
        ch = __shfl_sync(0xffffffffu, ch, 0);
        if (ch >= n_chunks) break;
        const int o0 = ch << chunk_log2, ol = o0 + lane;
        int nl = 0, bl = 0;
        if (lane < (1 << chunk_log2) && ol < n_binned) {
            nl = p.in_cnt[ol];
            bl = p.in_off[ol];
        }
        const bool ok = nl >= 1 && (int64_t)bl + nl <= p.cap_cells;
        const unsigned mid = __ballot_sync(0xffffffffu, ok && nl > M && nl <= kFbMidMax);
        const unsigned huge = __ballot_sync(0xffffffffu, ok && nl > kFbMidMax);
        if (mid | huge) {
            int bm = 0, bh = 0;
            if (lane == 0) {
                if (mid) bm = atomicAdd(p.counters + C_FB_BIG, __popc(mid));
                if (huge) bh = atomicAdd(p.counters + C_FB_HUGE, __popc(huge));
            }
            bm = __shfl_sync(0xffffffffu, bm, 0);
            bh = __shfl_sync(0xffffffffu, bh, 0);
            if ((mid >> lane) & 1) p.fb_big[bm + __popc(mid & below)] = ol;
            if ((huge >> lane) & 1) p.fb_big[p.n_hits - 1 - (bh + __popc(huge & below))] = ol;
        }
        unsigned todo = __ballot_sync(0xffffffffu, ok && nl <= M);
        while (todo) {
            const int t = __ffs(todo) - 1;
            todo &= todo - 1;
            const int n = __shfl_sync(0xffffffffu, nl, t);
            const int b = __shfl_sync(0xffffffffu, bl, t);
            const int a = fishbone_hit<1, M, NB, false>(p, o0 + t, n, b, lane, unit_thr, du, sm[w], nullptr, s_slot);
            if (a >= 0) my_alive += a;
            else list_pending(p, o0 + t, lane);
        }
    }
    add_alive(p, my_alive);
}

// The listed outer hits, a block at a time from a queue (kFromBack:
// the list at the back of the array).
template <int T, int M, int NB, bool kFromBack, int kMinBlocks>
__global__ void __launch_bounds__(32 * T, kMinBlocks) k_fishbone_large(Params p, float unit_thr, float du) {
    pdl_enter();
    __shared__ FbCells<M, NB> sm;
    __shared__ FbRange s_part[T];
    __shared__ uint8_t s_slot[PT_MAX_PAIRS];
    __shared__ int s_next;
    if (upstream_overflow(p, PT_FLAG_CELLS)) return;
    load_slots(p, s_slot);
    int my_alive = 0;
    const int n_list = p.counters[kFromBack ? C_FB_HUGE : C_FB_BIG];
    for (;;) {
        if (threadIdx.x == 0) s_next = atomicAdd(p.counters + (kFromBack ? C_FB_HUGE_NEXT : C_FB_BIG_NEXT), 1);
        __syncthreads();
        const int k = s_next;
        if (k >= n_list) break;
        const int o = p.fb_big[kFromBack ? p.n_hits - 1 - k : k];
        const int n = p.in_cnt[o];
        int a = -1;
        if (n <= M)
            a = fishbone_hit<T, M, NB, false>(p, o, n, p.in_off[o], threadIdx.x, unit_thr, du, sm, s_part, s_slot);
        if (a >= 0) my_alive += a;
        else list_pending(p, o, threadIdx.x);
        __syncthreads();
    }
    add_alive(p, my_alive);
}

// Exact pass: the outer hits listed by the kernels above (an undecided
// alignment test, or more cells than those hold), with the exact
// predicate and the pairwise loop for any number of cells.
template <int T, int M, int NB>
__global__ void __launch_bounds__(32 * T) k_fishbone_exact(Params p, float unit_thr, float du) {
    pdl_enter();
    __shared__ FbCells<M, NB> sm;
    __shared__ FbRange s_part[T];
    __shared__ uint8_t s_slot[PT_MAX_PAIRS];
    if (upstream_overflow(p, PT_FLAG_CELLS)) return;
    load_slots(p, s_slot);
    int my_alive = 0;
    const int n_list = p.counters[C_FB_PENDING];
    for (int k = blockIdx.x; k < n_list; k += gridDim.x) {
        const int o = p.hit_bin[k];
        const int n = p.in_cnt[o], b = p.in_off[o];
        my_alive += n <= M ? fishbone_hit<T, M, NB, true>(p, o, n, b, threadIdx.x, unit_thr, du, sm, s_part, s_slot)
                           : fishbone_pairwise<T>(p, o, n, b, threadIdx.x, s_part);
    }
    add_alive(p, my_alive);
}

void launch_fishbone(const Params &p, float unit_thr, float du, const Grid &g, cudaStream_t s) {
    {
        // at least four chunks for each resident warp
        int chunk_log2 = 0;
        while (chunk_log2 < 5 && (p.n_hits >> (chunk_log2 + 1)) >= 4 * 8 * g.blocks(kFbSmallBlocks)) chunk_log2++;
        KernelTimer t("k_fishbone_small", s);
        launch_pdl(k_fishbone_small<8, kFbSmallMax, 256, kFbSmallBlocks>, g.blocks(kFbSmallBlocks), 256, 0, s, p, unit_thr, du, chunk_log2);
    }
    {
        KernelTimer t("k_fishbone_medium", s);
        launch_pdl(k_fishbone_large<kFbMidWarps, kFbMidMax, 512, false, kFbMidBlocks>, g.blocks(kFbMidBlocks, 2),
                   32 * kFbMidWarps, 0, s, p, unit_thr, du);
    }
    {
        KernelTimer t("k_fishbone_large", s);
        launch_pdl(k_fishbone_large<kFbMaxWarps, 512, 1024, true, kFbMaxBlocks>, g.blocks(kFbMaxBlocks),
                   32 * kFbMaxWarps, 0, s, p, unit_thr, du);
    }
    KernelTimer t("k_fishbone_exact", s);
    launch_pdl(k_fishbone_exact<kFbExactWarps, 1024, 1024>, g.blocks(4), 32 * kFbExactWarps, 0, s, p, unit_thr, du);
}

}  // namespace ptk
