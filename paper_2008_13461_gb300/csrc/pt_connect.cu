// Step a3: Cellular-Automaton connection (Sec. 3.2).  Cells (a,b) and (b,c)
// sharing hit b are linked when the R-z alignment, dz, curvature and
// beamspot predicates of b's region (barrel or endcap, Sec. 4.2) pass.
//
// Cells (b,c) are taken in cell order (cells are grouped by their outer hit
// c, so neighbouring threads work on neighbouring middle hits).
// The cells ending on b were written by the Fishbone kernel ordered by
// a bucket of their R-z slope key relative to b (monotone in the key, about
// one cell per bucket), with their inner hits (-1 for a dead one), so the candidates (a,b) of a
// cell lie in a contiguous run of that array, the buckets of its key
// window; the Fishbone also leaves the ends of the buckets, so the run is
// found with two loads (a binary search took about seven one after the
// other: 2167 -> 1970 us for 64 PU200 events, and the ends cost the Fishbone 55).
// Lists that are longer than a team of the Fishbone sorts are searched.
//
// The R-z cut is very tight, so it is first used as a window on the slope
// key.  For a barrel b, with key = dz/dr of a segment,
//     X = (r_b-r_a)(z_c-z_b) - (z_b-z_a)(r_c-r_b) = dr_ab dr_bc (key_c - key_a)
// and |X| <= tol |ac| <= tol (|ab| + |bc|) give
//     |key_c - key_a| <= tol (sqrt(1+key_a^2)/dr_bc + sqrt(1+key_c^2)/dr_ab);
// for a disk b the same holds with r and z exchanged.  With sqrt(1+key_a^2)
// and 1/dr_ab bounded by their maximum over the cells ending on b, every
// aligned candidate falls in the window; the run searched is the window
// widened far beyond the rounding of the key differences, and inside it the
// window test itself, a float32 R-z test with an error bound and then the
// exact predicate chain decide.
//
// A warp takes 128 consecutive cells at a time, in order from a queue, and
// lists those that can have candidates (their inner hit's layer is the outer
// layer of a pair: about a quarter).  Each lane then finds the run of one of
// them, but what comes after is done on the runs laid end to end, an entry per
// lane, and the entries that pass the window are collected until 32 are
// there for the predicates: a run has 0 to ~10 entries, two on average, of
// which one in three passes, so with a cell per lane from start to end 12 of 32
// lanes were at work on average, and the loads of a run came one after the
// other.  What passes comes in the order of the cells, so the edges of a
// cell are contiguous in the order found (the depth-first search walks them
// backwards from the cell's edge range), and the warp writes the edges of its
// 128 cells with one reservation.
//
// The kernel waits on dependent L2 loads, so it is compiled for as many
// resident warps as its shared memory leaves (12 blocks of 4 per SM, 40
// registers; 10 blocks: 10% slower).  64 PU200 events 1970 -> 1410 us, 24
// events with pT > 0.3 GeV 1420 -> 940, 32 PU50 events 95 -> 70, one PU200
// event 78 -> 51.  Chunks of 64 or 96 cells take 14% and 6% longer (rounds of
// searches that are not full), of 192 or 256 no less, and leave an end of few
// warps in one event (63, 75 us); a claim of the next chunk ahead of time
// does the same (70 us).  One 64-byte record of what is read of a middle
// hit, and a search with four probes at a time, measured the same or worse.
//
// The predicates run as float32 filters only; a cell with a candidate they
// cannot decide (about one in 10^5) is left to a second pass that has the
// exact forms, which keeps the big-integer code and its registers out of
// the main kernel.
#include "pt_common.cuh"
#include "pt_kernels.cuh"

namespace ptk {

constexpr int kCaWarps = 4;
constexpr int kCaChunk = 4;         // rounds of 32 cells per edge reservation
constexpr int kCaPer = 32 * kCaChunk;
constexpr int kCaQueue = 160;         // edges a warp remembers

// The predicate chain: 1 connects, 0 does not; with kExact = false, 2 when
// a float32 filter cannot decide and none fails.
template <bool kExact>
__device__ __forceinline__ int ca_chain(const FHit &A, const FHit &B, const FHit &C, const pt_ca_cuts &rg,
                                        int32_t *cnt) {
    const int r1 = pred_rz<kExact>(A, B, C, rg.tol_rz2, cnt);
    if (!r1) return 0;
    const int r2 = pred_dz<kExact>(A, C, rg.zmax, cnt);
    if (!r2) return 0;
    const int r3 = pred_curv<kExact>(A, B, C, rg.k_curv, cnt);
    if (!r3) return 0;
    const int r4 = pred_beamspot<kExact>(A, B, C, rg.rmax2, cnt);
    if (!r4) return 0;
    return (r1 | r2 | r3 | r4) == 1 ? 1 : 2;
}

// the exact chain, out of line (only the pass over undecided cells uses it)
static __device__ __noinline__ int ca_test(const FHit A, const FHit B, const FHit C, const pt_ca_cuts rg,
                                           int32_t *cnt) {
    return ca_chain<true>(A, B, C, rg, cnt);
}

// Branch-free part of the R-z test: false only when the float32 evaluation
// with its error bound proves the alignment cut fails.
__device__ __forceinline__ bool rz_maybe(const float4 &a, const FHit &b, const FHit &c, float tol2) {
    const float X = det2(b.r - a.w, c.z - b.z, b.z - a.z, c.r - b.r);
    const float e1 = c.r - a.w, e2 = c.z - a.z;
    const float T = tol2 * (e1 * e1 + e2 * e2);
    return T - X * X >= -ferr(4, T + X * X);
}

template <bool kExact>
__device__ __forceinline__ int connects(const Params &p, const float4 &a, const FHit &B, const FHit &C,
                                        const pt_ca_cuts &rg) {
    if (!rz_maybe(a, B, C, rg.tol_rz2)) return 0;
    const FHit A = {a.x, a.y, a.z, a.w};
    if (kExact) return ca_test(A, B, C, rg, p.counters);
    return ca_chain<false>(A, B, C, rg, p.counters);
}

// exclusive prefix of v over the warp, and the warp total
__device__ __forceinline__ int warp_excl(int v, int lane, int &total) {
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += t;
    }
    total = __shfl_sync(0xffffffffu, incl, 31);
    return incl - v;
}

// first position of s[0, n) whose key's bucket is >= bk (buckets ascending);
// for the lists without ends of buckets
__device__ __forceinline__ int lower_bucket(const float2 *s, int n, int bk, float k0, float iw) {
    const float fb = (float)bk;
    int l = 0, h = bk > 0 ? n : 0;
    while (l < h) {
        const int m = (l + h) >> 1;
        if (sk_coord(__ldg(s + m).x, k0, iw) < fb) l = m + 1;
        else h = m;
    }
    return l;
}

// The candidates (a,b) of a cell x = (b,c): entries [r, end) of b's
// bucket-ordered arrays, of which those with |key - key_c| <= wdt pass the
// window.
struct Search {
    FHit B, C;
    float key_c, wdt;
    int32_t r, end;
    bool disk;
};

__device__ __forceinline__ Search search_of(const Params &p, int b, int c) {
    Search s;
    s.r = s.end = 0;
    const int64_t b0 = p.in_off[b];
    int ns = p.in_live[b];
    if (b0 + ns > p.cap_cells) ns = 0;
    if (ns == 0) return s;
    s.B = load_hit(p.bh, b);
    s.C = load_hit(p.bh, c);
    s.disk = p.layer[p.blayer[b]].kind == PT_LAYER_DISK;
    const float tol = s.disk ? p.region_tol[1] : p.region_tol[0];
    const float4 hk = p.hk[b];
    const float dr = s.C.r - s.B.r, dz = s.C.z - s.B.z;
    const float num = s.disk ? dr : dz, den = s.disk ? dz : dr;
    s.key_c = den != 0.f ? num / den : __int_as_float(0x7f800000);
    // window half-width, widened for float32 rounding of the keys
    float wdt = tol * (hk.x / fabsf(den) + sqrtf(1.0f + s.key_c * s.key_c) / hk.y);
    wdt = wdt * (1.0f + 1e-5f) + 1e-5f * (1.0f + fabsf(s.key_c) + hk.x);
    if (!(wdt == wdt) || den == 0.f) wdt = __int_as_float(0x7f800000);
    s.wdt = wdt;
    // keys passing the window test lie in [lo, hi]
    const float sl = (fabsf(s.key_c) + wdt) * 9.5367431640625e-7f;
    const float lo = s.key_c - wdt - sl;
    float hi = s.key_c + wdt + sl;
    if (!(hi == hi)) hi = __int_as_float(0x7f800000);
    // the cells are ordered by a bucket of their key, monotone in the key:
    // the run searched is that of the buckets of [lo, hi]
    const int nb = sk_buckets(ns);
    const int blo = sk_bucket(lo, hk.z, hk.w, nb), bhi = sk_bucket(hi, hk.z, hk.w, nb);
    if (ns <= kSkEnds) {
        const uint16_t *E = p.sk_end + b0;
        const int sh = sk_end_shift(ns), e0 = blo >> sh;
        s.r = e0 > 0 ? __ldg(E + e0 - 1) : 0;
        s.end = __ldg(E + (bhi >> sh));
    } else {
        const float2 *S = p.sk + b0;
        s.r = lower_bucket(S, ns, blo, hk.z, hk.w);
        s.end = bhi < nb - 1 ? lower_bucket(S, ns, bhi + 1, hk.z, hk.w) : ns;
    }
    s.r += (int32_t)b0;
    s.end += (int32_t)b0;
    return s;
}

// an entry passes the window (inner hit -1: a dead cell)
__device__ __forceinline__ bool in_window(const float2 &e, float key_c, float wdt) {
    return fabsf(e.x - key_c) <= wdt && __float_as_int(e.y) >= 0;
}

// Per warp: the cells of a chunk to search, the searches of up to 32 of them,
// and the edges found.
struct __align__(16) CaWarp {
    FHit B[32], C[32];
    float4 own[32];                  // key, half-width; as ints, entry minus flat index, and position | disk << 8
    int32_t cand[3][64];             // candidates that passed the window: entry, inner hit, search
    int32_t b[kCaPer], c[kCaPer];    // cells to search: inner and outer hit,
    uint8_t pos[kCaPer];             //   position in the chunk
    uint8_t acc_pos[kCaQueue];         // edges found, by position: position of the cell,
    int32_t acc[kCaQueue];             //   entry of the inner cell
    uint32_t und[kCaChunk];          // positions left to the exact pass
};

// Writes the na edges found, and the edge ranges of their cells: one
// reservation.  With last = false the cell of the last edge may have more to
// come, so its edges stay; if there are none but those, the cell is left to
// the exact pass (which takes any number).  Returns how many stay.
__device__ __noinline__ int write_edges(const Params &p, CaWarp &sm, int64_t x0, int na, bool last, int lane) {
    const unsigned below = (1u << lane) - 1u;
    // drop the edges of cells left to the exact pass (rare)
    if (__any_sync(0xffffffffu, lane < kCaChunk && sm.und[lane] != 0)) {
        int n = 0;
        for (int i0 = 0; i0 < na; i0 += 32) {
            const int i = i0 + lane;
            const int pos = i < na ? sm.acc_pos[i] : 0, k = i < na ? sm.acc[i] : 0;
            const bool keep = i < na && !((sm.und[pos >> 5] >> (pos & 31)) & 1);
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            __syncwarp();            // all have read what some now write over (a ballot alone orders no memory)
            if (keep) {
                sm.acc_pos[n + __popc(m & below)] = (uint8_t)pos;
                sm.acc[n + __popc(m & below)] = k;
            }
            n += __popc(m);
            __syncwarp();
        }
        na = n;
        if (na == 0) return 0;
    }
    int stay = 0;
    if (!last) {
        const int pos = sm.acc_pos[na - 1];
        for (int i = lane; i < na; i += 32) stay += sm.acc_pos[i] == pos;
        stay = __reduce_add_sync(0xffffffffu, stay);
        if (stay == na) {
            if (na + 32 <= kCaQueue) return na;
            __syncwarp();
            if (lane == 0) sm.und[pos >> 5] |= 1u << (pos & 31);
            __syncwarp();
            return 0;
        }
    }
    const int n = na - stay;
    int64_t base = 0;
    if (lane == 0) {
        base = atomicAdd(p.counters + C_EDGES, n);
        if (base + n > p.cap_edges) set_flag(p.counters, PT_FLAG_EDGES);
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int i = lane; i < n; i += 32) {
        const int pos = sm.acc_pos[i];
        const int ci = __ldg(p.sci + sm.acc[i]);
        if (base + i < p.cap_edges) {
            p.edge_src[base + i] = ci;
            p.edge_dst[base + i] = (int32_t)(x0 + pos);
        }
        p.has_out[ci] = 1;
        if (i == 0 || sm.acc_pos[i - 1] != pos) {
            int e = i + 1;
            while (e < n && sm.acc_pos[e] == pos) e++;
            p.edge_rng[x0 + pos] = make_int2((int32_t)(base + i), e - i);
        }
    }
    for (int i0 = 0; i0 < stay; i0 += 32) {
        const int i = i0 + lane;
        const int pos = i < stay ? sm.acc_pos[n + i] : 0, k = i < stay ? sm.acc[n + i] : 0;
        __syncwarp();
        if (i < stay) {
            sm.acc_pos[i] = (uint8_t)pos;
            sm.acc[i] = k;
        }
        __syncwarp();
    }
    return stay;
}

// the predicates on candidates 0..n-1 <= 32, a lane each; those that connect
// join the edges found
__device__ __forceinline__ int test_candidates(const Params &p, CaWarp &sm, int64_t x0, int n, int na, int lane) {
    while (na + 32 > kCaQueue) na = write_edges(p, sm, x0, na, false, lane);
    int v = 0, k = 0, pos = 0;
    if (lane < n) {
        const int i = sm.cand[2][lane];
        const float4 a = __ldg(p.bh + sm.cand[1][lane]);
        k = sm.cand[0][lane];
        const int at = __float_as_int(sm.own[i].w);
        pos = at & 255;
        v = connects<false>(p, a, sm.B[i], sm.C[i], p.region[at >> 8]);
        if (v == 2) atomicOr(&sm.und[pos >> 5], 1u << (pos & 31));
    }
    const unsigned m = __ballot_sync(0xffffffffu, v == 1);
    if (v == 1) {
        const int t = na + __popc(m & ((1u << lane) - 1u));
        sm.acc[t] = k;
        sm.acc_pos[t] = (uint8_t)pos;
    }
    __syncwarp();
    return na + __popc(m);
}

__global__ void __launch_bounds__(32 * kCaWarps, 12) k_connect(Params p) {
    pdl_enter();
    __shared__ CaWarp s_warp[kCaWarps];
    __shared__ uint8_t s_inner_is_outer[PT_MAX_PAIRS];
    if (upstream_overflow(p, PT_FLAG_CELLS)) return;
    if (threadIdx.x < PT_MAX_PAIRS) s_inner_is_outer[threadIdx.x] = p.pair_inner_is_outer[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    CaWarp &sm = s_warp[w];
    const unsigned below = (1u << lane) - 1u;
    const int64_t n_cells = min((int64_t)p.counters[C_CELLS], p.cap_cells);
    // fewer cells to a chunk where 128 would leave warps without one (one PU50
    // event 24 -> 16 us, 50 helices 18 -> 12)
    const int warps = gridDim.x * kCaWarps;
    const int rounds = (int)min((int64_t)kCaChunk, max((n_cells + 32 * warps - 1) / (32 * warps), (int64_t)1));
    const int per = 32 * rounds;
    const int n_chunks = (int)((n_cells + per - 1) / per);
    // the warps take the chunks in order from a queue: the chunks in flight
    // are neighbours, and so are the middle hits whose sorted cells they read
    for (;;) {
        int ch = 0;
        if (lane == 0) ch = atomicAdd(p.counters + C_CA_NEXT, 1);
        ch = __shfl_sync(0xffffffffu, ch, 0);
        if (ch >= n_chunks) break;
        const int64_t x0 = (int64_t)ch * per, x1 = min(x0 + per, n_cells);
        // 1) the live cells whose inner hit can have cells ending on it (no
        //    cell ends on a layer that is the outer layer of no pair; most
        //    cells start on BPix1: no edge range is written for them, and the
        //    search records read none), so that the searches run on full warps
        int nlist = 0;
        if (lane < kCaChunk) sm.und[lane] = 0;
#pragma unroll
        for (int it = 0; it < kCaChunk; it++) {
            const int pos = it * 32 + lane;
            const int64_t x = x0 + pos;
            const bool need = x < x1 && p.cell_alive[x] && s_inner_is_outer[p.cell_pair[x]];
            const unsigned m = __ballot_sync(0xffffffffu, need);
            if (need) {
                const int i = nlist + __popc(m & below);
                sm.b[i] = p.cell_inner[x];
                sm.c[i] = p.cell_outer[x];
                sm.pos[i] = (uint8_t)pos;
                p.edge_rng[x] = make_int2(0, 0);
            }
            nlist += __popc(m);
        }
        if (nlist == 0) continue;
        __syncwarp();
        // 2) the searches
        int na = 0;
        for (int i0 = 0; i0 < nlist; i0 += 32) {
            Search se;
            int cnt = 0, pos = 0;
            if (i0 + lane < nlist) {
                pos = sm.pos[i0 + lane];
                se = search_of(p, sm.b[i0 + lane], sm.c[i0 + lane]);
                cnt = se.end - se.r;
            }
            int total;
            const int excl = warp_excl(cnt, lane, total);
            const unsigned some = __ballot_sync(0xffffffffu, cnt > 0);
            if (cnt > 0) {
                const int i = __popc(some & below);
                sm.B[i] = se.B;
                sm.C[i] = se.C;
                sm.own[i] = make_float4(se.key_c, se.wdt, __int_as_float(se.r - excl),
                                        __int_as_float(pos | (se.disk ? 256 : 0)));
            }
            __syncwarp();
            int nq = 0, before = -1;
            for (int f = 0; f < total; f += 32) {
                // the search that flat entry f + lane belongs to: the last one starting at or before it
                const unsigned at = (unsigned)(excl - f);
                const unsigned starts = __reduce_or_sync(0xffffffffu, cnt > 0 && at < 32u ? 1u << at : 0u);
                const int i = before + __popc(starts & (below | (1u << lane)));
                before += __popc(starts);
                bool pass = false;
                int k = 0, inner = 0;
                if (f + lane < total) {
                    const float4 o = sm.own[i];
                    k = __float_as_int(o.z) + f + lane;
                    const float2 e = __ldg(p.sk + k);
                    inner = __float_as_int(e.y);
                    pass = in_window(e, o.x, o.y);
                }
                const unsigned m = __ballot_sync(0xffffffffu, pass);
                if (pass) {
                    const int c = nq + __popc(m & below);
                    sm.cand[0][c] = k;
                    sm.cand[1][c] = inner;
                    sm.cand[2][c] = i;
                }
                nq += __popc(m);
                __syncwarp();
                const bool end = f + 32 >= total;
                while (nq >= 32 || (end && nq > 0)) {
                    na = test_candidates(p, sm, x0, min(nq, 32), na, lane);
                    nq = max(nq - 32, 0);
                    if (lane < nq) {
#pragma unroll
                        for (int c = 0; c < 3; c++) sm.cand[c][lane] = sm.cand[c][32 + lane];
                    }
                    __syncwarp();
                }
            }
        }
        // 3) their edges
        if (na > 0) write_edges(p, sm, x0, na, true, lane);
        __syncwarp();
        // cells with an undecided candidate: left to the exact pass
        if (__any_sync(0xffffffffu, lane < kCaChunk && sm.und[lane] != 0)) {
#pragma unroll 1
            for (int it = 0; it < kCaChunk; it++) {
                if ((sm.und[it] >> lane) & 1) {
                    const int k = atomicAdd(p.counters + C_CA_PENDING, 1);
                    if (k < p.cap_cells) reinterpret_cast<int32_t *>(p.ck)[k] = (int32_t)(x0 + it * 32 + lane);
                    else set_flag(p.counters, PT_FLAG_CELLS);
                }
            }
            __syncwarp();
        }
    }
}

// The cells with an undecided candidate (a few hundred), a warp each, with the
// exact predicates: an entry per lane, so that a cell waits for one exact
// evaluation and not for those of its run one after the other, twice (a
// thread per cell: 63 -> 20 us for 24 events with pT > 0.3 GeV, 25 -> 11 for one
// PU200 event).  A run of more than 32 entries is gone through twice, to count
// and to write.
__global__ void __launch_bounds__(128) k_connect_exact(Params p) {
    pdl_enter();
    if (upstream_overflow(p, PT_FLAG_CELLS)) return;
    const int n = (int)min((int64_t)p.counters[C_CA_PENDING], p.cap_cells);
    const int32_t *list = reinterpret_cast<const int32_t *>(p.ck);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    // cells dealt round the blocks first: they spread over the SMs
    for (int k = w * gridDim.x + blockIdx.x; k < n; k += gridDim.x * (blockDim.x >> 5)) {
        const int x = list[k];
        const Search s = search_of(p, p.cell_inner[x], p.cell_outer[x]);
        const auto hit = [&](int e0) {
            const int e = e0 + lane;
            bool v = false;
            if (e < s.end) {
                const float2 q = __ldg(p.sk + e);
                if (in_window(q, s.key_c, s.wdt))
                    v = connects<true>(p, __ldg(p.bh + __float_as_int(q.y)), s.B, s.C, p.region[s.disk ? 1 : 0]);
            }
            return __ballot_sync(0xffffffffu, v);
        };
        unsigned found = hit(s.r);
        int m = __popc(found);
        for (int e0 = s.r + 32; e0 < s.end; e0 += 32) m += __popc(hit(e0));
        int64_t base = 0;
        if (lane == 0 && m > 0) base = atomicAdd(p.counters + C_EDGES, m);
        base = __shfl_sync(0xffffffffu, base, 0);
        int64_t at = base;
        for (int e0 = s.r; e0 < s.end && m > 0; e0 += 32) {
            if (e0 > s.r) found = hit(e0);
            if ((found >> lane) & 1) {
                const int ci = p.sci[e0 + lane];
                const int64_t t = at + __popc(found & below);
                if (t < p.cap_edges) {
                    p.edge_src[t] = ci;
                    p.edge_dst[t] = x;
                }
                p.has_out[ci] = 1;
            }
            at += __popc(found);
        }
        if (lane == 0) {
            if (base + m > p.cap_edges) set_flag(p.counters, PT_FLAG_EDGES);
            p.edge_rng[x] = make_int2((int32_t)base, m);
        }
    }
}

void launch_connect(const Params &p, const Grid &g, cudaStream_t s) {
    {
        KernelTimer t("k_connect", s);
        launch_pdl(k_connect, g.blocks(12, 2), 32 * kCaWarps, 0, s, p);
    }
    KernelTimer t("k_connect_exact", s);
    launch_pdl(k_connect_exact, g.blocks(4), 128, 0, s, p);
}

}  // namespace ptk
