// Step a1: doublets on layer pairs (Sec. 3.2, cuts of Table 1).
//
// Doublets: a group of G lanes owns one outer hit (the warps take the binned
// hits from a queue, in order).  For every layer pair ending on the outer
// hit's layer it derives the phi window (PhiW) and a conservative window
// along z (barrel) or r (disk) from ZIP and ZW, with margins above float32
// rounding, and sweeps the inner tiles' rows of that window laid end to end:
// consecutive lanes load consecutive binned hits (coalesced), evaluate ZW,
// ZIP, PhiW, PT exactly, and compact the accepted ones with a ballot into a
// shared-memory buffer.  The cells of one outer hit are written
// contiguously, so the cells sharing an outer hit (needed by the Fishbone
// and the CA connection) form one range.
//
// What bounds it is instruction issue (70% of the slots taken; a candidate
// costs about 80 instructions per warp, a window about 500).
#include "pt_common.cuh"
#include "pt_kernels.cuh"

namespace ptk {

constexpr float kTwoPiInv = 0.159154943f;
constexpr float kPi = 3.14159265f;

// What a sweep needs of a layer pair, in shared memory (a lane-wise index
// into the kernel's parameters serialises, and what does not depend on the
// outer hit is worked out once: 1623 -> 1544 us for 64 PU200 events, 105 -> 97
// for 32 PU50 events).  The angles and quotients of a window are those of CUDA's
// float32 functions: polynomials of 1e-5 for the angles gain little (1511 us
// against 1518 for 64 PU200 events, 95 / 98 for 32 PU50 events, 55 / 58 for one
// PU200 event) and search other rows of tiles where a window ends within 1e-5
// of an edge.
struct PairWin {
    float zlo, zhi, zmax, tan, k_pt, ez, ep, ec;     // cuts, and the filter's bounds
    float dphi;                                      // azimuthal half window of PhiW
    float pa, si, sx;                                // PT: 1 / (2 R) (0: no use), asin(rmin / 2R), asin(rmax / 2R) of the inner layer
    float rmin, rmax, za, zb;                        // inner layer; barrel: its z range, disk: the z range within the cuts
    float tscale;                                    // tiles per cm of its z (barrel) or r (disk)
    int32_t inner;                                   // inner layer, -1 - layer for a disk
};

// While every hit's r is the hypotenuse of its x and y (on_radius), |x|, |y|
// and so the filter's errors are bounded over the layers' envelopes, and the
// azimuth window may be narrowed by the radius.  With a hit off its radius in
// the batch, x and y are bounded by the grid alone (64 cm), and no window is
// narrowed: more candidates go to the sharper filters, which take their bounds
// from the operands.
constexpr float kGridXY = 64.0f * 64.0f;

__device__ __forceinline__ void load_windows(const Params &p, PairWin *win) {
    const int k = threadIdx.x;
    const bool off = p.counters[C_OFF_RADIUS] != 0;
    if (k < p.n_pairs) {
        const pt_pair_cuts pc = p.pair[k];
        const pt_layer li = p.layer[pc.inner];
        const bool barrel = li.kind == PT_LAYER_BARREL;
        PairWin w;
        w.zlo = pc.zlo, w.zhi = pc.zhi, w.zmax = pc.zmax, w.k_pt = pc.k_pt;
        w.tan = p.pair_tan[k], w.ez = p.pair_err_zip[k];
        w.ep = off ? 8.0f * kU * kGridXY * (1.0f + w.tan) : p.pair_err_phi[k];
        w.ec = off ? 4.0f * kU * kGridXY : p.pair_err_c[k];
        w.dphi = p.pair_dphi[k];
        // (an error of 2^-13 in each radius moves the arcsines' difference by
        // less than 6e-5 while 2R >= 10 cm and the radii are below 0.9 of it,
        // which is inside the margin of 1e-4)
        const float pa = p.pair_pt_a[k];
        w.pa = pa > 0.f && pa <= 0.1f && li.rmax * pa < 0.9f && !off ? pa : 0.f;
        w.si = asinf(li.rmin * w.pa), w.sx = asinf(li.rmax * w.pa);
        w.rmin = li.rmin, w.rmax = li.rmax;
        w.za = barrel ? li.zmin : fmaxf(li.zmin, pc.zlo);
        w.zb = barrel ? li.zmax : fminf(li.zmax, pc.zhi);
        w.tscale = barrel ? t_scale(li.zmin, li.zmax, p.n_t) : t_scale(li.rmin, li.rmax, p.n_t);
        w.inner = barrel ? pc.inner : -1 - pc.inner;
        win[k] = w;
    }
    __syncthreads();
}

// Conservative window of the inner hit's t coordinate for a pair, from ZIP
// (z-intercept within +-zmax) and ZW, over the inner layer's envelope.
__device__ __forceinline__ void t_window(const PairWin &w, float ro, float zo, float &tlo, float &thi) {
    const float zm = w.zmax;
    if (w.inner >= 0) {
        float f0 = w.rmin / ro, f1 = w.rmax / ro;
        float c0 = -zm + (zo + zm) * f0, c1 = -zm + (zo + zm) * f1;
        float c2 = zm + (zo - zm) * f0, c3 = zm + (zo - zm) * f1;
        tlo = fmaxf(fminf(fminf(c0, c1), fminf(c2, c3)), w.zlo);
        thi = fminf(fmaxf(fmaxf(c0, c1), fmaxf(c2, c3)), w.zhi);
        if (tlo > thi) tlo = thi = 0.5f * (tlo + thi);
    } else {
        const float za = w.za, zb = w.zb;
        if (fabsf(zo) > zm * 1.001f + 0.01f && za <= zb) {
            const float d0 = zo + zm, d1 = zo - zm;   // same sign
            float c0 = ro * (za + zm) / d0, c1 = ro * (zb + zm) / d0;
            float c2 = ro * (za - zm) / d1, c3 = ro * (zb - zm) / d1;
            tlo = fminf(fminf(c0, c1), fminf(c2, c3));
            thi = fminf(fmaxf(fmaxf(c0, c1), fmaxf(c2, c3)), ro);
            if (tlo > thi) tlo = thi = 0.5f * (tlo + thi);
        } else {
            tlo = w.rmin;
            thi = w.rmax;
        }
    }
}

// Fast filter of one candidate (i inner, o outer) for the main pass: 1 all
// four cuts hold, 0 one of them fails, 2 too close to a cut to say.
//
// The sharper filters bring their own error bounds and compensated products,
// about twice the operations (k_doublets 1721 -> 1652 us for 64 PU200 events),
// so the cuts are taken in forms with few operations and bounds that are
// constants of the pair; one candidate in ~10^5 lies within them and goes to
// the sharper filters.  With u = 2^-24, hits within their layers' envelopes and on
// their radius (both checked on input; load_windows says what is taken if a hit is off
// it) and every rounding at most u relative:
//  ZIP   F = (zmax ro - zmax ri) - |zi ro - zo ri|, each product and sum
//        rounded at most twice: off by less than 3u (|zo| ri + |zi| ro +
//        2 zmax (ro + ri)); taken as 8u with the layers' largest values.  F >
//        0 implies ro > ri.
//  PhiW  the condition is tan Dt - |C| >= 0 (Dt > 0 follows): |C| and Dt are
//        off by 2u ri ro, tan by 2u relative: less than 5u ri ro (1 + tan),
//        taken as 8u; |x|, |y| <= r + 2^-13.
//  PT    H = |o-i|^2 |i|^2 - k C^2 with k = k_pt / |o|^2: the first term is off
//        by 7u relative (differences of grid values are exact, sums of squares
//        3u), k by 8u (the quotient 4u) and its product with C^2 by two more,
//        C by c = 2u ri ro
//        (taken as 4u) and so k C^2 by k (2 |C| c + c^2) besides; taken as
//        16u (P + k C^2) + k (4 |C| c + 2 c^2).
struct PairFilter {
    float zlo, zhi, zmax, zr, tan, k, ez, ep, c4, kc2;
};

__device__ __forceinline__ int pair_filter(const PairFilter &f, const float4 &i, const float4 &o) {
    const float F = fmaf(-f.zmax, i.w, f.zr) - fabsf(fmaf(i.z, o.w, -(o.z * i.w)));
    const float C = fabsf(fmaf(i.x, o.y, -(i.y * o.x)));
    const float G = fmaf(f.tan, fmaf(i.x, o.x, i.y * o.y), -C);
    const float dx = o.x - i.x, dy = o.y - i.y;
    const float P = fmaf(dx, dx, dy * dy) * fmaf(i.x, i.x, i.y * i.y);
    const float q = f.k * C, t = q * C, H = P - t;
    const float e = fmaf(16.0f * kU, P + t, fmaf(f.c4, q, f.kc2));
    const bool zw = i.z >= f.zlo && i.z <= f.zhi;
    if (zw && F > f.ez && G > f.ep && H > e) return 1;
    return !zw || F < -f.ez || G < -f.ep || H < -e ? 0 : 2;
}

// One cell of outer hit o at index c.
__device__ __forceinline__ void write_cell(const Params &p, int64_t c, int i, int o, uint8_t pair) {
    if (c >= p.cap_cells) return;
    p.cell_inner[c] = i;
    p.cell_outer[c] = o;
    p.cell_pair[c] = pair;
    p.cell_alive[c] = 1;
    p.has_out[c] = 0;
}

// A cell in shared memory: the inner hit, and the pair above kIndexBits.  With
// more hits than that nothing is kept there: the outer hits are swept again.
constexpr int kIndexBits = 27;
static_assert(PT_MAX_PAIRS <= 1 << (32 - kIndexBits), "pair bits");

__device__ __forceinline__ void write_cell(const Params &p, int64_t c, uint32_t e, int o) {
    write_cell(p, c, (int)(e & ((1u << kIndexBits) - 1u)), o, (uint8_t)(e >> kIndexBits));
}

// Sweep all candidate inner hits of outer hit o.  kWrite = false: fill the
// shared buffer (up to cap entries, step apart) and count; kWrite = true: write
// cells directly at global index base + slot.  kExact = false: the
// predicates are float32 filters only, and *undecided is set on the lanes
// that met a candidate they cannot decide.  s_cand (or null): per-pair
// counts of the candidate inner hits tested, summed in shared memory.
template <int G, bool kWrite, bool kExact>
__device__ int sweep_outer(const Params &p, const PairWin *win, int o, int lane, unsigned gmask, int gshift, uint32_t *buf,
                           int step, int cap, int32_t *s_row, int64_t base, bool *undecided,
                           unsigned long long *s_cand = nullptr) {
    const float4 ho = __ldg(p.bh + o);
    const float xo = ho.x, yo = ho.y, zo = ho.z, ro = ho.w;
    const int Lo = p.blayer[o], ev = p.bev[o];
    const float phio = atan2f(yo, xo);
    const float io2 = __fdividef(1.0f, fmaf(xo, xo, yo * yo));
    const unsigned lanes = G == 32 ? 0xffffffffu : ((1u << G) - 1u);
    const unsigned below = (1u << lane) - 1u;
    int count = 0;
    const int npo = p.n_pairs_by_outer[Lo];
    for (int k = 0; k < npo; k++) {
        const int pi = p.pairs_by_outer[Lo][k];
        const PairWin &w = win[pi];
        float tlo, thi;
        t_window(w, ro, zo, tlo, thi);
        const float tmin = w.inner >= 0 ? w.za : w.rmin;
        // Tile ranges: the t window's float32 bounds are within ~1e-5 cm of
        // the exact ones, so a margin of 1e-4 cm keeps every accepted hit
        // inside; the half-width in phi already carries a 1e-4 rad margin
        // over PhiW's exact bound, far above the rounding of the angles.
        // Tile indices are monotone in t and phi (the binning uses the
        // same functions), so the tiles cover a superset of the accepted
        // hits whatever the tile counts.
        const float mt = 1e-4f + 1e-6f * fmaxf(fabsf(tlo), fabsf(thi));
        const int tb0 = t_tile(tlo - mt, tmin, w.tscale, p.n_t);
        const int tb1 = t_tile(thi + mt, tmin, w.tscale, p.n_t);
        // The PT cut (circumradius of beam line, inner and outer hit >= R)
        // accepts an azimuth difference up to |asin(r_o / 2R) - asin(r_i / 2R)|
        // or from pi - asin(r_o / 2R) - asin(r_i / 2R) on (both radii below
        // 2R: on a circle through the beam line a chord of length r makes
        // the angle asin(r / 2R) with the tangent there).  While the second
        // range lies beyond the pair's PhiW window, the first, taken over the
        // inner layer's radii with a margin far above the rounding of the
        // float32 arcsines, narrows the window to this outer hit.
        float dphi = w.dphi;
        if (w.pa > 0.f && ro * w.pa < 0.9f) {
            const float so = asinf(ro * w.pa);
            if (kPi - so - w.sx > dphi + 1e-3f) dphi = fminf(dphi, fmaxf(so - w.si, w.sx - so) + 1e-4f);
        }
        int f0 = __float2int_rd((phio - dphi + kPi) * (p.n_phi * kTwoPiInv));
        int f1 = __float2int_rd((phio + dphi + kPi) * (p.n_phi * kTwoPiInv));
        if (f1 - f0 + 1 >= p.n_phi) {
            f0 = 0;
            f1 = p.n_phi - 1;
        }
        PairFilter pf;
        pf.zlo = w.zlo;
        pf.zhi = w.zhi;
        pf.zmax = w.zmax;
        pf.zr = w.zmax * ro;
        pf.tan = w.tan;
        pf.k = w.k_pt * io2;
        pf.ez = w.ez;
        pf.ep = w.ep;
        pf.c4 = 4.0f * w.ec;
        pf.kc2 = 2.0f * pf.k * w.ec * w.ec;
        const int row0 = (ev * PT_N_LAYERS + (w.inner >= 0 ? w.inner : -1 - w.inner)) * p.n_phi;
        const int nrows = f1 - f0 + 1;
        unsigned cand = 0;
        // The rows of the window are separate ranges of the binned hits,
        // about as long as a group is wide: G of them at a time are laid
        // end to end in one range of slots, so the lanes stay busy across
        // row ends.  s_row holds, per row, the offset from slot to binned
        // index and the row's end in slot space.
        for (int r0 = 0; r0 < nrows; r0 += G) {
            int beg = 0, len = 0;
            if (r0 + lane < nrows) {
                const int f = f0 + r0 + lane;
                // (|phi| <= pi and dphi < 1.6: f lies within a turn of [0, n_phi))
                const int fb = f < 0 ? f + p.n_phi : f >= p.n_phi ? f - p.n_phi : f;
                const int tile = (row0 + fb) * p.n_t;
                beg = p.bin_cnt[tile + tb0];
                len = p.bin_cnt[tile + tb1 + 1] - beg;
            }
            int incl = len;
#pragma unroll
            for (int d = 1; d < G; d <<= 1) {
                const int t = __shfl_up_sync(gmask, incl, d, G);
                if (lane >= d) incl += t;
            }
            const int total = __shfl_sync(gmask, incl, G - 1, G);
            cand += (unsigned)total;
            if (total == 0) continue;
            __syncwarp(gmask);       // the previous rows' table is no longer read
            s_row[lane] = beg - (incl - len);
            s_row[G + lane] = incl;
            __syncwarp(gmask);
            for (int s0 = 0; s0 < total; s0 += G) {
                const int sl = s0 + lane;
                int v = 0;     // 1 accepted, 0 rejected, 2|3 undecided (kExact = false)
                int i = 0;
                if (sl < total) {
                    // the slot's row: the first whose end lies beyond it
                    int j = 0;
#pragma unroll
                    for (int h = G / 2; h > 0; h >>= 1)
                        if (s_row[G + j + h - 1] <= sl) j += h;
                    i = sl + s_row[j];
                    const float4 hi = __ldg(p.bh + i);
                    const float xi = hi.x, yi = hi.y, zi = hi.z, ri = hi.w;
                    v = pair_filter(pf, hi, ho);
                    if (v == 2) v = zi >= pf.zlo && zi <= pf.zhi ? 2 : 0;
                    if (v == 2) {
                        v = pred_zip<kExact>(xi, yi, zi, ri, xo, yo, zo, ro, pf.zmax, p.counters);
                        if (v) {
                            const int v2 = pred_phiw<kExact>(xi, yi, xo, yo, p.pair[pi].tan2_dphi, p.counters, zi, ri, zo, ro);
                            v = v2 ? (v | v2) : 0;
                        }
                        if (v) {
                            const int v3 = pred_pt<kExact>(xi, yi, zi, ri, xo, yo, zo, ro, p.pair[pi].k_pt, p.counters);
                            v = v3 ? (v | v3) : 0;
                        }
                    }
                }
                const bool acc = v == 1;
                if (!kExact && v > 1) *undecided = true;
                const unsigned m = (__ballot_sync(gmask, acc) >> gshift) & lanes;
                if (acc) {
                    const int slot = count + __popc(m & below);
                    if (kWrite) {
                        write_cell(p, base + slot, i, o, (uint8_t)pi);
                    } else if (slot < cap) {
                        buf[step * slot] = (uint32_t)i | (uint32_t)pi << kIndexBits;
                    }
                }
                count += __popc(m);
            }
        }
        if (s_cand && lane == 0 && cand) atomicAdd(s_cand + pi, (unsigned long long)cand);
    }
    return count;
}

__device__ __forceinline__ void write_range(const Params &p, int o, int64_t base, int n) {
    p.in_off[o] = (int32_t)base;
    p.in_cnt[o] = n;
    if (base + n > p.cap_cells) set_flag(p.counters, PT_FLAG_CELLS);
}

// Main pass: float32 filters only (no big-integer code, so far fewer
// registers); an outer hit with an undecided candidate (about one in 10^3)
// is listed for the exact pass.  It also counts the candidates tested per
// layer pair (the exact pass repeats a few of them and does not count).
// The cells of a warp's outer hits are reserved with one atomic and written
// by all its lanes, hit after hit: with an atomic and a loop for each hit, the
// one counter's L2 slice was 73% busy (all slices: 23%) and the byte arrays
// were written eight bytes at a time (164 -> 104 us for 32 PU50 events, 110 ->
// 100 us for one PU200 event, 1652 -> 1621 us for 64 of them).
// Two groups share a buffer and fill it from its ends; only if their cells
// don't fit together are both hits swept again, by all lanes of the warp.  With
// a buffer of 256 cells for each, and its own lanes sweeping a hit again while
// the others waited, 24 events with pT > 0.3 GeV, where every tenth hit has
// more cells, took 940 us against 799, and 64 PU200 events 1544 against 1535.
template <int G>
__global__ void __launch_bounds__(kThreads, 5) k_doublets(Params p) {
    pdl_enter();
    constexpr int kGroups = kThreads / G, kPerWarp = 32 / G;
    constexpr int kBuf = 40 * G;   // 40 KB of shared memory per block for every G
    constexpr int kPair = kPerWarp > 1 ? 2 : 1, kCap = kPair * kBuf;   // groups that share a buffer, from its ends
    __shared__ uint32_t s_buf[kGroups / kPair][kCap];
    __shared__ int32_t s_row[kGroups][2 * G];
    __shared__ unsigned long long s_cand[PT_MAX_PAIRS];
    __shared__ PairWin s_win[PT_MAX_PAIRS];
    if (threadIdx.x < PT_MAX_PAIRS) s_cand[threadIdx.x] = 0;
    load_windows(p, s_win);
    const int lane = threadIdx.x % G, grp = threadIdx.x / G, wl = threadIdx.x & 31, gw = wl / G;
    const int gshift = wl & ~(G - 1);
    const unsigned gmask = G == 32 ? 0xffffffffu : (((1u << G) - 1u) << gshift);
    const int cap = p.n_hits >> kIndexBits ? 0 : kCap;
    const bool odd = kPair > 1 && (gw & 1);
    const int n_binned = p.bin_cnt[p.n_bins];
    // the warps take the binned outer hits in order: the cells are laid out
    // nearly in the order of their outer hits
    for (;;) {
        int o0 = 0;
        if (wl == 0) o0 = atomicAdd(p.counters + C_DB_NEXT, kPerWarp);
        o0 = __shfl_sync(0xffffffffu, o0, 0);
        if (o0 >= n_binned) break;
        const int o = o0 + gw;
        int n = 0;
        bool und = false;
        if (o < n_binned)
            n = sweep_outer<G, false, false>(p, s_win, o, lane, gmask, gshift, s_buf[grp / kPair] + (odd ? kCap - 1 : 0),
                                             odd ? -1 : 1, cap, s_row[grp], 0, &und, s_cand);
        // what two hits leave in their buffer is whole if both fit
        const int both = kPair > 1 ? n + __shfl_xor_sync(0xffffffffu, n, G) : n;
        const unsigned um = __ballot_sync(0xffffffffu, und);
        const bool put = o < n_binned && !(um & gmask);
        // listed in hit_bin, free once the hits are binned (one slot per hit)
        if (o < n_binned && !put && lane == 0) p.hit_bin[atomicAdd(p.counters + C_DB_PENDING, 1)] = o;
        if (!put) n = 0;
        int first[kPerWarp + 1];     // the groups' cells end to end
        first[0] = 0;
#pragma unroll
        for (int q = 0; q < kPerWarp; q++) first[q + 1] = first[q] + __shfl_sync(0xffffffffu, n, q * G);
        const int total = first[kPerWarp];
        int64_t base = 0;
        if (wl == 0 && total > 0) base = atomicAdd(p.counters + C_CELLS, total);
        base = __shfl_sync(0xffffffffu, base, 0);
        int mine = 0;
#pragma unroll
        for (int q = 0; q < kPerWarp; q++) mine = gw == q ? first[q] : mine;
        if (put && lane == 0) write_range(p, o, base + mine, n);
        __syncwarp();
        const unsigned over = __ballot_sync(0xffffffffu, lane == 0 && n > 0 && both > cap);
        if (!over) {
            for (int k = wl; k < total; k += 32) {
                int q = 0, at = k;
#pragma unroll
                for (int t = 1; t < kPerWarp; t++)
                    if (k >= first[t]) {
                        q = t;
                        at = k - first[t];
                    }
                write_cell(p, base + k, s_buf[(grp - gw + q) / kPair][kPair > 1 && (q & 1) ? kCap - 1 - at : at], o0 + q);
            }
        } else {
            // beside hits with more cells than their buffer holds; those are swept again by all lanes
            if (both <= cap)
                for (int k = lane; k < n; k += G)
                    write_cell(p, base + mine + k, s_buf[grp / kPair][odd ? kCap - 1 - k : k], o);
            for (unsigned m = over; m; m &= m - 1) {
                const int from = __ffs(m) - 1;
                const int64_t at = base + __shfl_sync(0xffffffffu, mine, from);
                __syncwarp();
                sweep_outer<32, true, false>(p, s_win, o0 + from / G, wl, 0xffffffffu, 0, nullptr, 0, 0,
                                             s_row[grp - gw], at, &und);
            }
        }
        __syncwarp();
    }
    __syncthreads();
    if (threadIdx.x < p.n_pairs && s_cand[threadIdx.x])
        atomicAdd(reinterpret_cast<unsigned long long *>(p.counters + C_PAIR_CAND) + threadIdx.x, s_cand[threadIdx.x]);
}

// Exact pass over the listed outer hits (a few hundred): a warp per hit,
// the hits dealt round the blocks first, so that they spread over the SMs
// and no warp runs two hits' exact fallbacks one after the other.
__global__ void __launch_bounds__(kThreads) k_doublets_exact(Params p) {
    pdl_enter();
    constexpr int G = 32, kGroups = kThreads / G, kBuf = 40 * G;
    __shared__ uint32_t s_buf[kGroups][kBuf];
    __shared__ int32_t s_row[kGroups][2 * G];
    __shared__ PairWin s_win[PT_MAX_PAIRS];
    load_windows(p, s_win);
    const int lane = threadIdx.x % G, grp = threadIdx.x / G;
    const int cap = p.n_hits >> kIndexBits ? 0 : kBuf;
    const int n = p.counters[C_DB_PENDING];
    for (int k = grp * gridDim.x + blockIdx.x; k < n; k += gridDim.x * kGroups) {
        const int o = p.hit_bin[k];
        bool und = false;
        const int nc = sweep_outer<G, false, true>(p, s_win, o, lane, 0xffffffffu, 0, s_buf[grp], 1, cap, s_row[grp], 0,
                                                   &und);
        int64_t base = 0;
        if (lane == 0 && nc > 0) base = atomicAdd(p.counters + C_CELLS, nc);
        base = __shfl_sync(0xffffffffu, base, 0);
        if (lane == 0) write_range(p, o, base, nc);
        __syncwarp();
        if (nc <= cap)
            for (int j = lane; j < nc; j += G) write_cell(p, base + j, s_buf[grp][j], o);
        else
            sweep_outer<G, true, true>(p, s_win, o, lane, 0xffffffffu, 0, nullptr, 0, 0, s_row[grp], base, &und);
        __syncwarp();
    }
}

void launch_doublets(const Params &p, int lanes, const Grid &g, cudaStream_t s) {
    {
        KernelTimer t("k_doublets", s);
        const int grid = g.blocks(5);
        // Few hits: more lanes for each, so that every resident warp gets at
        // least four claims (one PU200 event: 1.3 claims with 8 lanes, 83 ->
        // 57 us with 32; one PU50 event 20 -> 17; from ~100 k hits on 8 lanes are
        // as good or better, 32 PU50 events 99 against 143 us with 16)
        while (lanes < 32 && (int64_t)p.n_hits * lanes < (int64_t)4 * kThreads * grid) lanes *= 2;
        switch (lanes) {
        case 4: launch_pdl(k_doublets<4>, grid, kThreads, 0, s, p); break;
        case 8: launch_pdl(k_doublets<8>, grid, kThreads, 0, s, p); break;
        case 16: launch_pdl(k_doublets<16>, grid, kThreads, 0, s, p); break;
        default: launch_pdl(k_doublets<32>, grid, kThreads, 0, s, p); break;
        }
    }
    KernelTimer t("k_doublets_exact", s);
    launch_pdl(k_doublets_exact, g.blocks(2), kThreads, 0, s, p);
}

}  // namespace ptk
