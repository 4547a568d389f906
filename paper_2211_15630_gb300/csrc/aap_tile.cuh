// aap_tile.cuh -- device code shared by the tile step kernels: tile geometry,
// the 25 source segments of a tile (its own 9 regions and the facing halo
// regions of its 8 neighbours, with periodic shifts or mirror maps, Sec. 2.4),
// warp-aggregated insertion into the next step's regions, the 3x3-cell
// neighbour sums (Eq. collision_VM / collision_NVM, the Langevin coupling
// sum), and the whole-block tile routine (stage, counting sort by cell,
// update, scatter) that serves tiles staged in global scratch.
#pragma once

#include <cuda_runtime.h>

#include "aap_device.cuh"
#include "aap_internal.cuh"

namespace aapk {

// Optional per-phase timing of the step kernel (tracing aid, compiled out
// unless AAP_PHASE_TIMING is defined): thread 0 of every block adds the clock
// cycles between phase marks to g_phase[].
#ifdef AAP_PHASE_TIMING
static __device__ unsigned long long g_phase[16];
#define PHASE_START() long long ph_t0_ = clock64()
#define PHASE_MARK(i)                                                         \
    do {                                                                      \
        if (threadIdx.x == 0) {                                               \
            const long long t_ = clock64();                                   \
            atomicAdd(&g_phase[i], (unsigned long long)(t_ - ph_t0_));        \
            ph_t0_ = t_;                                                      \
        }                                                                     \
    } while (0)
#else
#define PHASE_START() do { } while (0)
#define PHASE_MARK(i) do { } while (0)
#endif

// ------------------------------------------------------------ geometry ----
__device__ __forceinline__ int tile_x0(const Sys &S, int tx) { return S.x0tab[tx]; }
__device__ __forceinline__ int tile_y0(const Sys &S, int ty) { return S.y0tab[ty]; }
__device__ __forceinline__ int tile_of_x(const Sys &S, int cx)
{
    if (S.ncx < 32768) return (int)(((unsigned)(cx + 1) * (unsigned)S.ntx - 1u) / (unsigned)S.ncx);   // ntx <= ncx
    return (int)((((long long)cx + 1) * S.ntx - 1) / S.ncx);
}
__device__ __forceinline__ int tile_of_y(const Sys &S, int cy)
{
    if (S.ncy < 32768) return (int)(((unsigned)(cy + 1) * (unsigned)S.nty - 1u) / (unsigned)S.ncy);
    return (int)((((long long)cy + 1) * S.nty - 1) / S.ncy);
}
__device__ __forceinline__ int region_of(int lx, int ly, int tw, int th)
{
    const int rx = lx == 0 ? 0 : (lx == tw - 1 ? 2 : 1);
    const int ry = ly == 0 ? 0 : (ly == th - 1 ? 2 : 1);
    return ry * 3 + rx;
}

// Append rec to region `region` of tile `dtile` in buffer b, whose counters
// are cnt (per tile and region) and *spill_cnt.  Every lane of the warp must
// call; lanes with act == false take part in the vote only.  Lanes headed for
// the same region share one atomicAdd (warp aggregation).
__device__ __forceinline__ void warp_insert(const Sys &S, int b, bool act, int dtile, int region, int4 rec, int *cnt,
                                            int *spill_cnt)
{
    const int lane = threadIdx.x & 31;
    const int key = act ? dtile * kCntStride + region : -1 - lane;
    // most warps send every lane to one region: skip the match in that case
    const bool same = __all_sync(0xffffffffu, key == __shfl_sync(0xffffffffu, key, 0));
    const unsigned peers = same ? 0xffffffffu : __match_any_sync(0xffffffffu, key);
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (act && lane == leader) base = atomicAdd(&cnt[key], __popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (act) {
        const int slot = base + __popc(peers & ((1u << lane) - 1u));
        if (slot < S.cap[region]) {
            S.rec[b][(long long)dtile * S.tile_slots + S.off[region] + slot] = rec;
        } else {
            const int e = atomicAdd(spill_cnt, 1);
            if (e < S.spill_cap) {
                S.spill_rec[b][e] = rec;
                S.spill_key[b][e] = key;
                atomicOr(&S.spill_bits[b][dtile >> 5], 1u << (dtile & 31));
                atomicOr(S.err, ERR_SPILL);
            } else {
                atomicOr(S.err, ERR_LOST);
            }
        }
    }
}

__device__ __forceinline__ void warp_insert(const Sys &S, int b, bool act, int dtile, int region, int4 rec)
{
    warp_insert(S, b, act, dtile, region, rec, S.cnt[b], &S.spill_cnt[b]);
}

// ---------------------------------------------------------- tile context --
// Geometry of one tile and its neighbours' sizes.
struct TileGeo {
    int tx, ty, tw, th;
    int twL, twR, thD, thU;     // widths / heights of the neighbour tiles
};

struct TileCtx {
    Sys S;
    int sysi, tile, tx, ty, tw, th, W2, H2, nce;
    int twL, twR, thD, thU;     // widths / heights of the neighbour tiles
    int m_seg, n_spill, m, n_own;
    int part, parts;            // the update takes part `part` of `parts` of the tile's own particles
    int o_first, o_last;        // those: own indices (in cell order)
    int next;                   // index of the next tile this block takes
    int total, nsys;            // tiles and systems of the launch
    const int *tile_base;
    int pf_tile, pf_sys, pf_nsp;    // segments of the next tile, read ahead during this one
    TileGeo pf_geo;
    int segpre[kSegs + 1];
    int warp_tot[32];
    Seg seg[kSegs];
    Seg pf_seg[kSegs];
    long long red[5][32];
};

__device__ __forceinline__ int sys_of_tile(const int *tile_base, int nsys, int g)
{
    int lo = 0, hi = nsys;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (tile_base[mid] <= g) lo = mid; else hi = mid;
    }
    return lo;
}

// Resolve the halo column (side -1: left, +1: right) of tile t into a source
// tile column, the region column class there, and the position / cell maps.
__device__ __forceinline__ void resolve_axis(int side, int t, int nt, int w, int wlo, int refl, int s,
                                             int &src, int &cls, int &a, int &c, long long &b, int &flip)
{
    if (side == 0) {
        src = t; a = 1; c = 0; b = 0; flip = 0; cls = -1;
        return;
    }
    if (side < 0) {
        if (t > 0 || !refl) {
            src = (t > 0) ? t - 1 : nt - 1;
            cls = 2; a = 1; c = -wlo; b = -((long long)wlo << s); flip = 0;
        } else {        // mirror at the wall x = 0: X -> -X, cell 0 -> -1
            src = t; cls = 0; a = -1; c = -1; b = 0; flip = 1;
        }
    } else {
        if (t < nt - 1 || !refl) {
            src = (t < nt - 1) ? t + 1 : 0;
            cls = 0; a = 1; c = w; b = (long long)w << s; flip = 0;
        } else {        // mirror at the wall x = L: X -> 2 w 2^s - X, cell w-1 -> w
            src = t; cls = 2; a = -1; c = 2 * w - 1; b = 2 * ((long long)w << s); flip = 1;
        }
    }
}

__device__ __forceinline__ TileGeo tile_geo(const Sys &S, int tile)
{
    TileGeo G;
    G.tx = tile % S.ntx;
    G.ty = tile / S.ntx;
    const int x0 = S.x0tab[G.tx], y0 = S.y0tab[G.ty];
    G.tw = S.x0tab[G.tx + 1] - x0;
    G.th = S.y0tab[G.ty + 1] - y0;
    const int txl = G.tx > 0 ? G.tx - 1 : S.ntx - 1, txr = G.tx < S.ntx - 1 ? G.tx + 1 : 0;
    const int tyd = G.ty > 0 ? G.ty - 1 : S.nty - 1, tyu = G.ty < S.nty - 1 ? G.ty + 1 : 0;
    G.twL = S.x0tab[txl + 1] - S.x0tab[txl];
    G.twR = S.x0tab[txr + 1] - S.x0tab[txr];
    G.thD = S.y0tab[tyd + 1] - S.y0tab[tyd];
    G.thU = S.y0tab[tyu + 1] - S.y0tab[tyu];
    return G;
}

// Source segment s of a tile: s < 9 its own region s, then the 16 halo
// regions of the neighbour tiles (left, right, down, up edges, the corners)
// with their periodic shift or mirror map into the extended frame.
__device__ __forceinline__ Seg make_seg(const Sys &S, const TileGeo &G, int s, int cur)
{
    int bxo, byo, rx = -1, ry = -1;
    if (s < 9) {
        bxo = 0; byo = 0; rx = s % 3; ry = s / 3;
    } else {
        const int h = s - 9;
        if (h < 3)       { bxo = -1; byo = 0;  ry = h; }
        else if (h < 6)  { bxo = 1;  byo = 0;  ry = h - 3; }
        else if (h < 9)  { bxo = 0;  byo = -1; rx = h - 6; }
        else if (h < 12) { bxo = 0;  byo = 1;  rx = h - 9; }
        else { bxo = (h & 1) ? 1 : -1; byo = (h >= 14) ? 1 : -1; }
    }
    int srcx, clsx, ax, cx, fx, srcy, clsy, ay, cy, fy;
    long long bxx, byy;
    resolve_axis(bxo, G.tx, S.ntx, G.tw, G.twL, S.bx, S.sx, srcx, clsx, ax, cx, bxx, fx);
    resolve_axis(byo, G.ty, S.nty, G.th, G.thD, S.by, S.sy, srcy, clsy, ay, cy, byy, fy);
    if (clsx < 0) clsx = rx;
    if (clsy < 0) clsy = ry;
    Seg g;
    g.tile = srcy * S.ntx + srcx;
    g.region = clsy * 3 + clsx;
    g.base = S.rec[cur] + (long long)g.tile * S.tile_slots + S.off[g.region];
    const int c = S.cnt[cur][g.tile * kCntStride + g.region];
    g.count = min(c, S.cap[g.region]);
    g.ax = ax; g.ay = ay; g.cx = cx; g.cy = cy; g.bx = bxx; g.by = byy;
    g.flip = fx | (fy << 1);
    return g;
}

// Phase 1 of a tile: geometry, the 25 source segments (9 own regions, 16
// halo regions with their periodic or mirror maps), spill matches, and the
// number m of particles to stage.  The geometry and segments come from the
// read-ahead of the previous tile when it took this one.  Ends with the
// block synchronised.
template <int NT>
__device__ __forceinline__ void tile_setup(TileCtx &T, const Tables &tb, int cur, int nce_max,
                                           int *spill_e, unsigned char *spill_s, int spill_list_cap)
{
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const Sys &S = T.S;
    const bool pf = T.pf_tile == T.tile && T.pf_sys == T.sysi;
    const TileGeo G = pf ? T.pf_geo : tile_geo(S, T.tile);
    if (tid == 0) {
        T.tx = G.tx; T.ty = G.ty; T.tw = G.tw; T.th = G.th;
        T.W2 = G.tw + 2; T.H2 = G.th + 2; T.nce = (G.tw + 2) * (G.th + 2);
        T.twL = G.twL; T.twR = G.twR; T.thD = G.thD; T.thU = G.thU;
        T.n_spill = 0;
    }
    for (int i = tid; i < nce_max; i += NT) tb.hist[i] = 0;
    if (T.S.meas_until > 0)
        for (int i = tid; i < S.bins_theta + S.bins_nbr; i += NT) tb.mhist[i] = 0;
    if (tid < kSegs) T.seg[tid] = pf ? T.pf_seg[tid] : make_seg(S, G, tid, cur);
    const int nsp = pf ? T.pf_nsp : min(*((volatile int *)&S.spill_cnt[cur]), S.spill_cap);
    __syncthreads();
    if (tid == 0) T.pf_tile = -1;       // consumed (the read-ahead for the next tile comes later)
    if (warp == 0) {
        const int v = lane < kSegs ? T.seg[lane].count : 0;
        const int incl = warp_incl_scan(v);
        if (lane < kSegs) T.segpre[lane] = incl - v;
        if (lane == kSegs - 1) {
            T.segpre[kSegs] = incl;
            T.m_seg = incl;
        }
    }
    if (nsp > 0) {
        // particles parked in the spill list for one of our segments
        for (int e = tid; e < nsp; e += NT) {
            const int key = S.spill_key[cur][e];
            const int et = key / kCntStride, er = key % kCntStride;
            for (int s = 0; s < kSegs; ++s) {
                if (T.seg[s].tile == et && T.seg[s].region == er) {
                    const int j = atomicAdd(&T.n_spill, 1);
                    if (j < spill_list_cap) {
                        spill_e[j] = e;
                        spill_s[j] = (unsigned char)s;
                    }
                }
            }
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (T.n_spill > spill_list_cap) {
            atomicOr(S.err, ERR_STAGE);
            T.n_spill = spill_list_cap;
        }
        T.m = T.m_seg + T.n_spill;
    }
    __syncthreads();
}

// The 3x3-cell neighbour sum of one particle (Eq. collision_VM / NVM, or the
// Langevin coupling sum): rows of three consecutive cells are contiguous in
// the cell order.  The particle itself is included: it adds e^{i theta_i} to
// the VM/NVM sum and sin 0 to the Langevin sum; cnt counts it.  The staged
// (cos, sin) are integers in units of 2^-22 (kFixNb), so the sums are exact and
// do not depend on the order of the particles inside a cell.  ACC is int for
// at most 511 candidates (|sum| < 2^31) and long long beyond.
template <int MODEL, typename ACC>
__device__ __forceinline__ void neighbour_sum(const float4 *__restrict__ P, const int *cstart, int ec,
                                              int W2, float4 pi, float r2, ACC &sc, ACC &ss, int &cnt)
{
    sc = 0;
    ss = 0;
    cnt = 0;
    const float pcf = (float)__float_as_int(pi.z), psf = (float)__float_as_int(pi.w);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
        const int c0 = ec + dy * W2 - 1;
        const int a = cstart[c0], b = cstart[c0 + 3];
#pragma unroll 4
        for (int j = a; j < b; ++j) {
            const float4 pj = P[j];
            const float dx = pj.x - pi.x, dyy = pj.y - pi.y;
            const float d2 = fmaf(dx, dx, dyy * dyy);
            if (d2 <= r2) {
                int cj = __float_as_int(pj.z), sj = __float_as_int(pj.w);
                if (MODEL == 2 && fmaf(pcf, (float)cj, psf * (float)sj) < 0.f) {
                    cj = -cj;                         // Eq. (collision_NVM): the reversed direction
                    sj = -sj;
                }
                sc += cj;
                ss += sj;
                ++cnt;
            }
        }
    }
}

// Langevin sums with per-species couplings (Sec. 2.5): each neighbour's
// (cos o theta_j, sin o theta_j) weighted by grow[species of j] = Gamma_{s_i s_j} dt,
// rounded to integers in units of 2^-22 and summed exactly (order-free).
__device__ __forceinline__ void neighbour_sum_sp(const float4 *__restrict__ P, const unsigned short *spc,
                                                 const int *cstart, int ec, int W2, float4 pi, float r2,
                                                 const float *grow, long long &sc, long long &ss, int &cnt)
{
    sc = 0;
    ss = 0;
    cnt = 0;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
        const int c0 = ec + dy * W2 - 1;
        const int a = cstart[c0], b = cstart[c0 + 3];
        for (int j = a; j < b; ++j) {
            const float4 pj = P[j];
            const float dx = pj.x - pi.x, dyy = pj.y - pi.y;
            if (fmaf(dx, dx, dyy * dyy) <= r2) {
                const float g = grow[spc[j]];
                sc += __float2ll_rn(g * (float)__float_as_int(pj.z));
                ss += __float2ll_rn(g * (float)__float_as_int(pj.w));
                ++cnt;
            }
        }
    }
}

// First own index (own particles in row, cell order) of part k of K of a
// tile: the first start of a cell at or after the share n_own k / K, so that
// the parts do not depend on the arrival order inside a cell and are the same
// for every block that sorts the tile.  row_start(r), cell_start(r, c): own
// index of the first particle of own row r / of its own cell c or a later one.
// Every lane of the warp calls.
template <class R, class C>
__device__ __forceinline__ int part_start(int k, int K, int n_own, int tw, int th, R &&row_start, C &&cell_start)
{
    if (k <= 0) return 0;
    if (k >= K) return n_own;
    const int lane = threadIdx.x & 31;
    const int target = (int)((long long)n_own * k / K);
    int row = 0;                                        // the last row that starts at or before the share
    for (int r0 = 0; r0 < th; r0 += 32) {
        const unsigned b = __ballot_sync(0xffffffffu, r0 + lane < th && row_start(r0 + lane) <= target);
        if (b) row = r0 + 31 - __clz(b);
    }
    for (int c0 = 0; c0 < tw; c0 += 32) {
        const int s = c0 + lane < tw ? cell_start(row, c0 + lane) : -1;
        const unsigned b = __ballot_sync(0xffffffffu, s >= target);
        if (b) return __shfl_sync(0xffffffffu, s, __ffs(b) - 1);
    }
    return row + 1 < th ? row_start(row + 1) : n_own;
}

// Phase 2 of a tile, staged in A (shared memory or the block's scratch).
template <int NT, int MODEL>
__device__ __forceinline__ void tile_body(TileCtx &T, const Stage &A, const Tables &tb, long long step,
                                          const int *spill_e, const unsigned char *spill_s, int next_g)
{
    const int tid = threadIdx.x;
    const int lane = tid & 31, warp = tid >> 5;
    const Sys &S = T.S;
    const int cur = (int)(step & 1), nxt = cur ^ 1;
    const int m = T.m, m_seg = T.m_seg, W2 = T.W2, H2 = T.H2, nce = T.nce;
    const int tw = T.tw, th = T.th;
    PHASE_START();

    // --- segment of every 32nd staged index (chunk table) ---------------
    for (int i = tid; i * 32 < m_seg; i += NT) {
        const int k = i * 32;
        int lo = 0, hi = kSegs;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (T.segpre[mid] <= k) lo = mid; else hi = mid;
        }
        A.segc[i] = (unsigned char)lo;
    }
    __syncthreads();

    // --- stage: decode, map into the extended frame, histogram by cell ----
    for (int k = tid; k < m; k += NT) {
        int s;
        int4 r;
        if (k < m_seg) {
            s = A.segc[k >> 5];
            while (T.segpre[s + 1] <= k) ++s;
            r = T.seg[s].base[k - T.segpre[s]];
        } else {
            const int j = k - m_seg;
            s = spill_s[j];
            r = S.spill_rec[cur][spill_e[j]];
        }
        const Seg &g = T.seg[s];
        const int lx = r.x >> S.sx, ly = r.y >> S.sy;
        int ex = g.ax * lx + g.cx + 1, ey = g.ay * ly + g.cy + 1;
        if ((unsigned)ex >= (unsigned)W2 || (unsigned)ey >= (unsigned)H2) {
            atomicOr(S.err, ERR_BOUNDS);
            ex = min(max(ex, 0), W2 - 1);
            ey = min(max(ey, 0), H2 - 1);
        }
        const int ec = ey * W2 + ex;
        A.R[k] = make_int4((int)(g.ax * (long long)r.x + g.bx), (int)(g.ay * (long long)r.y + g.by), r.z, r.w);
        A.cell[k] = (unsigned short)(ec | (g.flip << 14));
        A.slot[k] = (unsigned short)atomicAdd(&tb.hist[ec], 1);
    }
    // the next tile's index, fetched by thread 0 at the start of this tile:
    // published only now, so that no warp waited for the atomic's round trip
    if (tid == 0) T.next = next_g;
    __syncthreads();
    PHASE_MARK(0);

    // --- block-level exclusive prefix scan of the cell histogram ----------
    {
        const int per = (nce + NT - 1) / NT;
        const int b0 = min(tid * per, nce), e0 = min(b0 + per, nce);
        int sum = 0;
        for (int i = b0; i < e0; ++i) sum += tb.hist[i];
        const int incl = warp_incl_scan(sum);
        if (lane == 31) T.warp_tot[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const int v = lane < NT / 32 ? T.warp_tot[lane] : 0;
            const int wi = warp_incl_scan(v);
            if (lane < NT / 32) T.warp_tot[lane] = wi - v;
            if (lane == NT / 32 - 1) tb.cstart[nce] = wi;
        }
        __syncthreads();
        int run = incl - sum + T.warp_tot[warp];
        for (int i = b0; i < e0; ++i) {
            tb.cstart[i] = run;
            run += tb.hist[i];
        }
    }
    __syncthreads();
    PHASE_MARK(1);

    // --- records into cell order (arrival order inside a cell: the sums are
    //     exact integers, so this order does not matter); own rows prefix ---
    const int xc = tw << (S.sx - 1), yc = th << (S.sy - 1);
    for (int k = tid; k < m; k += NT) {
        const unsigned short cf = A.cell[k];
        const int c = cf & 0x3fff;
        const int q = tb.cstart[c] + A.slot[k];
        const int4 rk = A.R[k];
        float thv = __int_as_float(rk.z);
        float sn, cs;
        if (MODEL == 1 && S.order != 1) {
            thv *= (float)S.order;
            sincosf(thv, &sn, &cs);
        } else {
            // |theta| <= pi: the hardware sine/cosine is within 2^-21.4 absolute
            __sincosf(thv, &sn, &cs);
        }
        const int flip = cf >> 14;
        if (flip & 1) {
            if (MODEL != 1 || (S.order & 1)) cs = -cs; else sn = -sn;
        }
        if (flip & 2) sn = -sn;
        A.P[q] = make_float4((float)(rk.x - xc) * S.ux, (float)(rk.y - yc) * S.uy,
                             __int_as_float(__float2int_rn(cs * kFixNbF)), __int_as_float(__float2int_rn(sn * kFixNbF)));
        A.sk[q] = (unsigned short)k;
        if (S.nsp > 1) A.gidx[q] = (unsigned short)species_of(S, (unsigned)rk.w);   // species by sorted position
    }
    if (warp == NT / 32 - 1) {
        int carry = 0;
        for (int r0 = 0; r0 < th; r0 += 32) {
            const int r = r0 + lane;
            int len = 0;
            if (r < th) len = tb.cstart[(r + 1) * W2 + tw + 1] - tb.cstart[(r + 1) * W2 + 1];
            const int incl = warp_incl_scan(len);
            if (r < th) tb.rowpre[r] = carry + incl - len;
            carry += __shfl_sync(0xffffffffu, incl, 31);
        }
        if (lane == 0) {
            tb.rowpre[th] = carry;
            T.n_own = carry;
        }
        int first = 0, last = carry;
        if (T.parts > 1) {
            __syncwarp();
            const auto row_start = [&](int r) { return tb.rowpre[r]; };
            const auto cell_start = [&](int r, int c) {
                return tb.rowpre[r] + tb.cstart[(r + 1) * W2 + 1 + c] - tb.cstart[(r + 1) * W2 + 1];
            };
            first = part_start(T.part, T.parts, carry, tw, th, row_start, cell_start);
            last = part_start(T.part + 1, T.parts, carry, tw, th, row_start, cell_start);
        }
        if (lane == 0) {
            T.o_first = first;
            T.o_last = last;
        }
    }
    __syncthreads();
    PHASE_MARK(2);
    PHASE_MARK(3);

    // --- interact, update, scatter ---------------------------------------
    const int o_last = T.o_last;
    const float r2 = S.r2;
    const int TWs = tw << S.sx, THs = th << S.sy;
    const bool measure = step < S.meas_until;   // on-the-fly histograms (Sec. 3.4)
    long long acc_c = 0, acc_s = 0, acc_n = 0, acc_c2 = 0, acc_s2 = 0;
    for (int base = T.o_first; base < o_last; base += NT) {
        const int o = base + tid;
        const bool act = o < o_last;
        int4 rec = make_int4(0, 0, 0, 0);
        int dtile = 0, region = 0;
        if (act) {
            // own particle o -> sorted position: the own row holding it
            int rlo = 0, rhi = th;
            while (rhi - rlo > 1) {
                const int mid = (rlo + rhi) >> 1;
                if (tb.rowpre[mid] <= o) rlo = mid; else rhi = mid;
            }
            const int q = tb.cstart[(rlo + 1) * W2 + 1] + (o - tb.rowpre[rlo]);
            const int k = A.sk[q];
            const int4 rk = A.R[k];
            const int X = rk.x, Y = rk.y;
            const float thi = __int_as_float(rk.z);
            const unsigned id = (unsigned)rk.w;
            const int ec = A.cell[k] & 0x3fff;
            const float4 pi = A.P[q];
            float sc, ss;                    // neighbour sums in units of 2^-22
            int cnt;
            const int sp = S.nsp > 1 ? species_of(S, id) : 0;
            if (MODEL == 1 && S.nsp > 1) {
                long long a, b;
                neighbour_sum_sp(A.P, A.gidx, tb.cstart, ec, W2, pi, r2, S.sp_gamma_dt + sp * kMaxSpecies, a, b,
                                 cnt);
                sc = (float)a;
                ss = (float)b;
            } else {
                const int ncand = tb.cstart[ec - W2 + 2] - tb.cstart[ec - W2 - 1] + tb.cstart[ec + 2] -
                                  tb.cstart[ec - 1] + tb.cstart[ec + W2 + 2] - tb.cstart[ec + W2 - 1];
                if (ncand < 512) {
                    int a, b;
                    neighbour_sum<MODEL, int>(A.P, tb.cstart, ec, W2, pi, r2, a, b, cnt);
                    sc = (float)a;
                    ss = (float)b;
                } else {
                    long long a, b;
                    neighbour_sum<MODEL, long long>(A.P, tb.cstart, ec, W2, pi, r2, a, b, cnt);
                    sc = (float)a;
                    ss = (float)b;
                }
            }
            const int nb = cnt - 1;          // the particle itself was counted
            if (measure) {
                int bt = (int)floorf((thi + AAP_PI_F) * ((float)S.bins_theta * (1.0f / AAP_2PI_F)));
                bt = min(max(bt, 0), S.bins_theta - 1);
                atomicAdd(&tb.mhist[bt], 1);
                atomicAdd(&tb.mhist[S.bins_theta + min(nb, S.bins_nbr - 1)], 1);
            }
            uint32_t c4[4] = {id, (uint32_t)step, (uint32_t)((unsigned long long)step >> 32), 0u};
            philox4x32_10(c4, S.seed_lo, S.seed_hi);
            const float u0 = u01f(c4[0]);
            float thn, cn, sn;
            int dX, dY;
            if (MODEL != 1) {
                // Eq. (collision_VM) / (collision_NVM) + noise; Eq. (streaming)
                thn = arg2(ss, sc) + S.sp_omega_step[sp] + S.sp_eta_pi[sp] * (2.0f * u0 - 1.0f);
                __sincosf(thn, &sn, &cn);
                dX = __float2int_rn(S.sp_kx[sp] * cn);
                dY = __float2int_rn(S.sp_ky[sp] * sn);
            } else {
                // Eq. (Langevin_dynamics), one Euler-Maruyama step
                const float u1 = u01f(c4[1]);
                const float h = S.wlen > 0 ? S.wtab[min(nb, S.wlen - 1)]
                                           : (S.weight ? 1.0f : 1.0f / (1.0f + (float)nb));
                // sum_j sin(o (theta_j - theta_i)) from the exact sums (units 2^-22 x 2^-22);
                // Gamma dt inside with several species
                const float tsum = ((float)__float_as_int(pi.z) * ss - (float)__float_as_int(pi.w) * sc) *
                                   (1.0f / (kFixNbF * kFixNbF));
                const float gz = sqrtf(-2.0f * logf(u0)) * cospif(2.0f * u1);
                const float drift = S.nsp > 1 ? h * tsum : S.gamma_dt * h * tsum;
                thn = thi + drift + S.sp_omega_step[sp] + S.sp_noise_amp[sp] * gz;
                float co, so;
                __sincosf(thi, &so, &co);    // streaming direction theta(t), |theta| <= pi
                dX = __float2int_rn(S.sp_kx[sp] * co);
                dY = __float2int_rn(S.sp_ky[sp] * so);
                cn = 0.f;
                sn = 0.f;
            }
            // boundary rule (Sec. 2.4) in exact fixed point
            int Xn = X + dX, Yn = Y + dY;
            int dtx = T.tx, dty = T.ty, twd = tw, thd = th;
            bool fx = false, fy = false;
            if (Xn < 0) {
                if (S.bx && T.tx == 0) { Xn = -Xn; fx = true; }
                else { dtx = T.tx > 0 ? T.tx - 1 : S.ntx - 1; twd = T.twL; Xn += T.twL << S.sx; }
            } else if (Xn >= TWs) {
                if (S.bx && T.tx == S.ntx - 1) {
                    if (Xn == TWs) Xn = TWs - 1; else { Xn = TWs - (Xn - TWs); fx = true; }
                } else { dtx = T.tx < S.ntx - 1 ? T.tx + 1 : 0; twd = T.twR; Xn -= TWs; }
            }
            if (Yn < 0) {
                if (S.by && T.ty == 0) { Yn = -Yn; fy = true; }
                else { dty = T.ty > 0 ? T.ty - 1 : S.nty - 1; thd = T.thD; Yn += T.thD << S.sy; }
            } else if (Yn >= THs) {
                if (S.by && T.ty == S.nty - 1) {
                    if (Yn == THs) Yn = THs - 1; else { Yn = THs - (Yn - THs); fy = true; }
                } else { dty = T.ty < S.nty - 1 ? T.ty + 1 : 0; thd = T.thU; Yn -= THs; }
            }
            if (fx) { thn = AAP_PI_F - thn; cn = -cn; }
            if (fy) { thn = -thn; sn = -sn; }
            if (thn >= AAP_PI_F || thn < -AAP_PI_F)
                thn -= AAP_2PI_F * floorf((thn + AAP_PI_F) * (1.0f / AAP_2PI_F));
            if (MODEL == 1) __sincosf(thn, &sn, &cn);
            if (!isfinite(thn)) atomicOr(S.err, ERR_NAN);
            dtile = dty * S.ntx + dtx;
            region = region_of(Xn >> S.sx, Yn >> S.sy, twd, thd);
            rec = make_int4(Xn, Yn, __float_as_int(thn), (int)id);
            acc_c += __float2int_rn(cn * kFixStepF);
            acc_s += __float2int_rn(sn * kFixStepF);
            acc_c2 += __float2int_rn(fmaf(cn, cn, -sn * sn) * kFixStepF);
            acc_s2 += __float2int_rn(2.0f * cn * sn * kFixStepF);
            acc_n += nb;
            if (S.nbr_out && id < (unsigned long long)S.n) S.nbr_out[id] = nb;
        }
        warp_insert(S, nxt, act, dtile, region, rec);
    }
    // --- read ahead: the last warp (often idle in the last round of the
    //     update) prepares the next tile's geometry and segments, so that the
    //     next tile_setup starts without its chain of global loads ----------
    if (warp == NT / 32 - 1 && T.next < T.total) {
        const int g = T.next;
        const int si = T.nsys > 1 ? sys_of_tile(T.tile_base, T.nsys, g) : 0;
        if (si == T.sysi) {
            const TileGeo G = tile_geo(S, g - (T.nsys > 1 ? T.tile_base[si] : 0));
            if (lane < kSegs) T.pf_seg[lane] = make_seg(S, G, lane, cur);
            if (lane == 0) {
                T.pf_geo = G;
                T.pf_nsp = min(*((volatile int *)&S.spill_cnt[cur]), S.spill_cap);
                T.pf_tile = g - (T.nsys > 1 ? T.tile_base[si] : 0);
                T.pf_sys = si;
            }
        }
    }
    PHASE_MARK(4);
    // --- per-tile integer sums -> the step's accumulators ----------------
    acc_c = warp_sum_ll(acc_c);
    acc_s = warp_sum_ll(acc_s);
    acc_n = warp_sum_ll(acc_n);
    acc_c2 = warp_sum_ll(acc_c2);
    acc_s2 = warp_sum_ll(acc_s2);
    if (lane == 0) {
        T.red[0][warp] = acc_c;
        T.red[1][warp] = acc_s;
        T.red[2][warp] = acc_n;
        T.red[3][warp] = acc_c2;
        T.red[4][warp] = acc_s2;
    }
    __syncthreads();
    if (tid < 5) {
        long long v = 0;
        for (int w = 0; w < NT / 32; ++w) v += T.red[tid][w];
        unsigned long long *slot = S.acc + ((size_t)cur * kAccSlots + (T.tile & (kAccSlots - 1))) * kAccWords;
        atomicAdd(slot + tid, (unsigned long long)v);
    }
    if (measure) {
        for (int i = tid; i < S.bins_theta + S.bins_nbr; i += NT)
            if (tb.mhist[i]) atomicAdd(S.hist + i, (unsigned long long)tb.mhist[i]);
    }
    PHASE_MARK(5);
}

// What the update needs of a tile sorted by half cell.
struct OutMeta {
    int tile;                   // -1: no more tiles, -2: skip (the buffer holds part of a wide tile)
    int rbuf, rwide;            // raw buffer of the tile's staged records, and whether it spans the next one too
    int o_first, n_own;         // the own particles to update: o_first .. n_own - 1
    int tx, ty, tw, th, W2, twL, twR, thD, thU;   // W2: half cells per extended row, 2 tw + 4
    int wide;                   // a half cell holds enough particles for 512 candidates
    int dense;                  // more than 1.5 staged records per half cell on average
};

// ------------------------------------ the update of a half-cell-sorted tile --
// The neighbour sum of one particle over three rows of five half cells,
// each row contiguous in the half-cell order.  The particle itself is
// included (it adds e^{i theta_i} to the VM/NVM sum and sin 0 to the
// Langevin sum; cnt counts it).  The staged (cos, sin) are integers in units
// of 2^-22, so the sums are exact and order-free; ACC is int below 512
// candidates and long long beyond.  LPP lanes share a particle: lane `sub` of
// them takes every LPP-th candidate of a row (the callers add the shares up).
template <int MODEL, typename ACC, int UNR, int LPP = 1>
__device__ __forceinline__ void neighbour_sum_h(const float4 *__restrict__ P, const unsigned short *cstart, int ec,
                                                int W2, float4 pi, float r2, ACC &sc, ACC &ss, int &cnt, int sub = 0)
{
    sc = 0;
    ss = 0;
    cnt = 0;
    const float pcf = (float)__float_as_int(pi.z), psf = (float)__float_as_int(pi.w);
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
        const int c0 = ec + dy * W2 - 2;
        const int a = cstart[c0], b = cstart[c0 + 5];
#pragma unroll UNR
        for (int j = LPP > 1 ? a + sub : a; j < b; j += LPP) {
            const float4 pj = P[j];
            const float dx = pj.x - pi.x, dyy = pj.y - pi.y;
            const float d2 = fmaf(dx, dx, dyy * dyy);
            if (d2 <= r2) {
                int cj = __float_as_int(pj.z), sj = __float_as_int(pj.w);
                if (MODEL == 2 && fmaf(pcf, (float)cj, psf * (float)sj) < 0.f) {
                    cj = -cj;                         // Eq. (collision_NVM): the reversed direction
                    sj = -sj;
                }
                sc += cj;
                ss += sj;
                ++cnt;
            }
        }
    }
}

constexpr float kMagicF = 12582912.0f;              // 1.5 2^23
constexpr unsigned kMagicBits = 0x4B400000u;
__device__ __forceinline__ float stage_cos_species(int c, int sp)
{
    return __uint_as_float(((kMagicBits + (unsigned)c) & 0x00ffffffu) | ((unsigned)sp << 24));
}
__device__ __forceinline__ float staged_cos(float z)
{
    return __uint_as_float((__float_as_uint(z) & 0x00ffffffu) | 0x4B000000u) - kMagicF;
}

// (cos, sin) of a sorted record as the update reads it.
template <int MODEL, bool SP>
__device__ __forceinline__ void stage_angle(const Sys &S, int id, int c, int s, float &zc, float &zs)
{
    if (SP && MODEL == 1) {
        zc = stage_cos_species(c, species_of(S, (unsigned)id));
        zs = (float)s;
    } else {
        zc = __int_as_float(c);
        zs = __int_as_float(s);
    }
}

// The Langevin sums with per-species couplings (neighbour_sum_sp above) over
// the half cells, for couplings and candidate numbers of any size (out of
// line: its 64-bit conversions run on the narrow FP64 pipe, and inlined the
// compiler predicates them into every neighbour's path).
template <int LPP>
__device__ __noinline__ void neighbour_sum_sp_h(const float4 *__restrict__ P, const unsigned short *cstart, int ec,
                                                int W2, float4 pi, float r2, const float *grow, long long *out, int sub)
{
    long long sc = 0, ss = 0;
    int cnt = 0;
    for (int dy = -1; dy <= 1; ++dy) {
        const int c0 = ec + dy * W2 - 2;
        const int a = cstart[c0], b = cstart[c0 + 5];
        for (int j = LPP > 1 ? a + sub : a; j < b; j += LPP) {
            const float4 pj = P[j];
            const float dx = pj.x - pi.x, dyy = pj.y - pi.y;
            if (fmaf(dx, dx, dyy * dyy) <= r2) {
                const float g = grow[__float_as_uint(pj.z) >> 24];
                sc += __float2ll_rn(g * staged_cos(pj.z));
                ss += __float2ll_rn(g * pj.w);
                ++cnt;
            }
        }
    }
    out[0] = sc;
    out[1] = ss;
    out[2] = cnt;
}

// The same sums when every |Gamma dt| is below 1 and there are fewer than 512
// candidates.  A staged record then holds its cosine c (an integer, |c| <=
// 2^22) as the low 24 bits of the float 1.5 2^23 + c with its species above
// them, and its sine as a float.  Gamma c is rounded to an integer as the bits
// of fl(Gamma c) + 1.5 2^23 (one addition whose rounding lands on an integer,
// ties to even: what __float2ll_rn(fl(Gamma c)) gives for |Gamma c| <= 2^22),
// so that no conversion runs per neighbour; the sum of n such words minus n
// biases is the exact integer sum (below 2^31).
template <int UNR, int LPP>
__device__ __forceinline__ void neighbour_sum_spm(const float4 *__restrict__ P, const unsigned short *cstart, int ec,
                                                  int W2, float4 pi, float r2, const float *grow, int &sc, int &ss,
                                                  int &cnt, int sub)
{
    unsigned wc = 0, ws = 0;
    cnt = 0;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
        const int c0 = ec + dy * W2 - 2;
        const int a = cstart[c0], b = cstart[c0 + 5];
#pragma unroll UNR
        for (int j = LPP > 1 ? a + sub : a; j < b; j += LPP) {
            const float4 pj = P[j];
            const float dx = pj.x - pi.x, dyy = pj.y - pi.y;
            if (fmaf(dx, dx, dyy * dyy) <= r2) {
                const float g = grow[__float_as_uint(pj.z) >> 24];
                wc += __float_as_uint(__fadd_rn(__fmul_rn(g, staged_cos(pj.z)), kMagicF));
                ws += __float_as_uint(__fadd_rn(__fmul_rn(g, pj.w), kMagicF));
                ++cnt;
            }
        }
    }
    sc = (int)(wc - kMagicBits * (unsigned)cnt);
    ss = (int)(ws - kMagicBits * (unsigned)cnt);
}

struct Acc {
    long long c, s, n, c2, s2;
};

// The system's own counters of its buffer `nxt`.
struct ToSystem {
    __device__ __forceinline__ int *cnt(const Sys &S, int nxt) const { return S.cnt[nxt]; }
    __device__ __forceinline__ int *spill(const Sys &S, int nxt) const { return &S.spill_cnt[nxt]; }
};

// One particle per lane (own index o, inactive when o >= n_own); every lane
// of the warp must call (the scatter is warp-aggregated).  `to` names the
// counters of the buffer the new records go to, asked for only where they are
// used (registers).  SP: several species (each
// particle's speed, noise and chirality looked up by its id).  LPP: lanes per
// particle (a power of two; o is the same for each group of LPP lanes).
template <int MODEL, bool SP, int LPP, class TO>
__device__ __forceinline__ void update_one(const Sys &S, const OutMeta &O, const float4 *__restrict__ P,
                                           const unsigned short *cstart, const int4 *RB, const unsigned short *OR,
                                           const unsigned short *OQ,
                                           int o, long long step, bool measure, int *mhist, Acc &acc,
                                           const TO &to)
{
    const int nxt = (int)(step & 1) ^ 1;
    const int sub = LPP > 1 ? (int)(threadIdx.x & (LPP - 1)) : 0;
    const unsigned group = ((1u << LPP) - 1u) << (threadIdx.x & 31 & ~(LPP - 1));   // the particle's lanes
    bool act = o < O.n_own;
    int4 rec = make_int4(0, 0, 0, 0);
    int dtile = 0, region = 0;
    int X = 0, Y = 0, cnt = 0, sp = 0;
    float thi = 0.f, sc = 0.f, ss = 0.f;     // neighbour sums in units of 2^-22
    unsigned id = 0;
    float4 pi = make_float4(0.f, 0.f, 0.f, 0.f);
    const int tw = O.tw, th = O.th;
    if (act) {
        const int W2 = O.W2;
        const int4 rk = RB[OR[o]];                // own regions map to themselves (no shift, no mirror)
        X = rk.x;
        Y = rk.y;
        thi = __int_as_float(rk.z);
        id = (unsigned)rk.w;
        const int ec = ((Y >> S.sy) + 1) * W2 + (X >> (S.sx - 1)) + 2;      // extended half cell
        pi = P[OQ[o]];
        sp = SP ? species_of(S, id) : 0;
        bool narrow = !O.wide;
        if (SP && MODEL == 1) {
            const float *grow = S.sp_gamma_dt + sp * kMaxSpecies;
            if (S.small_gamma && narrow) {
                int a, b;
                neighbour_sum_spm<2, LPP>(P, cstart, ec, W2, pi, S.r2, grow, a, b, cnt, sub);
#pragma unroll
                for (int d = 1; d < LPP; d <<= 1) {
                    a += __shfl_xor_sync(group, a, d);
                    b += __shfl_xor_sync(group, b, d);
                }
                sc = (float)a;
                ss = (float)b;
            } else {
                long long out[3];
                neighbour_sum_sp_h<LPP>(P, cstart, ec, W2, pi, S.r2, grow, out, sub);
                cnt = (int)out[2];
#pragma unroll
                for (int d = 1; d < LPP; d <<= 1) {
                    out[0] += __shfl_xor_sync(group, out[0], d);
                    out[1] += __shfl_xor_sync(group, out[1], d);
                }
                sc = (float)out[0];
                ss = (float)out[1];
            }
            pi.z = __int_as_float((int)staged_cos(pi.z));       // as the other models stage them
            pi.w = __int_as_float((int)pi.w);
        } else {
            if (!narrow) {
                const int ncand = cstart[ec - W2 + 3] - cstart[ec - W2 - 2] + cstart[ec + 3] - cstart[ec - 2] +
                                  cstart[ec + W2 + 3] - cstart[ec + W2 - 2];
                narrow = ncand < 512;
            }
            if (narrow) {
                // short candidate rows run faster unrolled twice, long ones
                // (dense tiles) four times
                int a, b;
                if (O.dense) neighbour_sum_h<MODEL, int, 4, LPP>(P, cstart, ec, W2, pi, S.r2, a, b, cnt, sub);
                else neighbour_sum_h<MODEL, int, 2, LPP>(P, cstart, ec, W2, pi, S.r2, a, b, cnt, sub);
#pragma unroll
                for (int d = 1; d < LPP; d <<= 1) {
                    a += __shfl_xor_sync(group, a, d);
                    b += __shfl_xor_sync(group, b, d);
                }
                sc = (float)a;
                ss = (float)b;
            } else {
                long long a, b;
                neighbour_sum_h<MODEL, long long, 4, LPP>(P, cstart, ec, W2, pi, S.r2, a, b, cnt, sub);
#pragma unroll
                for (int d = 1; d < LPP; d <<= 1) {
                    a += __shfl_xor_sync(group, a, d);
                    b += __shfl_xor_sync(group, b, d);
                }
                sc = (float)a;
                ss = (float)b;
            }
        }
#pragma unroll
        for (int d = 1; d < LPP; d <<= 1) cnt += __shfl_xor_sync(group, cnt, d);
    }
    if (LPP > 1) act = act && sub == 0;
    if (act) {
        const int nb = cnt - 1;          // the particle itself was counted
        if (measure) {
            int bt = (int)floorf((thi + AAP_PI_F) * ((float)S.bins_theta * (1.0f / AAP_2PI_F)));
            bt = min(max(bt, 0), S.bins_theta - 1);
            atomicAdd(&mhist[bt], 1);
            atomicAdd(&mhist[S.bins_theta + min(nb, S.bins_nbr - 1)], 1);
        }
        uint32_t c4[4] = {id, (uint32_t)step, (uint32_t)((unsigned long long)step >> 32), 0u};
        philox4x32_10(c4, S.seed_lo, S.seed_hi);
        const float u0 = u01f(c4[0]);
        float thn, cn, sn;
        int dX, dY;
        if (MODEL != 1) {
            // Eq. (collision_VM) / (collision_NVM) + noise; Eq. (streaming)
            thn = arg2(ss, sc) + (SP ? S.sp_omega_step[sp] : S.omega_step) +
                  (SP ? S.sp_eta_pi[sp] : S.eta_pi) * (2.0f * u0 - 1.0f);
            __sincosf(thn, &sn, &cn);
            dX = __float2int_rn((SP ? S.sp_kx[sp] : S.kx) * cn);
            dY = __float2int_rn((SP ? S.sp_ky[sp] : S.ky) * sn);
        } else {
            // Eq. (Langevin_dynamics), one Euler-Maruyama step
            const float u1 = u01f(c4[1]);
            const float h = S.wlen > 0 ? S.wtab[min(nb, S.wlen - 1)]
                                       : (S.weight ? 1.0f : 1.0f / (1.0f + (float)nb));
            // sum_j sin(o (theta_j - theta_i)) from the exact sums (units 2^-22 x 2^-22);
            // Gamma dt inside with several species
            const float tsum = ((float)__float_as_int(pi.z) * ss - (float)__float_as_int(pi.w) * sc) *
                               (1.0f / (kFixNbF * kFixNbF));
            const float gz = sqrtf(-2.0f * logf(u0)) * cospif(2.0f * u1);
            const float drift = SP ? h * tsum : S.gamma_dt * h * tsum;
            thn = thi + drift + (SP ? S.sp_omega_step[sp] : S.omega_step) + (SP ? S.sp_noise_amp[sp] : S.noise_amp) * gz;
            float co, so;
            __sincosf(thi, &so, &co);    // streaming direction theta(t), |theta| <= pi
            dX = __float2int_rn((SP ? S.sp_kx[sp] : S.kx) * co);
            dY = __float2int_rn((SP ? S.sp_ky[sp] : S.ky) * so);
            cn = 0.f;
            sn = 0.f;
        }
        // boundary rule (Sec. 2.4) in exact fixed point
        const int TWs = tw << S.sx, THs = th << S.sy;
        int Xn = X + dX, Yn = Y + dY;
        int dtx = O.tx, dty = O.ty, twd = tw, thd = th;
        bool fx = false, fy = false;
        if (Xn < 0) {
            if (S.bx && O.tx == 0) { Xn = -Xn; fx = true; }
            else { dtx = O.tx > 0 ? O.tx - 1 : S.ntx - 1; twd = O.twL; Xn += O.twL << S.sx; }
        } else if (Xn >= TWs) {
            if (S.bx && O.tx == S.ntx - 1) {
                if (Xn == TWs) Xn = TWs - 1; else { Xn = TWs - (Xn - TWs); fx = true; }
            } else { dtx = O.tx < S.ntx - 1 ? O.tx + 1 : 0; twd = O.twR; Xn -= TWs; }
        }
        if (Yn < 0) {
            if (S.by && O.ty == 0) { Yn = -Yn; fy = true; }
            else { dty = O.ty > 0 ? O.ty - 1 : S.nty - 1; thd = O.thD; Yn += O.thD << S.sy; }
        } else if (Yn >= THs) {
            if (S.by && O.ty == S.nty - 1) {
                if (Yn == THs) Yn = THs - 1; else { Yn = THs - (Yn - THs); fy = true; }
            } else { dty = O.ty < S.nty - 1 ? O.ty + 1 : 0; thd = O.thU; Yn -= THs; }
        }
        if (fx) { thn = AAP_PI_F - thn; cn = -cn; }
        if (fy) { thn = -thn; sn = -sn; }
        if (thn >= AAP_PI_F || thn < -AAP_PI_F)
            thn -= AAP_2PI_F * floorf((thn + AAP_PI_F) * (1.0f / AAP_2PI_F));
        if (MODEL == 1) __sincosf(thn, &sn, &cn);
        if (!isfinite(thn)) atomicOr(S.err, ERR_NAN);
        dtile = dty * S.ntx + dtx;
        region = region_of(Xn >> S.sx, Yn >> S.sy, twd, thd);
        rec = make_int4(Xn, Yn, __float_as_int(thn), (int)id);
        acc.c += __float2int_rn(cn * kFixStepF);
        acc.s += __float2int_rn(sn * kFixStepF);
        acc.c2 += __float2int_rn(fmaf(cn, cn, -sn * sn) * kFixStepF);
        acc.s2 += __float2int_rn(2.0f * cn * sn * kFixStepF);
        acc.n += nb;
        if (S.nbr_out && id < (unsigned long long)S.n) S.nbr_out[id] = nb;
    }
    warp_insert(S, nxt, act, dtile, region, rec, to.cnt(S, nxt), to.spill(S, nxt));
}

// Warp sum of v, exact for |v| < 2^42 (32 high parts below 2^26 fit a signed
// word): two 32-bit warp reductions of its low 16 and its high bits instead of
// five rounds of 64-bit shuffles.  Of a step's sums a lane holds at most 256
// particles of 2^30 each.
__device__ __forceinline__ long long warp_redux_ll(long long v)
{
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)v & 0xffffu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(v >> 16));
    return (long long)hi * 65536 + (long long)lo;
}

// A warp's integer sums of one system (exact, so order-free) into that
// system's step accumulators.
template <bool REDUX>
__device__ __forceinline__ void flush_acc(const Acc &acc, unsigned long long *sys_acc, int cur)
{
    const long long a[5] = {acc.c, acc.s, acc.n, acc.c2, acc.s2};
    const int lane = threadIdx.x & 31;
    unsigned long long *slot =
        sys_acc + ((size_t)cur * kAccSlots + ((blockIdx.x * 32 + (threadIdx.x >> 5)) & (kAccSlots - 1))) * kAccWords;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const long long v = REDUX ? warp_redux_ll(a[k]) : warp_sum_ll(a[k]);
        if (lane == 0 && v) atomicAdd(slot + k, (unsigned long long)v);
    }
}

// Close step `step` of one system (one warp): p(t + 1) and q(t + 1) from the
// step's integer sums (its 64 accumulator slots loaded at once past the L1,
// then cleared), the trace and the on-the-fly measurement (Sec. 3.4).
__device__ __forceinline__ void close_sums(const Sys &S, long long step, int lane)
{
    static_assert(kAccSlots == 64, "two accumulator slots per lane");
    const int cur = (int)(step & 1);
    unsigned long long *a = S.acc + (size_t)cur * kAccSlots * kAccWords;
    // everything read up front: loads that stand behind a store wait for it in
    // turn (the 13 measurement sums one after another took most of this)
    double *const last = S.last, *const stats = S.stats, *const trace = S.trace, *const trace_nbar = S.trace_nbar;
    const bool measure = step < S.meas_until;
    const long long i1 = step + 1 - S.trace_base, cap = trace ? S.trace_cap : 0;
    const double n = (double)S.n;
    const double p0 = last[0], q0 = last[1];
    double st = measure && lane < 13 ? stats[lane] : 0.0;      // lane k: sum k
    unsigned long long x0[5], x1[5];
#pragma unroll
    for (int w = 0; w < 5; ++w) {
        x0[w] = __ldcg(a + lane * kAccWords + w);
        x1[w] = __ldcg(a + (lane + 32) * kAccWords + w);
    }
    __syncwarp();
#pragma unroll
    for (int w = 0; w < 5; ++w) {
        a[lane * kAccWords + w] = 0;
        a[(lane + 32) * kAccWords + w] = 0;
    }
    long long v[5];
#pragma unroll
    for (int w = 0; w < 5; ++w) v[w] = __shfl_sync(0xffffffffu, warp_sum_ll((long long)(x0[w] + x1[w])), 0);   // exact
    const double dc = (double)v[0] / kFixStep, ds = (double)v[1] / kFixStep;
    const double dc2 = (double)v[3] / kFixStep, ds2 = (double)v[4] / kFixStep;
    const double phi = n > 0 ? sqrt(dc * dc + ds * ds) / n : 0.0;
    const double q = n > 0 ? sqrt(dc2 * dc2 + ds2 * ds2) / n : 0.0;
    const double nbar = n > 0 ? (double)v[2] / n : 0.0;
    if (measure) {
        // on-the-fly measurement (Sec. 3.4): state t contributes the powers of
        // p(t), q(t) and of the mean neighbour number measured on it
        // (the last product, of the fourth moment, is added without rounding it)
        const double b = lane < 4 ? p0 : (lane < 8 ? q0 : nbar);
        const int m = lane & 3;
        double pk = b;
        for (int k = 0; k < min(m, 2); ++k) pk = __dmul_rn(pk, b);
        st = lane == 12 ? st + 1.0 : (m == 3 ? __fma_rn(pk, b, st) : __dadd_rn(st, pk));
        if (lane < 13) stats[lane] = st;
    }
    __syncwarp();
    if (lane == 0) {
        if (i1 >= 0 && i1 < cap) trace[i1] = phi;
        if (i1 >= 1 && i1 <= cap) trace_nbar[i1 - 1] = nbar;
        last[0] = phi;
        last[1] = q;
        last[2] = nbar;
        last[3] = (double)(step + 1);
    }
}

}  // namespace aapk
