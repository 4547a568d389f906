// aap_multi.cu -- many time steps of one small system in one launch (sm_103a).
//
// A system of a few hundred tiles leaves most of the chip idle whatever its
// kernels do: a step is then a chain of launches and dependent loads, not
// work.  Here every tile has a block of its own, all blocks are resident at
// once (a cooperative launch), and the blocks run up to a few dozen steps
// with one grid barrier each.  A block keeps its tile's geometry, its 25
// source segments and the system's parameters in shared memory over the
// steps, so what is left of a step is: the segments' record counts (one
// load), the records (one load), the counting sort by half cell and the
// update in shared memory (the arithmetic of the pipelined step, so the
// trajectories are equal bit for bit), the scatter into the next step's
// regions (one returning atomic), and the barrier.
//
// Bound: latency, about 15,000 cycles a step of which the barrier takes
// 3,700 (its fence, the arrivals and the polls are L2 round trips), the scatter
// and its returning atomics 4,300, the counts and records 3,700.  p(t) of 200
// steps at N = 1000: 4403 -> 1671 us (21.0 -> 7.9 us per step); 40 measured
// steps at N = 8192: 1245 -> 545 us.
//
// Buffers between the steps of a launch: records alternate between the two
// region buffers as always.  The region counters of the steps inside a launch
// rotate over three private sets: step i reads set (i - 1) % 3, fills set
// i % 3 and clears set (i - 2) % 3, which every block finished reading before
// the last barrier; so one barrier per step orders everything.  The first
// step reads the system's own counters and the last one fills them, so that
// between launches the state looks as any other step kernel leaves it.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "aap_device.cuh"
#include "aap_internal.cuh"
#include "aap_kernels.cuh"
#include "aap_tile.cuh"

namespace aapk {

namespace {

constexpr int kMultiWarps = 512 / 32;                   // of the widest block
constexpr long long kMultiWaitCycles = 4000000000ll;    // bound of a barrier wait, about 2 s at 2 GHz

// test hooks (aap_test_pipe_wait): the wait bound (<= 0: the default) and
// whether block 0 withholds its first arrival
__constant__ long long c_multi_wait_cycles;
__constant__ int c_multi_stall;

struct MultiShared {
    Sys S;
    OutMeta O;
    long long off[kSegs];       // first record of segment s in a region buffer
    int cidx[kSegs];            // its counter
    int cap[kSegs];
    int4 map[kSegs];            // as RawMeta::map of the pipelined step
    int segpre[kSegs + 1];
    int n_spill, own_spill, n_list;     // spill matches, those of the tile's own regions, those listed
    int slice;                  // scratch slice held, -1: none came free
    int warp_tot[kMultiWarps];
    int maxc;
    int ok;
    int load, staged;           // the tile's largest load and staged set over the launch's steps
};

// Staging arrays of one tile: shared memory, or the block's global scratch
// for a tile that outgrows it.
struct MultiStage {
    float4 *P;                  // records in half-cell order
    int4 *R;                    // staged records, mapped into the extended frame
    unsigned short *cellw, *slotw, *oq, *orr;
};

// The counters of a step's new records.
struct ToStep {
    int *c, *s;
    __device__ __forceinline__ int *cnt(const Sys &, int) const { return c; }
    __device__ __forceinline__ int *spill(const Sys &, int) const { return s; }
};

__device__ __forceinline__ MultiStage carve_multi(unsigned char *p, int cap)
{
    MultiStage A;
    A.P = (float4 *)p;
    p += (size_t)cap * 16;
    A.R = (int4 *)p;
    p += (size_t)cap * 16;
    A.cellw = (unsigned short *)p;
    p += (size_t)cap * 2;
    A.slotw = (unsigned short *)p;
    p += (size_t)cap * 2;
    A.oq = (unsigned short *)p;
    p += (size_t)cap * 2;
    A.orr = (unsigned short *)p;
    return A;
}

struct MultiTables {
    unsigned short *cst;        // [nceh + 1] half-cell starts
    int *hist;                  // [nceh]
    int *rowoff;                // own index = position in P + rowoff[ey]
    int *mhist;                 // measured theta / |Omega| counts of the launch
};

// Grid barrier: `target` arrivals in all.  Bounded; false when the bound ran
// out (ERR_TIMEOUT is set) or another block's did.
__device__ __forceinline__ bool multi_barrier(unsigned *bar, unsigned target, int *err, bool arrive, int *s_ok)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (arrive) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        const long long t0 = clock64();
        const long long bound = c_multi_wait_cycles > 0 ? c_multi_wait_cycles : kMultiWaitCycles;
        int ok = 1;
        for (;;) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (v >= target) break;
            if (clock64() - t0 > bound) {
                atomicOr(err, ERR_TIMEOUT);
                ok = 0;
                break;
            }
        }
        __threadfence();
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// A free scratch slice, taken until free_slice (one thread calls; the slices are
// fewer than the tiles of systems beyond some 300, and only dense tiles want one).  A
// block that holds one waits for no other block, so the wait ends; it is bounded
// all the same: -1 and ERR_TIMEOUT when the bound ran out.
__device__ __forceinline__ int take_slice(int *locks, int slices, int *err)
{
    const long long t0 = clock64();
    const long long bound = c_multi_wait_cycles > 0 ? c_multi_wait_cycles : kMultiWaitCycles;
    for (int i = blockIdx.x % slices;; i = i + 1 == slices ? 0 : i + 1) {
        if (atomicCAS(locks + i, 0, 1) == 0) {
            __threadfence();
            return i;
        }
        if (clock64() - t0 > bound) {
            atomicOr(err, ERR_TIMEOUT);
            return -1;
        }
    }
}

__device__ __forceinline__ void free_slice(int *locks, int i)
{
    __threadfence();
    atomicExch(locks + i, 0);
}

// List the spill matches of the block's tile (entry, segment) in the staging
// area's sorted records, which nothing uses before all records are mapped.
template <int NT>
__device__ __forceinline__ void list_spills(MultiShared &sh, const MultiStage &A, int cur, int nsp, int n)
{
    int *const spill_e = (int *)A.P;
    unsigned char *const spill_s = (unsigned char *)(spill_e + n);
    for (int e = threadIdx.x; e < nsp; e += NT) {
        const int key = __ldcg(sh.S.spill_key[cur] + e);
        for (int s = 0; s < kSegs; ++s)
            if (sh.cidx[s] == key) {
                const int j = atomicAdd(&sh.n_list, 1);
                if (j < n) {
                    spill_e[j] = e;
                    spill_s[j] = (unsigned char)s;
                }
            }
    }
    __syncthreads();
}

// One step of the block's tile, staged in A.  m records in all, of which
// m_seg from the segments and the rest from the spill matches; own of them
// are the tile's own by the counters.  true when the warp updated particles.
// A record's rank in its half cell takes all 16 bits of slotw (the global
// scratch stages up to 65,472 records, and nothing keeps them out of a single
// half cell), so the mirror flips are not stored beside it: a record in the
// halo beyond a reflecting wall is a mirror image, and no other record is.
template <int NT, int MODEL, bool SP>
__device__ __forceinline__ bool multi_tile(MultiShared &sh, const MultiStage &A, const MultiTables &tb, int m, int m_seg,
                                           int own, long long step, int *wc, int *ws, Acc &acc)
{
    const Sys &S = sh.S;
    const int *const spill_e = (const int *)A.P;                // list_spills
    const unsigned char *const spill_s = (const unsigned char *)(spill_e + (m - m_seg));
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cur = (int)(step & 1);
    const int tw = sh.O.tw, th = sh.O.th, W2 = sh.O.W2, H2 = th + 2, nce = W2 * H2;
    // --- records into the extended frame, histogram by half cell ----------
    for (int k = tid; k < m; k += NT) {
        int s = 0;
        int4 rr;
        if (k < m_seg) {
#pragma unroll
            for (int d = 16; d > 0; d >>= 1)        // the last segment starting at or before k
                if (s + d < kSegs && sh.segpre[s + d] <= k) s += d;
            rr = __ldcg(S.rec[cur] + sh.off[s] + (k - sh.segpre[s]));
        } else {
            s = spill_s[k - m_seg];
            rr = __ldcg(S.spill_rec[cur] + spill_e[k - m_seg]);
        }
        const int4 g = sh.map[s];
        const int mx = -(g.z & 1), my = -(g.w & 1);       // all ones where the axis is mirrored
        const int lx = rr.x >> (S.sx - 1), ly = rr.y >> S.sy;
        int ex = ((lx ^ mx) - mx) + (g.z >> 1), ey = ((ly ^ my) - my) + (g.w >> 1);
        if ((unsigned)ex >= (unsigned)W2 || (unsigned)ey >= (unsigned)H2) {
            atomicOr(S.err, ERR_BOUNDS);
            ex = min(max(ex, 0), W2 - 1);
            ey = min(max(ey, 0), H2 - 1);
        }
        const unsigned Xe = ((unsigned)rr.x ^ (unsigned)mx) - (unsigned)mx + (unsigned)g.x;
        const unsigned Ye = ((unsigned)rr.y ^ (unsigned)my) - (unsigned)my + (unsigned)g.y;
        A.R[k] = make_int4((int)Xe, (int)Ye, rr.z, rr.w);
        A.cellw[k] = (unsigned short)((ey << 8) | ex);
        A.slotw[k] = (unsigned short)atomicAdd(&tb.hist[ey * W2 + ex], 1);
    }
    __syncthreads();
    // --- prefix scan of the histogram (cleared for the next step) ----------
    {
        const int per = (nce + NT - 1) / NT;
        const int b0 = min(tid * per, nce), e0 = min(b0 + per, nce);
        int sum = 0, maxc = 0;
        for (int i = b0; i < e0; ++i) {
            const int h = tb.hist[i];
            sum += h;
            maxc = max(maxc, h);
        }
        const int incl = warp_incl_scan(sum);
        if (lane == 31) sh.warp_tot[warp] = incl;
        const int wmax = __reduce_max_sync(0xffffffffu, maxc);
        if (lane == 0) atomicMax(&sh.maxc, wmax);
        __syncthreads();
        int run = incl - sum;
        for (int w = 0; w < warp; ++w) run += sh.warp_tot[w];
        for (int i = b0; i < e0; ++i) {
            tb.cst[i] = (unsigned short)run;
            run += tb.hist[i];
            tb.hist[i] = 0;
        }
        if (tid == NT - 1) tb.cst[nce] = (unsigned short)run;
    }
    __syncthreads();
    // own rows: offsets, computed by every warp for itself (the same values)
    int n_own = 0;
    for (int r0 = 0; r0 < th; r0 += 32) {
        const int rw = r0 + lane;
        int len = 0, first = 0;
        if (rw < th) {
            first = tb.cst[(rw + 1) * W2 + 2];
            len = tb.cst[(rw + 1) * W2 + 2 * tw + 2] - first;
        }
        const int incl = warp_incl_scan(len);
        if (rw < th) tb.rowoff[rw + 1] = n_own + incl - len - first;
        n_own += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) {
        sh.O.o_first = 0;
        sh.O.n_own = n_own;
        sh.O.wide = 15 * sh.maxc >= 512;
        sh.O.dense = 2 * m > 3 * nce;
        if (n_own != own) atomicOr(S.err, ERR_BOUNDS);
    }
    __syncwarp();
    // --- records into half-cell order, own particles listed ----------------
    const int xc = tw << (S.sx - 1), yc = th << (S.sy - 1);
    // first and last column (row) that a mirror image cannot lie in
    const int mxl = S.bx && sh.O.tx == 0 ? 2 : 0, mxr = S.bx && sh.O.tx == S.ntx - 1 ? 2 * tw + 1 : W2;
    const int myl = S.by && sh.O.ty == 0 ? 1 : 0, myr = S.by && sh.O.ty == S.nty - 1 ? th : H2;
    for (int k = tid; k < m; k += NT) {
        const unsigned cf = A.cellw[k];
        const int ex = cf & 255, ey = cf >> 8;
        const int q = tb.cst[ey * W2 + ex] + A.slotw[k];
        const int4 rk = A.R[k];
        float thv = __int_as_float(rk.z);
        float sn, cs;
        if (MODEL == 1 && S.order != 1) {
            thv *= (float)S.order;
            sincosf(thv, &sn, &cs);
        } else {
            __sincosf(thv, &sn, &cs);       // |theta| <= pi: within 2^-21.4 absolute
        }
        if (ex < mxl || ex > mxr) {
            if (MODEL != 1 || (S.order & 1)) cs = -cs; else sn = -sn;
        }
        if (ey < myl || ey > myr) sn = -sn;
        float zc, zs;
        stage_angle<MODEL, SP>(S, rk.w, __float2int_rn(cs * kFixNbF), __float2int_rn(sn * kFixNbF), zc, zs);
        A.P[q] = make_float4((float)(rk.x - xc) * S.ux, (float)(rk.y - yc) * S.uy, zc, zs);
        if (ex >= 2 && ex < 2 * tw + 2 && ey >= 1 && ey <= th) {
            const int o = q + tb.rowoff[ey];
            A.oq[o] = (unsigned short)q;
            A.orr[o] = (unsigned short)k;
        }
    }
    __syncthreads();
    // --- interact, update, scatter ------------------------------------------
    // a tile of few particles gives each of them two or four lanes: its warps
    // are otherwise idle, and the candidate rows are the longest chain
    const bool measure = step < S.meas_until;
    const ToStep to = {wc, ws};
    const auto run = [&](auto lpp) {
        constexpr int LPP = decltype(lpp)::value;
        for (int o0 = warp * (32 / LPP); o0 < n_own; o0 += NT / LPP)
            update_one<MODEL, SP, LPP>(S, sh.O, A.P, tb.cst, A.R, A.orr, A.oq, o0 + lane / LPP, step, measure, tb.mhist,
                                       acc, to);
    };
    int lpp = 1;
    if (4 * n_own <= NT) {
        lpp = 4;
        run(std::integral_constant<int, 4>{});
    } else if (2 * n_own <= NT) {
        lpp = 2;
        run(std::integral_constant<int, 2>{});
    } else {
        run(std::integral_constant<int, 1>{});
    }
    if (tid == NT - 1) {
        sh.load = max(sh.load, tile_load(n_own, m, nce));
        sh.staged = max(sh.staged, m);
    }
    return warp * (32 / lpp) < n_own;
}

// One step of a tile that outgrows the block's shared memory, staged in a
// slice of the scratch: the block's own, or, of fewer slices than tiles, one
// taken for the step (several species: there is one for every tile).  false when
// none came free.
template <int NT, int MODEL, bool SP>
__device__ __forceinline__ bool multi_scratch(Acc &acc, bool &any, MultiShared &sh, const MultiTables &tb, int *locks,
                                              int slices, int tiles, unsigned char *scratch, size_t scratch_per_block,
                                              int scratch_cap, int m, int m_seg, int own, int nsp, long long step,
                                              int *wc, int *ws)
{
    const bool shared = !SP && slices < tiles;
    int sl = blockIdx.x;
    if (shared) {
        if (threadIdx.x == 0) sh.slice = take_slice(locks, slices, sh.S.err);
        __syncthreads();
        sl = sh.slice;
        if (sl < 0) return false;
    }
    const MultiStage Ag = carve_multi(scratch + scratch_per_block * sl, scratch_cap);
    if (m > m_seg) list_spills<NT>(sh, Ag, (int)(step & 1), nsp, m - m_seg);
    any = multi_tile<NT, MODEL, SP>(sh, Ag, tb, m, m_seg, own, step, wc, ws, acc);
    if (shared) {
        __syncthreads();
        if (threadIdx.x == 0) free_slice(locks, sl);
    }
    return true;
}

// The same out of line with its own sums, so that its registers do not weigh
// on the tiles in shared memory (N = 100,000: 13.5 -> 13.2 us per step; coupled species,
// whose sums need the most registers, lose 6% by the call and inline it).
template <int NT, int MODEL, bool SP>
__device__ __noinline__ bool multi_scratch_call(MultiShared &sh, const MultiTables &tb, int *locks, int slices, int tiles,
                                                unsigned char *scratch, size_t scratch_per_block, int scratch_cap, int m,
                                                int m_seg, int own, int nsp, long long step, int *wc, int *ws)
{
    Acc acc = {0, 0, 0, 0, 0};
    bool any = false;
    const bool ok = multi_scratch<NT, MODEL, SP>(acc, any, sh, tb, locks, slices, tiles, scratch, scratch_per_block,
                                                 scratch_cap, m, m_seg, own, nsp, step, wc, ws);
    if (any) flush_acc<true>(acc, sh.S.acc, (int)(step & 1));
    return ok;
}

// nsteps steps of the system from its current step; block b does tile b, and
// one more block closes the steps (p(t), the trace, the measured moments: a
// chain of FP64 operations that would hold up every tile's block).
// bar[0]: barrier arrivals, bar[1]: blocks that have left (both 0 between
// launches), bar[4 + i]: whether scratch slice i is taken.  cnt3: three counter
// sets of `stride` ints, zero between launches.
template <int NT, int BPS, int MODEL, bool SP>
__global__ void __launch_bounds__(NT, BPS)
k_multi(Sys *__restrict__ sys, Ctl *ctl, int nsteps, int cap, int nceh, int hist_words, int *cnt3, int stride,
        unsigned *bar, unsigned char *scratch, size_t scratch_per_block, int scratch_cap, int spill_list_cap, int slices)
{
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ MultiShared sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blockIdx.x, nblk = gridDim.x;
    MultiTables tb;
    {
        unsigned char *p = smem + (size_t)cap * 40;
        tb.hist = (int *)p;
        p += (size_t)round_up(nceh, 4) * 4;
        tb.rowoff = (int *)p;
        p += (size_t)(kMaxTile + 4) * 4;
        tb.mhist = (int *)p;
        p += (size_t)round_up(hist_words, 4) * 4;
        tb.cst = (unsigned short *)p;
    }
    const MultiStage As = carve_multi(smem, cap);
    {
        const int words = (int)(sizeof(Sys) / 4);
        const int *src = reinterpret_cast<const int *>(sys);
        int *dst = reinterpret_cast<int *>(&sh.S);
        for (int i = tid; i < words; i += NT) dst[i] = src[i];
    }
    for (int i = tid; i < nceh; i += NT) tb.hist[i] = 0;
    for (int i = tid; i < hist_words; i += NT) tb.mhist[i] = 0;
    const long long step0 = ctl->step;
    __syncthreads();
    const Sys &S = sh.S;
    // after a wait has run out the handle is unusable: later steps do nothing
    if (tid == 0) {
        sh.ok = (*((volatile int *)S.err) & ERR_TIMEOUT) == 0;
        sh.maxc = 0;
        sh.load = sh.staged = 0;
    }
    const bool closer = tile == nblk - 1;
    if (warp == 0 && !closer) {
        const TileGeo G = tile_geo(S, tile);
        if (lane < kSegs) {
            const Seg sg = make_seg(S, G, lane, 0);
            const int mxr = sg.ax < 0;
            sh.off[lane] = (long long)sg.tile * S.tile_slots + S.off[sg.region];
            sh.cidx[lane] = sg.tile * kCntStride + sg.region;
            sh.cap[lane] = S.cap[sg.region];
            sh.map[lane] = make_int4((int)(unsigned)(unsigned long long)sg.bx, (int)(unsigned)(unsigned long long)sg.by,
                                     2 * (2 * sg.cx + mxr + 2) + mxr, 2 * (sg.cy + 1) + (sg.ay < 0));
        }
        if (lane == 0) {
            OutMeta &O = sh.O;
            O.tile = tile;
            O.rbuf = O.rwide = 0;
            O.tx = G.tx; O.ty = G.ty; O.tw = G.tw; O.th = G.th; O.W2 = 2 * G.tw + 4;
            O.twL = G.twL; O.twR = G.twR; O.thD = G.thD; O.thU = G.thU;
        }
    }
    __syncthreads();
    if (!sh.ok) return;
    const int spw = stride - kCntStride;            // the spill counter of a private set
    unsigned arrived = 0;
    bool ok = true;
    for (int i = 0; i < nsteps; ++i) {
        const long long step = step0 + i;
        const int cur = (int)(step & 1);
        const int *rc = i == 0 ? S.cnt[cur] : cnt3 + (size_t)((i + 2) % 3) * stride;
        const int *rs = i == 0 ? &S.spill_cnt[cur] : rc + spw;
        int *wc = i == nsteps - 1 ? S.cnt[cur ^ 1] : cnt3 + (size_t)(i % 3) * stride;
        int *ws = i == nsteps - 1 ? &S.spill_cnt[cur ^ 1] : wc + spw;
        if (closer) {
            if (i == 0 && tid < 2) S.err[1 + tid] = 0;
            // the sums of the step before (complete since the last barrier),
            // and the spill count it consumed
            if (i >= 1 && warp == 0) {
                close_sums(S, step - 1, lane);
                if (lane == 0) *(i == 1 ? &S.spill_cnt[step0 & 1] : cnt3 + (size_t)((i + 1) % 3) * stride + spw) = 0;
            }
        } else {
            // counters consumed by the step before (every block is past reading them)
            if (i >= 1 && warp == NT / 32 - 1 && lane < kCntStride)
                (i == 1 ? S.cnt[step0 & 1] : cnt3 + (size_t)((i + 1) % 3) * stride)[tile * kCntStride + lane] = 0;
        }
        if (i == 1 && nsteps == 2) {
            // the last step of two fills the counters the first one read:
            // they have to be clear first
            arrived += nblk;
            if (!(ok = multi_barrier(bar, arrived, S.err, true, &sh.ok))) break;
        }
        if (!closer) {
            // the segments' record counts and their prefix (every warp for
            // itself, the same values: no block barrier before the records)
            if (tid == 0) {
                sh.maxc = 0;
                sh.n_spill = sh.own_spill = sh.n_list = 0;
            }
            const int c = lane < kSegs ? min(__ldcg(rc + sh.cidx[lane]), sh.cap[lane])
                                       : (lane == 31 ? min(__ldcg(rs), S.spill_cap) : 0);
            const int incl = warp_incl_scan(lane < kSegs ? c : 0);
            if (lane <= kSegs) sh.segpre[lane] = lane < kSegs ? incl - c : incl;
            const int m_seg = __shfl_sync(0xffffffffu, incl, kSegs - 1), nsp = __shfl_sync(0xffffffffu, c, 31);
            __syncwarp();
            int m = m_seg, own = sh.segpre[kRegions];
            if (nsp > 0) {
                // records parked in the spill list for one of the segments
                __syncthreads();
                for (int e = tid; e < nsp; e += NT) {
                    const int key = __ldcg(S.spill_key[cur] + e);
                    for (int s = 0; s < kSegs; ++s)
                        if (sh.cidx[s] == key) {
                            atomicAdd(&sh.n_spill, 1);
                            if (s < kRegions) atomicAdd(&sh.own_spill, 1);
                        }
                }
                __syncthreads();
                if (tid == 0 && sh.n_spill > spill_list_cap) atomicOr(S.err, ERR_STAGE);
                m += min(sh.n_spill, spill_list_cap);
                own += sh.own_spill;
            }
            Acc acc = {0, 0, 0, 0, 0};
            bool any = false;
            if (m <= cap) {
                if (m > m_seg) list_spills<NT>(sh, As, cur, nsp, m - m_seg);
                any = multi_tile<NT, MODEL, SP>(sh, As, tb, m, m_seg, own, step, wc, ws, acc);
            } else if (m <= scratch_cap) {
                int *const locks = (int *)(bar + 4);
                if constexpr (SP && MODEL == 1)
                    ok = multi_scratch<NT, MODEL, SP>(acc, any, sh, tb, locks, slices, nblk - 1, scratch, scratch_per_block,
                                                      scratch_cap, m, m_seg, own, nsp, step, wc, ws);
                else
                    ok = multi_scratch_call<NT, MODEL, SP>(sh, tb, locks, slices, nblk - 1, scratch, scratch_per_block,
                                                           scratch_cap, m, m_seg, own, nsp, step, wc, ws);
                if (!ok) break;
            } else if (tid == 0) {
                atomicOr(S.err, ERR_STAGE | ERR_LOST);
            }
            if (any) flush_acc<true>(acc, S.acc, cur);
        }
        arrived += nblk;
        if (!(ok = multi_barrier(bar, arrived, S.err, !(c_multi_stall && i == 0 && tile == 0), &sh.ok))) break;
    }
    if (!ok) return;
    // --- the state as every step kernel leaves it ----------------------------
    const long long last = step0 + nsteps - 1;
    if (closer) {
        if (warp == 0) {
            close_sums(S, last, lane);
            if (lane == 0) {
                *(nsteps == 1 ? &S.spill_cnt[step0 & 1] : cnt3 + (size_t)((nsteps + 1) % 3) * stride + spw) = 0;
                ctl->step = step0 + nsteps;
            }
        }
    } else {
        if (warp == 0 && lane < kCntStride)
            (nsteps == 1 ? S.cnt[step0 & 1] : cnt3 + (size_t)((nsteps + 1) % 3) * stride)[tile * kCntStride + lane] = 0;
        if (tid == NT - 1) {
            atomicMax(S.err + 1, sh.load);      // the closing block cleared them before the first barrier
            atomicMax(S.err + 2, sh.staged);
        }
        if ((tile & 31) == 0 && tid == 32) S.spill_bits[last & 1][tile >> 5] = 0u;
        if (step0 < S.meas_until)
            for (int i = tid; i < S.bins_theta + S.bins_nbr; i += NT)
                if (tb.mhist[i]) atomicAdd(S.hist + i, (unsigned long long)tb.mhist[i]);
    }
    if (tid == 0 && atomicAdd(bar + 1, 1u) == (unsigned)nblk - 1) {
        bar[0] = 0;         // every block is past its last wait
        bar[1] = 0;
    }
}

size_t multi_smem(int cap, int nceh, int hist_words)
{
    return (size_t)cap * 40 + (size_t)round_up(nceh, 4) * 4 + (size_t)(kMaxTile + 4) * 4 +
           (size_t)round_up(hist_words, 4) * 4 + (size_t)round_up(nceh + 1, 8) * 2;
}

typedef void (*MultiKernel)(Sys *, Ctl *, int, int, int, int, int *, int, unsigned *, unsigned char *, size_t, int, int,
                            int);

template <int NT, int BPS>
MultiKernel multi_kernel_t(int model, bool species)
{
    switch (model) {
    case 0: return species ? k_multi<NT, BPS, 0, true> : k_multi<NT, BPS, 0, false>;
    case 1: return species ? k_multi<NT, BPS, 1, true> : k_multi<NT, BPS, 1, false>;
    case 2: return species ? k_multi<NT, BPS, 2, true> : k_multi<NT, BPS, 2, false>;
    default: return nullptr;
    }
}

MultiKernel multi_kernel(int model, bool species, int threads)
{
    return threads == 512 ? multi_kernel_t<512, 1>(model, species) : multi_kernel_t<256, 4>(model, species);
}

}  // namespace

cudaError_t set_multi_test(long long wait_cycles, int stall)
{
    cudaError_t e = cudaMemcpyToSymbol(c_multi_wait_cycles, &wait_cycles, sizeof(wait_cycles));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(c_multi_stall, &stall, sizeof(stall));
}

cudaError_t configure_multi(LaunchCfg &L, bool species, int ntiles, int sm_count, int min_cap)
{
    L.multi = 0;
    // One block of 512 threads (128 registers each) per SM while that holds every
    // tile, else up to four blocks of 256 threads (N = 50,021 in 400 tiles,
    // uniform: 46 us per step in single launches, 13 us so; the caller goes back
    // to single steps while some tile is dense).
    const int blocks = ntiles + 1;
    const int threads = blocks <= sm_count ? 512 : 256;
    if (ntiles < 1 || blocks > 4 * sm_count) return cudaSuccess;
    int dev = 0, coop = 0, optin = 0, per_sm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess) return e;
    if (!coop) return cudaSuccess;
    const MultiKernel k = multi_kernel(L.model, species, threads);
    if (!k) return cudaErrorInvalidValue;
    // the kernel's static shared memory, looked up once per kernel (a handle is
    // laid out several times while it is made)
    static std::atomic<int> stat[2][3][2];
    std::atomic<int> &st = stat[threads == 512][L.model][species];
    if (st.load() == 0) {
        cudaFuncAttributes a;
        if ((e = cudaFuncGetAttributes(&a, k)) != cudaSuccess) return e;
        st.store((int)a.sharedSizeBytes + 1);
    }
    // every block resident at once: as much staging as that leaves each
    const int bps = (blocks + sm_count - 1) / sm_count;
    const long long room = std::min<long long>(optin, per_sm / bps - 1024) - (st.load() - 1);
    int cap = 4096;
    while (cap >= min_cap && (long long)multi_smem(cap, L.pipe_nceh, L.hist_words) > room) cap -= 32;
    if (cap < min_cap) return cudaSuccess;
    const int smem = (int)multi_smem(cap, L.pipe_nceh, L.hist_words);
    // the limit belongs to the kernel, not to a handle: keep the largest any
    // handle of this process asked for
    static std::atomic<int> limit{0};
    int prev = limit.load();
    while (smem > prev && !limit.compare_exchange_weak(prev, smem)) {
    }
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, std::max(smem, limit.load()));
    if (e != cudaSuccess) return e;
    // bps blocks fit an SM: their registers by the launch bounds, their shared
    // memory by `room` (the cooperative launch itself checks)
    L.multi = 1;
    L.multi_species = species ? 1 : 0;
    L.multi_cap = cap;
    L.multi_threads = threads;
    L.multi_tiles = ntiles;
    return cudaSuccess;
}

cudaError_t launch_multi(const LaunchCfg &L, int nsteps, cudaStream_t st)
{
    const MultiKernel k = multi_kernel(L.model, L.multi_species != 0, L.multi_threads);
    Sys *sys = L.sys;
    Ctl *ctl = L.ctl;
    int cap = L.multi_cap, nceh = L.pipe_nceh, hw = L.hist_words, stride = multi_stride(L.multi_tiles);
    int *cnt3 = L.multi_cnt;
    unsigned *bar = reinterpret_cast<unsigned *>(L.multi_cnt + 3 * (size_t)stride);
    unsigned char *scratch = L.scratch;
    size_t spb = L.scratch_per_block;
    int scap = L.scratch_cap, slc = L.spill_list_cap, slices = L.multi_slices;
    void *args[] = {&sys, &ctl, &nsteps, &cap, &nceh, &hw, &cnt3, &stride, &bar, &scratch, &spb, &scap, &slc, &slices};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k), dim3(L.multi_tiles + 1), dim3(L.multi_threads), args,
                                       multi_smem(cap, nceh, hw), st);
}

}  // namespace aapk
