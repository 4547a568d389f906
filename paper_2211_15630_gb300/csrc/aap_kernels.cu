// aap_kernels.cu -- sm_103a kernels of the aligning-active-particles step.
//
// One time step (Sec. 2 of Kuersten, "Aligning Active Particles Py Package"):
//   k_step     per tile: stage the tile and its one-cell halo (cell lists,
//              Sec. 3.2, with periodic or mirror images, Sec. 2.4), counting
//              sort by cell in shared memory (block histogram + block prefix
//              scan; arrival order inside a cell), sum over the 3x3 cells
//              (Eq. collision_VM / collision_NVM or the Langevin sum of
//              Eq. Langevin_dynamics) in exact integers, so that the result
//              does not depend on that arrival order, draw Philox
//              noise, stream (Eq. streaming or Euler-Maruyama), apply the
//              boundary rule, and scatter the new record into the region of
//              its new cell through a warp-aggregated atomic counter.  Also
//              accumulates p = |sum e^{i theta}| / N (Sec. 3.4) in exact
//              64-bit integers.
//              Tiles whose staged set does not fit shared memory are staged
//              in the block's slice of global scratch by the same code.
//   k_finish   turns the step's integer sums into p(t), clears the counters
//              of the buffer just consumed and advances the step counter.
#include <algorithm>

#include <atomic>
#include <cuda_runtime.h>

#include "aap_device.cuh"
#include "aap_internal.cuh"
#include "aap_kernels.cuh"
#include "aap_tile.cuh"

namespace aapk {

// Persistent blocks pull tiles in raster order (so halos are L2-hot) from a
// device counter; the next tile index is fetched while the current one runs.
// A tile whose staged set exceeds the shared-memory capacity is staged in the
// block's slice of global scratch instead.  All systems of one launch share
// the model.
template <int NT, int MODEL>
__global__ void __launch_bounds__(NT, NT >= 512 ? 2 : 3)
k_step(const Sys *__restrict__ sys, int nsys, const int *__restrict__ tile_base, Ctl *ctl,
       int stage_cap, int nce_max, unsigned char *scratch, size_t scratch_per_block, int scratch_cap,
       int spill_list_cap)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ TileCtx T;
    pdl_wait();
    pdl_next();
    const long long step = ctl->step;
    const int cur = (int)(step & 1);
    const int total = tile_base[nsys];
    Stage As;
    carve_stage(As, smem, stage_cap);
    Tables tb;
    carve_tables(tb, smem + stage_bytes(stage_cap), nce_max);
    unsigned char *mine = scratch + scratch_per_block * blockIdx.x;
    Stage Ag;
    carve_stage(Ag, mine, scratch_cap);
    int *spill_e = (int *)(mine + stage_bytes(scratch_cap));
    unsigned char *spill_s = (unsigned char *)(spill_e + spill_list_cap);
    if (threadIdx.x == 0) {
        T.sysi = -1;
        T.pf_tile = -1;
        T.part = 0;
        T.parts = 1;
        T.total = total;
        T.nsys = nsys;
        T.tile_base = tile_base;
        T.next = atomicAdd(&ctl->tile_next, 1);
    }
    __syncthreads();
    for (;;) {
        const int g = T.next;
        if (g >= total) break;
        const int si = nsys > 1 ? sys_of_tile(tile_base, nsys, g) : 0;
        if (si != T.sysi) {
            const int words = (int)(sizeof(Sys) / 4);
            const int *src = reinterpret_cast<const int *>(sys + si);
            int *dst = reinterpret_cast<int *>(&T.S);
            for (int i = threadIdx.x; i < words; i += NT) dst[i] = src[i];
        }
        __syncthreads();
        int next_g = 0;         // thread 0: the tile after this one (published in tile_body)
        if (threadIdx.x == 0) {
            T.sysi = si;
            T.tile = g - tile_base[si];
            next_g = atomicAdd(&ctl->tile_next, 1);
        }
        __syncthreads();
#ifdef AAP_PHASE_TIMING
        const long long ts0 = clock64();
#endif
        tile_setup<NT>(T, tb, cur, nce_max, spill_e, spill_s, spill_list_cap);
#ifdef AAP_PHASE_TIMING
        if (threadIdx.x == 0) {
            atomicAdd(&g_phase[6], (unsigned long long)(clock64() - ts0));
            atomicAdd(&g_phase[7], 1ull);
            atomicAdd(&g_phase[8], (unsigned long long)T.m);
            atomicAdd(&g_phase[9], (unsigned long long)(T.m > stage_cap));
        }
#endif
#ifdef AAP_PHASE_TIMING
        const long long tb0 = clock64();
#endif
        if (T.m <= stage_cap) {
            tile_body<NT, MODEL>(T, As, tb, step, spill_e, spill_s, next_g);
        } else if (T.m <= scratch_cap) {
            // a dense tile: staged in global scratch, except the records the
            // candidate loops read, which still fit the shared staging area
            Stage Ah = Ag;
            if ((size_t)T.m * sizeof(float4) <= stage_bytes(stage_cap)) Ah.P = reinterpret_cast<float4 *>(smem);
            tile_body<NT, MODEL>(T, Ah, tb, step, spill_e, spill_s, next_g);
        } else if (threadIdx.x == 0) {
            atomicOr(T.S.err, ERR_STAGE | ERR_LOST);
            T.next = next_g;
        }
#ifdef AAP_PHASE_TIMING
        if (threadIdx.x == 0)
            atomicAdd(&g_phase[T.m <= stage_cap ? 10 : 11], (unsigned long long)(clock64() - tb0));
#endif
        __syncthreads();
    }
}

// Close the step: p(t+1) from the integer sums, clear the consumed buffer's
// counters, advance the step.  Every thread clears counter words of the flat
// range over all systems' tiles; the warps of all blocks take one system each
// for the sums (its 64 accumulator slots loaded at once, then cleared); the
// last block to arrive advances the step.
__global__ void __launch_bounds__(1024) k_finish(Sys *sys, int nsys, const int *__restrict__ tile_base, Ctl *ctl)
{
    __shared__ int s_last;
    pdl_wait();
    pdl_next();
    const long long step = ctl->step;
    const int cur = (int)(step & 1);
    const long long gt = blockIdx.x * (long long)blockDim.x + threadIdx.x, gs = (long long)gridDim.x * blockDim.x;
    if (nsys == 1) {
        // one system: its counter lines are one array (16-byte aligned, 64
        // bytes a tile), cleared by 16-byte stores through pointers read once
        int4 *c4 = reinterpret_cast<int4 *>(sys[0].cnt[cur]);
        unsigned *sb = sys[0].spill_bits[cur];
        const int nt = tile_base[1];
        const long long n4 = (long long)nt * (kCntStride / 4);
        for (long long i = gt; i < n4; i += gs) c4[i] = make_int4(0, 0, 0, 0);
        for (long long i = gt; i < (nt + 31) / 32; i += gs) sb[i] = 0u;    // the tiles' spill marks
    } else {
        const long long nw = (long long)tile_base[nsys] * (kCntStride / 4);     // 16-byte words
        for (long long i = gt; i < nw; i += gs) {
            const int g = (int)(i / (kCntStride / 4)), w = (int)(i % (kCntStride / 4));
            const int si = sys_of_tile(tile_base, nsys, g);
            const int t = g - tile_base[si];
            reinterpret_cast<int4 *>(sys[si].cnt[cur])[(long long)t * (kCntStride / 4) + w] = make_int4(0, 0, 0, 0);
            if (w == 0 && (t & 31) == 0) sys[si].spill_bits[cur][t >> 5] = 0u;    // the tiles' spill marks
        }
    }
    const int lane = threadIdx.x & 31;
    const int gw = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nwarps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int si = gw; si < nsys; si += nwarps) {
        Sys &S = sys[si];
        close_sums(S, step, lane);
        if (lane == 0) S.spill_cnt[cur] = 0;
    }
    // the step advances when every block is done with it (a single block: at
    // once, without the fence and the ticket's round trip)
    if (threadIdx.x == 0) s_last = 1;
    __syncthreads();
    if (gridDim.x > 1) {
        if (threadIdx.x == 0) {
            __threadfence();
            s_last = (atomicAdd(&ctl->finish_ticket, 1) == (int)gridDim.x - 1);
        }
        __syncthreads();
    }
    if (s_last && threadIdx.x == 0) {
        ctl->tile_next = 0;
        ctl->finish_ticket = 0;
        ctl->dense_count = 0;
        ctl->dense_next = 0;
        ctl->step = step + 1;
    }
}

// ------------------------------------------------------- order of the tiles --
// The order in which the pipelined step claims its work: a step ends when its
// longest job does, so the longest start first, and a tile that would keep its
// SM longer than some 60% of what an SM has to do on average is split into up to
// eight parts, each of which stages and sorts the whole tile and updates its
// share of the particles (a clustered state of N = 524,288: its densest tile
// has three times the pairs of an average SM).  One block sorts the jobs of
// all systems by the class of their cost (two classes per factor of two),
// stable inside a class, so that neighbours stay together.  Only for systems of
// few tiles per SM (pipe_few): with many, dense tiles one after another leave
// the pipeline's roles waiting for each other where light ones between them
// fill the gaps (N = 2^24, clustered: 0.83 -> 0.86 ms per step).  Run every few
// dozen steps: loads change slowly.  An even state gets a list in raster order, and
// the finding that the order does not matter: the host then launches the variant
// without the list (kernel k_step_pipe).  A state is even while no tile leads or is
// split and the longest is not longer than the mean by more than a share (even_share) of
// what an SM has to do.  The list then gains about 0.3 of that excess, and its variant costs
// VM some 5%, Langevin 2%, NVM nothing: with the list against raster order, us per step, VM
// uniform 76.2 / 73.0 (excess 0.06), 49.1 / 51.1 (0.36), flocks 80.2 / 86.8 (0.31), at low
// density 54.1 / 51.6 (0.14), 54.1 / 53.6 (0.45); Langevin uniform 62.9 / 61.7 (0.03), 64.9 / 67.4
// (0.06, walls), 54.0 / 53.5 (0.06), 70.1 / 78.6 (0.17, walls); NVM uniform 92.4 / 92.1
// (0.02), 47.3 / 47.9 (0.14).
// jobs: [total + kMaxParts] {tile, part | parts << 8}; cost: [total] scratch;
// meta: the number of leading jobs that whole blocks do first (tiles of more
// own particles than own_max, two buffers of the pipeline), of all jobs, and the
// finding (a single system's goes to its fourth error word too).
__device__ __forceinline__ float even_share(int model) { return model == 0 ? 0.15f : model == 1 ? 0.05f : 0.0f; }
constexpr float kSplitAbove = 0.6f, kSplitTo = 2.0f;       // of an SM's average: split tiles above, into parts of 1 / kSplitTo
__global__ void __launch_bounds__(1024) k_tile_order(const Sys *__restrict__ sys, int nsys,
                                                     const int *__restrict__ tile_base, const Ctl *__restrict__ ctl,
                                                     int own_max, int blocks, int2 *jobs, float *cost, int *meta)
{
    constexpr int kClasses = 17;                // 0: whole blocks first
    __shared__ float s_sum[32], s_max[32];
    __shared__ int s_cnt[kClasses], s_warp[32][kClasses], s_extra, s_kmax, s_lead;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int b = (int)(ctl->step & 1), total = tile_base[nsys];
    float sum = 0.f, top = 0.f;
    for (int g = tid; g < total; g += 1024) {
        const int si = nsys > 1 ? sys_of_tile(tile_base, nsys, g) : 0;
        const Sys &S = sys[si];
        const int *c = S.cnt[b] + (size_t)(g - tile_base[si]) * kCntStride;
        int own = 0;
#pragma unroll
        for (int r = 0; r < kRegions; ++r) own += c[r];
        // staging and update per particle, and the candidates of 15 half
        // cells; negative: a tile for whole blocks
        const float f = (float)own * (24.0f + 7.5f * (float)own / (float)(S.twmax * S.thmax));
        cost[g] = own > own_max ? -f : f;
        sum += f;
        top = fmaxf(top, f);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    }
    if (lane == 0) {
        s_sum[warp] = sum;
        s_max[warp] = top;
    }
    if (tid < kClasses) s_cnt[tid] = 0;
    if (tid == 0) {
        s_extra = s_lead = 0;
        s_kmax = 1;
    }
    __syncthreads();
    float all = 0.f, longest = 0.f;
    for (int w = 0; w < 32; ++w) {
        all += s_sum[w];
        longest = fmaxf(longest, s_max[w]);
    }
    const float mean = fmaxf(all / (float)max(total, 1), 1e-20f), share = fmaxf(all / (float)blocks, 1e-20f);
    const auto cls = [&](float f, int K) {
        if (f < 0.f) return 0;
        return 1 + min(max((int)floorf(8.0f - 2.0f * __log2f(fmaxf(f, 1e-20f) / ((float)K * mean))), 0), kClasses - 2);
    };
    const auto parts = [&](float f) {
        return fabsf(f) > kSplitAbove * share && fabsf(f) > 1.5f * mean ? min((int)ceilf(kSplitTo * fabsf(f) / share), 8) : 1;
    };
    for (int g = tid; g < total; g += 1024) {
        const int K = parts(cost[g]);
        if (K > 1) {
            atomicAdd(&s_extra, K - 1);
            atomicMax(&s_kmax, K);
        }
        if (cost[g] < 0.f) s_lead = 1;
    }
    __syncthreads();
    const bool dense = s_extra > 0 || s_lead || longest - mean > even_share(sys[0].model) * share;
    if (nsys == 1 && tid == 0) sys[0].err[3] = dense;
    if (!dense) {
        for (int g = tid; g < total; g += 1024) jobs[g] = make_int2(g, 1 << 8);
        if (tid < 3) meta[tid] = tid == 1 ? total : 0;
        return;
    }
    const bool split = s_extra <= kMaxParts;
    const int kmax = split ? s_kmax : 1;
    for (int g = tid; g < total; g += 1024) {
        const int K = split ? parts(cost[g]) : 1;
        atomicAdd(&s_cnt[cls(cost[g], K)], K);
    }
    __syncthreads();
    if (tid == 0) {
        int run = 0;
        meta[0] = s_cnt[0];
        for (int k = 0; k < kClasses; ++k) {
            const int n = s_cnt[k];
            s_cnt[k] = run;
            run += n;
        }
        meta[1] = run;
        meta[2] = 1;
    }
    __syncthreads();
    for (int g0 = 0; g0 < total; g0 += 1024) {
        const int g = g0 + tid;
        const float f = g < total ? cost[g] : 0.f;
        const int K = g < total ? (split ? parts(f) : 1) : 0;
        for (int p = 0; p < kmax; ++p) {
            const int k = p < K ? cls(f, K) : -1;
            const unsigned peers = __match_any_sync(0xffffffffu, k);
            if (lane < kClasses) s_warp[warp][lane] = 0;
            __syncwarp();
            if (k >= 0 && lane == __ffs(peers) - 1) s_warp[warp][k] = __popc(peers);
            __syncthreads();
            if (tid < kClasses) {
                int run = s_cnt[tid];
                for (int w = 0; w < 32; ++w) {
                    const int n = s_warp[w][tid];
                    s_warp[w][tid] = run;
                    run += n;
                }
                s_cnt[tid] = run;
            }
            __syncthreads();
            if (k >= 0) jobs[s_warp[warp][k] + __popc(peers & ((1u << lane) - 1u))] = make_int2(g, p | (K << 8));
            __syncthreads();
        }
    }
}

// ------------------------------------------------- state in and out --------
// llrint(p / cs * scale), scale a power of two, without the FP64 division (the
// FP64 pipe is narrow on this GPU; two divisions a particle took most of the
// insert: N = 2^24, 854 us).  p r, r = 1 / cs rounded, is within 2^-51 relative
// of the rounded quotient, so the two round to the same integer unless p r
// scale lies that close to a half-integer: then the division decides (for
// fewer than one particle in a thousand, out of line).
__device__ __noinline__ long long grid_round_div(double p, double cs, double scale) { return llrint(p / cs * scale); }

__device__ __forceinline__ long long grid_round(double p, double cs, double r, double scale)
{
    const double v = p * r * scale;
    const double i = rint(v);
    if (!(fabs(v - i) < 0.5 - fabs(v) * 1e-15)) return grid_round_div(p, cs, scale);
    return (long long)i;
}

// Place one particle given in box coordinates into buffer b (exact rounding
// of the position to the fixed-point grid).  mode 0: from arrays; mode 1: draw
// the uniform isotropic initial state from Philox, tag 1.
__global__ void k_insert(Sys S, int b, const double *x, const double *y, const float *th, int mode, double rx, double ry)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const bool act = i < S.n;
    int dtile = 0, region = 0;
    int4 rec = make_int4(0, 0, 0, 0);
    if (act) {
        double px, py;
        float pt;
        if (mode == 1) {
            uint32_t c4[4] = {(uint32_t)i, 0u, 0u, 1u};
            philox4x32_10(c4, S.seed_lo, S.seed_hi);
            px = S.lx * u01d(c4[0]);
            py = S.ly * u01d(c4[1]);
            pt = (float)(3.14159265358979323846 * (2.0 * u01d(c4[2]) - 1.0));
        } else {
            px = x[i];
            py = y[i];
            pt = th[i];
        }
        long long gx = grid_round(px, S.csx_d, rx, (double)(1ll << S.sx));
        long long gy = grid_round(py, S.csy_d, ry, (double)(1ll << S.sy));
        const long long wx = (long long)S.ncx << S.sx, wy = (long long)S.ncy << S.sy;
        if (gx >= wx) gx = S.bx ? wx - 1 : gx - wx;
        if (gx < 0) gx = S.bx ? 0 : gx + wx;
        if (gy >= wy) gy = S.by ? wy - 1 : gy - wy;
        if (gy < 0) gy = S.by ? 0 : gy + wy;
        const int cx = (int)(gx >> S.sx), cy = (int)(gy >> S.sy);
        const int tx = tile_of_x(S, cx), ty = tile_of_y(S, cy);
        const int x0 = tile_x0(S, tx), y0 = tile_y0(S, ty);
        const int X = (int)(gx - ((long long)x0 << S.sx)), Y = (int)(gy - ((long long)y0 << S.sy));
        const int tw = tile_x0(S, tx + 1) - x0, th_ = tile_y0(S, ty + 1) - y0;
        if (pt >= AAP_PI_F || pt < -AAP_PI_F) pt -= AAP_2PI_F * floorf((pt + AAP_PI_F) * (1.0f / AAP_2PI_F));
        dtile = ty * S.ntx + tx;
        region = S.flat ? 0 : region_of(X >> S.sx, Y >> S.sy, tw, th_);
        rec = make_int4(X, Y, __float_as_int(pt), (int)i);
    }
    warp_insert(S, b, act, dtile, region, rec);
}

// The lowest index whose position lies outside [0, lx] x [0, ly] (bad[0])
// and whose orientation is not finite (bad[1]); both start at all ones.
__global__ void k_validate_state(const double *x, const double *y, const float *th, long long n, double lx,
                                 double ly, unsigned long long *bad)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        if (!(x[i] >= 0.0 && x[i] <= lx) || !(y[i] >= 0.0 && y[i] <= ly)) atomicMin(bad, (unsigned long long)i);
        if (!isfinite(th[i])) atomicMin(bad + 1, (unsigned long long)i);
    }
}

// Warp `w` of `nw` visits its share of the stored records of buffer b (a warp
// or several a tile, only the valid slots of its nine regions taken as one index
// range; a flat system's single region in runs of 32 records), and of the
// spill list: f(record, tile column, tile row), some lanes idle.  (A thread per
// slot, empty ones included, with two divisions each to find its region, took
// 1671 us to gather N = 2^24 at the start's four-fold capacity.)
template <class F>
__device__ __forceinline__ void warp_records(const Sys &S, int b, long long w, long long nw, F &&f)
{
    const int lane = threadIdx.x & 31;
    if (S.flat) {
        const int n = min(S.cnt[b][0], S.cap[0]);
        for (long long k = w * 32 + lane; k < n; k += nw * 32) f(S.rec[b][S.off[0] + k], 0, 0);
    } else {
        // several warps a tile while there are more warps than tiles
        const int parts = (int)min(max(nw / max(S.ntiles, 1), 1ll), 32ll);
        for (long long t = w; t < (long long)S.ntiles * parts; t += nw) {
            const int tile = (int)(t / parts), part = (int)(t - (long long)tile * parts), ty = tile / S.ntx, tx = tile - ty * S.ntx;
            const int c = lane < kRegions ? min(S.cnt[b][tile * kCntStride + lane], S.cap[lane]) : 0;
            const int incl = warp_incl_scan(c);
            const int total = __shfl_sync(0xffffffffu, incl, kRegions - 1);
            int end[kRegions - 1];              // one past the last record of each region but the last
#pragma unroll
            for (int r = 0; r < kRegions - 1; ++r) end[r] = __shfl_sync(0xffffffffu, incl, r);
            // slot of record k: k plus the offset of its region past the records before it
            const int shift = lane < kRegions ? S.off[lane] - (incl - c) : 0;
            const int4 *base = S.rec[b] + (long long)tile * S.tile_slots;
            for (int k0 = 32 * part; k0 < total; k0 += 32 * parts) {
                const int k = k0 + lane;
                int r = 0;
#pragma unroll
                for (int q = 0; q < kRegions - 1; ++q) r += k >= end[q];
                const int at = k + __shfl_sync(0xffffffffu, shift, r);
                if (k < total) f(base[at], tx, ty);
            }
        }
    }
    const int nsp = min(S.spill_cnt[b], S.spill_cap);
    for (long long e = w * 32 + lane; e < nsp; e += nw * 32) {
        const int tile = S.spill_key[b][e] / kCntStride;
        f(S.spill_rec[b][e], tile % S.ntx, tile / S.ntx);
    }
}

// The largest tile load and staged set of the state in buffer b into err[1]
// and err[2] (what the step kernels report of later states): a warp per tile, a
// lane per source segment, and the spilled records of those segments.
__global__ void __launch_bounds__(128) k_tile_load(Sys S, int b)
{
    __shared__ int s_key[4][kSegs];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tile = blockIdx.x * 4 + warp;
    if (tile >= S.ntiles) return;
    const TileGeo G = tile_geo(S, tile);
    int m = 0;
    if (lane < kSegs) {
        const Seg g = make_seg(S, G, lane, b);
        m = g.count;
        s_key[warp][lane] = g.tile * kCntStride + g.region;
    }
    int own = lane < kRegions ? m : 0;
    __syncwarp();
    const int nsp = min(S.spill_cnt[b], S.spill_cap);
    for (int e = lane; e < nsp; e += 32) {
        const int key = S.spill_key[b][e];
        for (int s = 0; s < kSegs; ++s)
            if (s_key[warp][s] == key) {
                ++m;
                own += s < kRegions;
            }
    }
    own = __reduce_add_sync(0xffffffffu, own);
    m = __reduce_add_sync(0xffffffffu, m);
    if (lane == 0) {
        atomicMax(S.err + 1, tile_load(own, m, (2 * G.tw + 4) * (G.th + 2)));
        atomicMax(S.err + 2, m);
    }
}

// Position (FP64, exact) of a record in box coordinates.
struct BoxMap {
    double fx, fy, ux, uy;
    __device__ __forceinline__ explicit BoxMap(const Sys &S)
        : fx((double)(1ll << S.sx)), fy((double)(1ll << S.sy)), ux(S.csx_d / fx), uy(S.csy_d / fy)
    {
    }
    __device__ __forceinline__ double x(const Sys &S, int tx, int X) const
    {
        return ((double)tile_x0(S, tx) * fx + (double)X) * ux;          // the sum is exact
    }
    __device__ __forceinline__ double y(const Sys &S, int ty, int Y) const
    {
        return ((double)tile_y0(S, ty) * fy + (double)Y) * uy;
    }
};

// The state by particle id.  BUCKET false: straight into x, y, th.  true: into
// `mix`, one aligned 32-byte entry per particle, which k_split then spreads
// over the arrays: scattered writes of whole sectors instead of three partial
// ones per particle, for states that outgrow the L2.
template <bool BUCKET>
__global__ void k_gather(Sys S, int b, double *x, double *y, float *th, int4 *mix, int *seen)
{
    const BoxMap m(S);
    int n = 0;
    warp_records(S, b, (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5, (long long)gridDim.x * blockDim.x >> 5,
                 [&](const int4 &r, int tx, int ty) {
                     const unsigned id = (unsigned)r.w;
                     if (id >= (unsigned long long)S.n) {
                         atomicOr(S.err, ERR_BOUNDS);
                         return;
                     }
                     const double px = m.x(S, tx, r.x), py = m.y(S, ty, r.y);
                     if (BUCKET) {
                         const long long u = __double_as_longlong(px), v = __double_as_longlong(py);
                         int4 *o = mix + 2 * (size_t)id;
                         o[0] = make_int4((int)u, (int)(u >> 32), (int)v, (int)(v >> 32));
                         o[1] = make_int4(r.z, 0, 0, 0);
                     } else {
                         x[id] = px;
                         y[id] = py;
                         th[id] = __int_as_float(r.z);
                     }
                     ++n;
                 });
    n = __reduce_add_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(seen, n);
}

__global__ void k_split(const int4 *__restrict__ mix, long long n, double *x, double *y, float *th)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int4 u = mix[2 * i];
        const int t = mix[2 * i + 1].x;
        x[i] = __hiloint2double(u.y, u.x);
        y[i] = __hiloint2double(u.w, u.z);
        th[i] = __int_as_float(t);
    }
}

// p and q of buffer b (Sec. 3.4) of one or more systems, in exact 64-bit
// integer sums (order-free, so the result is reproducible bit for bit), plus
// the number of records: out[8 s + 0..4] of system s, which the blocks of grid
// row s sum up.
__device__ __forceinline__ void observe_system(const Sys &S, int b, unsigned long long *out)
{
    __shared__ long long red[5][8];
    long long a[5] = {0, 0, 0, 0, 0};
    warp_records(S, b, (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5, (long long)gridDim.x * blockDim.x >> 5,
                 [&](const int4 &r, int, int) {
                     const float t = __int_as_float(r.z);
                     if (!isfinite(t)) atomicOr(S.err, ERR_NAN);
                     float s1, c1, s2, c2;
                     sincosf(t, &s1, &c1);
                     sincosf(2.0f * t, &s2, &c2);
                     a[0] += __float2ll_rn(c1 * 4294967296.0f);
                     a[1] += __float2ll_rn(s1 * 4294967296.0f);
                     a[2] += __float2ll_rn(c2 * 4294967296.0f);
                     a[3] += __float2ll_rn(s2 * 4294967296.0f);
                     a[4] += 1;
                 });
    // one atomic per block and sum (N = 10^6: 71 us with one per warp, whose
    // atomics on the five words queue up, 63 so)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        const long long v = warp_sum_ll(a[k]);
        if (lane == 0) red[k][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < 5) {
        long long v = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v += red[threadIdx.x][w];
        if (v) atomicAdd(out + threadIdx.x, (unsigned long long)v);
    }
}

__global__ void __launch_bounds__(256) k_observe(Sys S, int b, unsigned long long *out) { observe_system(S, b, out); }

__global__ void __launch_bounds__(256) k_observe_all(const Sys *__restrict__ sys, int b, unsigned long long *out)
{
    observe_system(sys[blockIdx.y], b, out + 8 * (size_t)blockIdx.y);
}

// Start a measurement window at the current state of every system: its p and
// q (from the observed sums) seed last[0..1], and the steps before `until` are
// measured.  The squares are added with one rounding, as aap_observe does on the
// host, so that a window's first sample is the observed value bit for bit.
__global__ void k_begin_measure(Sys *sys, int nsys, const unsigned long long *sums, long long until)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nsys) return;
    const unsigned long long *o = sums + 8 * (size_t)i;
    Sys &S = sys[i];
    const double n = (double)S.n;
    const double c1 = (double)(long long)o[0] / kFix, s1 = (double)(long long)o[1] / kFix;
    const double c2 = (double)(long long)o[2] / kFix, s2 = (double)(long long)o[3] / kFix;
    S.last[0] = n > 0 ? sqrt(__fma_rn(c1, c1, __dmul_rn(s1, s1))) / n : 0.0;
    S.last[1] = n > 0 ? sqrt(__fma_rn(c2, c2, __dmul_rn(s2, s2))) / n : 0.0;
    S.meas_until = until;
}

// --------------------------------------------------------------- launchers --
size_t step_smem_bytes(int stage_cap, int nce_max, int hist_words)
{
    return stage_bytes(stage_cap) + table_bytes(nce_max, hist_words);
}

template <int NT, int MODEL>
static cudaError_t launch_step_t(const LaunchCfg &L, cudaStream_t st, cudaEvent_t *ev)
{
    const size_t smem = step_smem_bytes(L.stage_cap, L.nce_max, L.hist_words);
    cudaError_t e;
    if (ev && (e = cudaEventRecord(ev[0], st)) != cudaSuccess) return e;
    if (L.pipe) {
        e = L.pipe_species ? launch_step_pipe_species(L, st) : launch_step_pipe(L, st);
    } else {
        e = launch_after(k_step<NT, MODEL>, L.grid_step, NT, smem, st, L.sys, L.nsys, L.tile_base, L.ctl, L.stage_cap,
                         L.nce_max, L.scratch, L.scratch_per_block, L.scratch_cap, L.spill_list_cap);
    }
    if (e != cudaSuccess) return e;
    if (ev && (e = cudaEventRecord(ev[1], st)) != cudaSuccess) return e;
    e = launch_after(k_finish, L.grid_finish, L.grid_finish == 1 ? 1024 : 256, 0, st, L.sys, L.nsys, L.tile_base, L.ctl);
    if (e != cudaSuccess) return e;
    if (ev && (e = cudaEventRecord(ev[2], st)) != cudaSuccess) return e;
    return cudaSuccess;
}

template <int MODEL>
static cudaError_t launch_step_m(const LaunchCfg &L, cudaStream_t st, cudaEvent_t *ev)
{
    if (L.pipe) return launch_step_t<512, MODEL>(L, st, ev);     // the pipelined kernel has its own shape
    switch (L.threads) {
    case 256: return launch_step_t<256, MODEL>(L, st, ev);
    case 512: return launch_step_t<512, MODEL>(L, st, ev);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_step(const LaunchCfg &L, cudaStream_t st, cudaEvent_t *ev)
{
    if (L.knn > 0) {
        cudaError_t e = launch_mf_step(L, st, ev);
        if (e != cudaSuccess) return e;
        e = launch_after(k_finish, L.grid_finish, L.grid_finish == 1 ? 1024 : 256, 0, st, L.sys, L.nsys, L.tile_base, L.ctl);
        if (e != cudaSuccess) return e;
        if (ev && (e = cudaEventRecord(ev[2], st)) != cudaSuccess) return e;
        return cudaSuccess;
    }
    switch (L.model) {
    case 0: return launch_step_m<0>(L, st, ev);
    case 1: return launch_step_m<1>(L, st, ev);
    case 2: return launch_step_m<2>(L, st, ev);
    default: return cudaErrorInvalidValue;
    }
}

template <int NT, int MODEL>
static cudaError_t config_t(size_t smem, int *bps)
{
    // The limit belongs to the kernel, not to a handle: raise it to the
    // largest size any handle of this process asked for, so that creating a
    // smaller system never breaks the launches of a larger one.
    static std::atomic<int> limit{0};
    int want = (int)smem, prev = limit.load();
    while (want > prev && !limit.compare_exchange_weak(prev, want)) {
    }
    cudaError_t e = cudaFuncSetAttribute(k_step<NT, MODEL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         std::max(want, limit.load()));
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(bps, k_step<NT, MODEL>, NT, smem);
}

cudaError_t configure_step_kernel(int model, int threads, size_t smem_bytes, int *blocks_per_sm)
{
    if (threads == 256) {
        if (model == 0) return config_t<256, 0>(smem_bytes, blocks_per_sm);
        if (model == 1) return config_t<256, 1>(smem_bytes, blocks_per_sm);
        if (model == 2) return config_t<256, 2>(smem_bytes, blocks_per_sm);
    } else if (threads == 512) {
        if (model == 0) return config_t<512, 0>(smem_bytes, blocks_per_sm);
        if (model == 1) return config_t<512, 1>(smem_bytes, blocks_per_sm);
        if (model == 2) return config_t<512, 2>(smem_bytes, blocks_per_sm);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_insert(const Sys &S, int b, const double *x, const double *y, const float *th,
                          int mode, cudaStream_t st)
{
    const long long n = S.n;
    if (n == 0) return cudaSuccess;
    const int bs = 256;
    const long long grid = (n + bs - 1) / bs;
    k_insert<<<(unsigned)grid, bs, 0, st>>>(S, b, x, y, th, mode, 1.0 / S.csx_d, 1.0 / S.csy_d);
    return cudaGetLastError();
}

cudaError_t launch_tile_order(const LaunchCfg &L, cudaStream_t st)
{
    if (!L.pipe_few) return cudaSuccess;
    k_tile_order<<<1, 1024, 0, st>>>(L.sys, L.nsys, L.tile_base, L.ctl, 2 * L.pipe_cap_own, L.pipe_grid, L.jobs,
                                     job_cost(L), job_meta(L));
    return cudaGetLastError();
}

cudaError_t copy_dense(const LaunchCfg &L, int *dst, cudaStream_t st)
{
    return cudaMemcpyAsync(dst, job_meta(L) + 2, sizeof(int), cudaMemcpyDeviceToHost, st);
}

cudaError_t launch_tile_load(const Sys &S, int b, cudaStream_t st)
{
    k_tile_load<<<(unsigned)((S.ntiles + 3) / 4), 128, 0, st>>>(S, b);
    return cudaGetLastError();
}

cudaError_t launch_validate(const double *x, const double *y, const float *th, long long n, double lx, double ly,
                            unsigned long long *bad, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(bad, 0xff, 2 * sizeof(unsigned long long), st);
    if (e != cudaSuccess || n == 0) return e;
    k_validate_state<<<(unsigned)std::min<long long>((n + 255) / 256, 4096), 256, 0, st>>>(x, y, th, n, lx, ly, bad);
    return cudaGetLastError();
}

// Blocks of 256 threads that gather the records of n particles: 1024 particles a
// block (at most eight blocks per SM), fewer in small systems, which are a chain of
// latencies (N = 1000: 59 us to read a state with 1024 a block, 50 with 64; N =
// 200,000: 79 and 91, the counts of so many warps queue up).
static unsigned record_blocks(long long n)
{
    const long long few = std::min<long long>((n + 63) / 64, 128);
    return (unsigned)std::max<long long>(1, std::min<long long>(std::max((n + 1023) / 1024, few), 1216));
}

cudaError_t launch_gather(const Sys &S, int b, double *x, double *y, float *th, int *seen,
                          cudaStream_t st)
{
    // the region buffer of the other parity holds nothing between steps: room
    // for the 32-byte entries when the regions have at least two slots a
    // particle.  Below 2^21 particles (40 MB of arrays) the L2 collects the
    // partial writes itself.  N = 2^24, one pass: 1313 us of a get_state.
    const size_t room = (size_t)S.ntiles * S.tile_slots * sizeof(int4);
    if (S.n >= (1ll << 21) && room >= (size_t)S.n * 32) {
        int4 *mix = S.rec[b ^ 1];
        k_gather<true><<<record_blocks(S.n), 256, 0, st>>>(S, b, nullptr, nullptr, nullptr, mix, seen);
        k_split<<<1216, 256, 0, st>>>(mix, S.n, x, y, th);
    } else {
        k_gather<false><<<record_blocks(S.n), 256, 0, st>>>(S, b, x, y, th, nullptr, seen);
    }
    return cudaGetLastError();
}

cudaError_t launch_observe(const Sys &S, int b, unsigned long long *out, cudaStream_t st)
{
    const long long blocks = std::max<long long>(1, std::min<long long>((S.n + 255) / 256, 1024));
    k_observe<<<(unsigned)blocks, 256, 0, st>>>(S, b, out);
    return cudaGetLastError();
}

cudaError_t launch_begin_measure(Sys *sys, int nsys, long long max_n, int b, unsigned long long *sums, long long until,
                                 cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(sums, 0, 8 * sizeof(unsigned long long) * (size_t)nsys, st);
    if (e != cudaSuccess) return e;
    for (int s0 = 0; s0 < nsys; s0 += 65535) {
        const int n = std::min(nsys - s0, 65535);
        const dim3 grid((unsigned)std::max<long long>(1, std::min<long long>((max_n + 1023) / 1024, 256)), (unsigned)n);
        k_observe_all<<<grid, 256, 0, st>>>(sys + s0, b, sums + 8 * (size_t)s0);
    }
    k_begin_measure<<<(unsigned)((nsys + 63) / 64), 64, 0, st>>>(sys, nsys, sums, until);
    return cudaGetLastError();
}


#ifdef AAP_PHASE_TIMING
cudaError_t read_phase_times(unsigned long long *out16)
{
    return cudaMemcpyFromSymbol(out16, g_phase, sizeof(unsigned long long) * 16);
}
#endif

}  // namespace aapk
