// sp_kernels.cu -- sm_103a kernels of the region-scheduled leapfrog.
//
//   reset_kernel   arms the dependency counters and seeds the ready queue (learned
//                  order and base 32; ticket_reset_kernel: a fixed order)
//   region_kernel  persistent: takes regions in order and evolves each on chip
//   sweep_kernel   monolithic whole-grid step (the comparator)
//   feature_kernel inputs of the region cost model
//
// All arithmetic of the evolution goes through sp::site_update (sp_update.h).
#include <cuda_runtime.h>
#include <stdint.h>

#include "sp_crossing.cuh"
#include "sp_device.cuh"
#include "sp_kernels.h"
#include "sp_region_common.cuh"

namespace sp {

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ int find_sim(const RegionArgs &a, unsigned g)
{
    int lo = 0, hi = a.n_sims - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (a.sims[mid].tile_base <= g)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// ------------------------------------------------------------ queue reset
// Region id of the t-th seed of the launch (t < n_seed): the seeds of a
// simulation are its first band-0 region ids (the types without same-band
// predecessors, which lead the type order).
__device__ __forceinline__ int seed_region(const RegionArgs &a, unsigned t)
{
    int lo = 0, hi = a.n_sims - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (a.sims[mid].seed_base <= t)
            lo = mid;
        else
            hi = mid - 1;
    }
    return (int)(a.sims[lo].tile_base + (t - a.sims[lo].seed_base));
}

__global__ void reset_kernel(RegionArgs a)
{
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0) {
        a.ctl->head = 0;
        a.ctl->tail = a.n_seed;
        a.ctl->error = 0;
        a.ctl->error_info = 0;
        for (int b = 0; b < kBuckets; ++b) {
            a.ctl->bcount[b] = 0;
            a.ctl->bcursor[b] = 0;
        }
    }
    if (t >= a.total) return;
    const int s = find_sim(a, t);
    const SimDev &sd = a.sims[s];
    const TypeMeta *M = sd.tab->type;
    const unsigned local = t - sd.tile_base;
    const unsigned per_band = 8u * (unsigned)sd.Jtot;
    const unsigned band = local / per_band;
    const int S = (int)((local - band * per_band) / (unsigned)sd.Jtot);
    a.counters[t] = M[S].same_preds + (band > 0 ? M[S].prev_preds + (sd.mb_reuse ? M[S].reuse_preds : 0) : 0);
    // queue position t: the first n_seed positions hold the seeds (with the
    // learned ordering seed_kernel writes them, bucket by bucket)
    a.queue[t] = (t < a.n_seed && !a.prio) ? seed_region(a, t) : -1;
}

// Ticket order: a fresh ticket counter and error word, and an epoch above every
// done flag written before.
__global__ void ticket_reset_kernel(Ctl *ctl, int *epoch)
{
    ctl->head = 0;
    ctl->error = 0;
    ctl->error_info = 0;
    ++*epoch;
}

// Learned ordering: seeds per bucket (after reset_kernel zeroed the counts).
__global__ void seed_count_kernel(RegionArgs a)
{
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < a.n_seed) atomicAdd(&a.ctl->bcount[a.prio[seed_region(a, t)]], 1u);
}

// Learned ordering: the seeds in queue positions [0, n_seed),
// bucket 0 first (order within a bucket is immaterial).
__global__ void seed_kernel(RegionArgs a)
{
    const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= a.n_seed) return;
    const int v = seed_region(a, t);
    const int b = a.prio[v];
    unsigned base = 0;
    for (int q = 0; q < b; ++q) base += a.ctl->bcount[q];
    a.queue[base + atomicAdd(&a.ctl->bcursor[b], 1u)] = v;
}

// ------------------------------------------------------------ region kernel
// Warp-specialised persistent kernel.  A group is a manager warp (the paper's
// manager process, Sec. 4) and the NW threads of a worker that evolves one
// region at a time; a CTA holds one group or several (region_kernel, below).
//
// Manager, fixed order: manager_tickets.  With the learned order (manager_loop),
// while the workers evolve region R it waits (bounded) for the next queue
// position to be filled.  As soon as the workers report R done it hands them the
// next region and only then releases R's successors (GPU-scope fence, acq_rel
// decrements, push at zero), so the release overlaps the next region's work.
// If the next region is not ready it releases R first (the next region may be
// one of R's successors).
//
// Shared memory of a group: two phi buffers (levels of alternating
// parity) of (B+2)^3 float2 for the region box plus its halo; one float4
// (pi, c) per own cell (B^3, slots permuted by pc_slot); the band's level
// coefficients.  Of the CTA: the launch's tables (geometry and routing per
// region type) and import lists.  The tables and import lists are copied once per launch and
// the simulation descriptor travels with the handoff, so no step of a region
// waits on a table read from global memory (export entries are read through
// L1, one level ahead).
//
// Copies: the band base and the band's coefficients are requested when the
// region starts (copy group 0), the sloped initial surface of level L
// (group L) at the start of level L-1, each landing directly in its final
// place (the level-L phi buffer, L & 1, and the (pi, c) array).  This is safe
// because the cells imported for level L lie outside everything levels L-2
// and L-1 read or write (checked on the host for every region type).  Before
// level k is computed a thread waits for groups 0..k-1.
//
// One worker barrier per level.  The face cells of level k-1 are exported
// after level k is computed, before the next barrier: they are read from the
// level-(k-1) buffer and from (pi, c) of cells outside A(k) (the planner checks
// this), while level k writes the other buffer and (pi, c) of A(k).  Their
// table entries are loaded into registers before the compute.
static_assert(sizeof(SimDev) / 16 <= 32, "the manager warp copies a descriptor with one int4 per lane");

// Export entries of a level are loaded into registers before the compute of
// the next level (up to kExportPrefetch per worker thread); any remainder is
// read in batches.  Two cover the average level of base 16 with 256 workers;
// more cost registers and unrolled code for entries that rarely exist
// (128^3, base 16, 128 steps: 3.54 ms with one, 3.36 two, 3.41 three; base 8,
// 64 steps: 2.75, 2.74, 2.79).
constexpr int kExportPrefetch = 2;
constexpr int kExportBatch = 4;
constexpr int kBaseRun = 4;  // most cells of a unit of the base copy
// Most threads of a CTA (workers and manager warps of its groups), which set the
// register budget: eight regions of 64 workers, four of 128, one of more.
__host__ __device__ constexpr int region_max_groups(int nw) { return nw <= 64 ? 8 : nw <= 128 ? 4 : 1; }
__host__ __device__ constexpr int region_reporter(int nw) { return nw > 64 ? 32 : 0; }  // threads
__host__ __device__ constexpr int region_max_threads(int nw) { return region_max_groups(nw) * (nw + 32) + region_reporter(nw); }

// What one of several groups shares beside its buffers: descriptor and decoded
// region of each handoff slot, mailbox base by consumer code (type | offset bits
// << 3), and the handoff with its manager.
struct alignas(16) GroupShared {
    SimDev sd[2];
    RegionInfo ri[2];
    float2 *mb[64];
    int slot[4], handoff, done, reported, last, abort;
};

__host__ __device__ constexpr size_t region_group_bytes(int B)
{
    return (size_t)2 * (B + 2) * (B + 2) * (B + 2) * sizeof(float2) + (size_t)B * B * B * sizeof(float4) +
           kMaxHDev * sizeof(LevelCoef);
}

__device__ __forceinline__ void export_one(int2 e, float2 *const *mb_of, const float2 *__restrict__ phi,
                                           const float4 *__restrict__ pc)
{
    float2 *mb = mb_of[(e.x >> 25) & 63];
    __stcg(mb + (e.y & 0xFFFF), phi[e.x & 0x1FFF]);
    if (e.x < 0) __stcg(reinterpret_cast<float4 *>(mb + ((unsigned)e.y >> 16)), pc[(e.x >> 13) & 0xFFF]);
}

template <int NW>
__device__ __forceinline__ void export_entries(const int2 *__restrict__ el, int ne, const int2 (&pre)[kExportPrefetch],
                                               float2 *const *mb_of, const float2 *__restrict__ phi,
                                               const float4 *__restrict__ pc, int wt)
{
#pragma unroll
    for (int u = 0; u < kExportPrefetch; ++u)
        if (wt + u * NW < ne) export_one(pre[u], mb_of, phi, pc);
    for (int base = wt + kExportPrefetch * NW; base < ne; base += kExportBatch * NW) {
        int2 e[kExportBatch];
#pragma unroll
        for (int u = 0; u < kExportBatch; ++u)
            if (base + u * NW < ne) e[u] = __ldg(el + base + u * NW);
#pragma unroll
        for (int u = 0; u < kExportBatch; ++u)
            if (base + u * NW < ne) export_one(e[u], mb_of, phi, pc);
    }
}

template <int NW>
__device__ __forceinline__ void prefetch_entries(const int2 *__restrict__ el, int ne, int2 (&pre)[kExportPrefetch],
                                                 int wt)
{
#pragma unroll
    for (int u = 0; u < kExportPrefetch; ++u)
        if (wt + u * NW < ne) pre[u] = __ldg(el + wt + u * NW);
}

// Sloped initial surface of one level: mailbox chunk -> its places in shared
// memory ((pi, c) and phi of full cells, phi of neighbour-only cells).  The
// lists are in shared memory; a full cell's phi index follows from its
// (pi, c) index.
template <int NW>
__device__ __forceinline__ void import_level(const float2 *__restrict__ mb, int nf, int np,
                                             const unsigned short *fl, const unsigned short *pl, float2 *dst,
                                             float4 *pc_s, int B, int P, int wt)
{
    const int lgB = 31 - __clz(B);  // B is a power of two (4, 8 or 16)
    for (int i = wt; i < nf; i += NW) {
        const int c = fl[i];
        const int pidx = (((c >> (2 * lgB)) + 1) * P + ((c >> lgB) & (B - 1)) + 1) * P + (c & (B - 1)) + 1;
        cp_async16(pc_s + pc_slot(c, lgB, B), mb + 2 * i);
        cp_async8(dst + pidx, mb + 2 * nf + i);
    }
    for (int i = NW - 1 - wt; i < np; i += NW) cp_async8(dst + pl[i], mb + 3 * nf + i);
}

// The cells of level k are taken in 2x2x2 blocks (every extent of an active
// box is even): linear index j -> block m = j >> 3, counted z fastest, then x,
// then y (a = w0/2 and c = w2/2 blocks along x and z),
// and corner j & 7 of the block.  Eight consecutive threads then cover one
// block: a block pair along z spans all sixteen 8-byte bank pairs of a phi
// buffer (pitch B+2 = 2 mod 16 cells, plane pitch = 4 mod 16), and pc_slot
// gives the block's eight (pi, c) pairs eight different bank groups.
__device__ __forceinline__ void block_cell(int j, const LevelBox &L, int &ux, int &uy, int &uz)
{
    const int m = j >> 3;
    const int r = mdiv(m, L.rc);   // m / c
    const int jj = mdiv(r, L.ra);  // r / a
    ux = L.lo[0] + 2 * (r - jj * L.a) + (j & 1);
    uy = L.lo[1] + 2 * jj + ((j >> 1) & 1);
    uz = L.lo[2] + 2 * (m - r * L.c) + ((j >> 2) & 1);
}

// Shared-memory slot of the (pi, c) pair of the cell at local u-coordinates.
__device__ __forceinline__ int pc_slot_of(int ux, int uy, int uz, int B)
{
    const int x = ux - 1, y = uy - 1, z = uz - 1;
    return (z * B + y) * B + (x ^ ((((y & 1) << 1) | ((z & 1) << 2)) & (B - 1)));
}

// Cell i of a level's box (see block_cell).
__device__ __forceinline__ void evolve_cell(int i, const LevelBox &L, int P, int PP, int B, const float2 *__restrict__ prev_buf,
                                            float2 *__restrict__ cur, float4 *__restrict__ pc_s, const LevelCoef &co,
                                            const PhysConst &q)
{
    int ux, uy, uz;
    block_cell(i, L, ux, uy, uz);
    const int p = (uz * P + uy) * P + ux, c = pc_slot_of(ux, uy, uz, B);
    const float4 v = pc_s[c];
    float2 pi = make_float2(v.x, v.y), cc = make_float2(v.z, v.w);
    cur[p] = site_update(prev_buf[p], prev_buf[p - 1], prev_buf[p + 1], prev_buf[p - P], prev_buf[p + P], prev_buf[p - PP],
                         prev_buf[p + PP], pi, cc, co, q);
    pc_s[c] = make_float4(pi.x, pi.y, cc.x, cc.y);
}

// The manager warp asks L2 for the next region's inputs while the worker is
// still on the current region: the band base (rows of its box in the state
// arrays, one request per 128-byte line) and the region's whole mailbox (all
// levels; the region is ready, so every chunk is written).  Prefetches of
// addresses inside the arrays never fault and change no data.  Used at base
// 16 (one region per SM: 192^3, 64 steps 6.57 ms without, 6.20 with it); at base
// 8, with several regions per SM prefetching, it measured 10 % slower.
__device__ void prefetch_region_l2(const SimDev &sd, const TypeMeta &M, const RegionInfo &r, int lane)
{
    const int B = sd.B, H = sd.H;
    int gb[3];
    for (int d = 0; d < 3; ++d) gb[d] = (r.band & 1) * H + r.j[d] * B - (((r.S >> d) & 1) ? H + 1 : 1);
    const Box3 bp = M.base_phi;
    const int w1 = bp.hi[1] - bp.lo[1], rows = w1 * (bp.hi[2] - bp.lo[2]);
    const int nx = sd.n[0], ny = sd.n[1], nz = sd.n[2];
    for (int row = lane; row < rows; row += 32) {
        const int uy = bp.lo[1] + row % w1, uz = bp.lo[2] + row / w1;
        const long long rb = (long long)nx * (wrap_axis(gb[1] + uy, ny) + (long long)ny * wrap_axis(gb[2] + uz, nz));
        for (int ux = bp.lo[0]; ux < bp.hi[0] + 7; ux += 8) {  // every 8 cells and the last one
            const long long gi = rb + wrap_axis(gb[0] + min(ux, bp.hi[0] - 1), nx);
            prefetch_l2(sd.pc + gi);
            if (((ux - bp.lo[0]) & 15) == 0 || ux >= bp.hi[0] - 1) prefetch_l2(sd.phi + gi);
        }
    }
    const float2 *mb = sd.mbox + (long long)(r.band & 1) * sd.mb_slot + sd.mb_type_off[r.S] + (long long)r.jl * M.mb_size;
    for (int i = 16 * lane; i < M.mb_size; i += 16 * 32) prefetch_l2(mb + i);
}

// Manager warp: hand regions to the worker, release finished ones.
__device__ void manager_loop(const RegionArgs &a, const TablesDev *s_tabs, int *s_slot, SimDev *s_sd,
                             RegionInfo *s_ri, int *s_handoff, int *s_done, bool prefetch)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long limit = a.ctl->wait_limit_ns;
    int seq = 0;           // handoffs made
    int pending = -1;      // region handed at seq, not yet released
    RegionInfo pend_info = {};
    unsigned idx = 0;
    if (lane == 0) idx = atomicAdd(&a.ctl->head, 1u);
    idx = __shfl_sync(0xffffffffu, idx, 0);
    int got = 0, v = -1;
    int prepared = 0;  // the next region's descriptor is in its handoff slot
    RegionInfo ni = pend_info;
    unsigned long long t0 = globaltimer_ns();
    unsigned long long t_progress = t0;  // last handoff or release
    for (unsigned spin = 0;; ++spin) {
        int done = 0;
        if (lane == 0) {
            if (!got) {
                if (idx >= a.total) {
                    got = 1;
                    v = -1;
                } else {
                    const int q = ld_acquire_gpu(a.queue + idx);
                    if (q >= 0) {
                        got = 1;
                        v = q;
                    } else if (ld_relaxed_gpu(&a.ctl->error) != 0) {
                        got = 1;
                        v = -2;
                    } else if ((spin & 15u) == 15u && globaltimer_ns() - t0 > limit) {
                        atomicCAS(&a.ctl->error, 0, kDevTimeout);
                        atomicExch(&a.ctl->error_info, (int)idx);
                        got = 1;
                        v = -2;
                    }
                }
            }
        }
        const int have = __shfl_sync(0xffffffffu, got, 0);
        const int next = __shfl_sync(0xffffffffu, v, 0);
        if (have && !prepared) {
            // while the worker is still busy: decode the next region and put it
            // and its simulation's descriptor into the free handoff slot
            if (next >= 0) {
                ni = decode_region(a.sims, a.n_sims, next);
                const int slot = (seq + 1) & 1;
                const int4 *src = reinterpret_cast<const int4 *>(a.sims + ni.sim);
                int4 *dst = reinterpret_cast<int4 *>(s_sd + slot);
                if (lane < (int)(sizeof(SimDev) / 16)) dst[lane] = src[lane];
                if (lane == 0) s_ri[slot] = ni;
                __syncwarp();
                if (prefetch) {
                    const SimDev &nsd = s_sd[slot];
                    prefetch_region_l2(nsd, s_tabs[nsd.tab_index].type[ni.S], ni, lane);
                }
            }
            prepared = 1;
        }
        if (lane == 0) done = ld_acquire_cta_shared(s_done) == seq;
        done = __shfl_sync(0xffffffffu, done, 0);
        if (done && have) {
            if (lane == 0) {
                s_slot[(seq + 1) & 3] = next;
                st_release_cta_shared(s_handoff, seq + 1);
            }
            ++seq;
            if (pending >= 0) {
                const SimDev &sd = a.sims[pend_info.sim];
                release_successors(a, sd, s_tabs[sd.tab_index], pend_info, lane, 0ull, pending);
            }
            pending = next;
            if (next < 0) break;
            pend_info = ni;
            prepared = 0;
            if (lane == 0) {
                got = 0;
                idx = atomicAdd(&a.ctl->head, 1u);
                t0 = globaltimer_ns();
                t_progress = t0;
            }
            continue;
        }
        if (done && pending >= 0) {
            // the next region is not ready yet: it may wait on this release
            const SimDev &sd = a.sims[pend_info.sim];
            release_successors(a, sd, s_tabs[sd.tab_index], pend_info, lane, 0ull, pending);
            pending = -1;
            if (lane == 0) t_progress = globaltimer_ns();
            continue;
        }
        // no handoff and no release for 4 wait limits: the worker is stuck;
        // record it and stop (the worker's own bounded wait then ends it too)
        int stuck = 0;
        if (lane == 0 && (spin & 15u) == 15u && globaltimer_ns() - t_progress > 4 * limit) {
            atomicCAS(&a.ctl->error, 0, kDevTimeout);
            stuck = 1;
        }
        if (__shfl_sync(0xffffffffu, stuck, 0)) break;
        if (!have) __nanosleep(32);  // waiting on the queue backs off; waiting on the worker polls shared memory
    }
}

// The region of ticket t: bands in order, within a band the types by phase (a
// predecessor's type is a subset of the region's, one phase or more earlier),
// within a type the positions of all simulations.  Region ids stay those of
// the queue (simulation by simulation).
__device__ __forceinline__ RegionInfo decode_ticket(const RegionArgs &a, unsigned t, int *id)
{
    RegionInfo r;
    const unsigned all = (unsigned)a.all_tiles;
    const unsigned run = t / all, pos = t - run * all;
    r.band = (int)(run >> 3);
    r.S = (int)(kPhaseOrder >> (4 * (run & 7u))) & 7;
    int lo = 0, hi = a.n_sims - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((unsigned)a.sims[mid].tile_first <= pos)
            lo = mid;
        else
            hi = mid - 1;
    }
    const SimDev &sd = a.sims[lo];
    r.sim = lo;
    r.jl = (int)(pos - (unsigned)sd.tile_first);
    r.j[0] = r.jl % sd.J[0];
    r.j[1] = (r.jl / sd.J[0]) % sd.J[1];
    r.j[2] = r.jl / (sd.J[0] * sd.J[1]);
    *id = (int)(sd.tile_base + (unsigned)((r.band * 8 + r.S) * sd.Jtot + r.jl));
    return r;
}

// Flag of predecessor i of region r, or nullptr when it has fewer.
__device__ __forceinline__ const int *pred_flag(const RegionArgs &a, const SimDev &sd, const TablesDev &T, const RegionInfo &r,
                                                int i)
{
    const int kinds = r.band == 0 ? 0 : sd.mb_reuse ? 2 : 1;
    if (i >= T.pred_n[r.S][kinds]) return nullptr;
    const Pred p = T.preds[((r.band & 1) * kTypes + r.S) * kMaxPreds + i];
    int jc = 0, mul = 1;
    for (int d = 0; d < 3; ++d) {
        int v = r.j[d] + p.e[d];
        v += (v < 0) ? sd.J[d] : 0;
        v -= (v >= sd.J[d]) ? sd.J[d] : 0;
        jc += v * mul;
        mul *= sd.J[d];
    }
    const int band = r.band - (p.type_prev >> 3);
    return a.flags + (sd.tile_base + (unsigned)((band * 8 + (p.type_prev & 7)) * sd.Jtot + jc));
}

// What a group's manager, its worker and the reporter warp share: the regions
// handed over (by count mod 4), finished and reported so far, and how many there
// will be (-1: not known).
struct GroupSync {
    int *slot, *handoff, *done, *reported, *last;
};

// Sets the done flag of the group's next finished region, if there is one past
// the first seq: the release orders the worker's surfaces (its done count is
// acquired) before the flag.
__device__ __forceinline__ bool report_next(const RegionArgs &a, int epoch, const GroupSync &y, int seq)
{
    if (ld_acquire_cta_shared(y.done) <= seq) return false;
    const int g = y.slot[(seq + 1) & 3];
    if (g != a.fault_drop) st_release_gpu(a.flags + g, epoch);
    return true;
}

// Manager warp in ticket order: takes the next ticket, stages its region while
// the worker evolves the current one, polls the done flags of the region's
// predecessors (two per lane) and hands it over, before the worker has finished
// if it can, so that the worker goes from one region to the next by itself.  No
// queue and no counters: a release is one store where decrementing every
// successor and pushing the ready ones took about 3 us, as long as a base-8
// region, and all managers shared the queue's head and tail.  Tickets are taken
// in a topological order and every ticket is held by a resident manager whose
// worker has only smaller ones before it, so the waits end; each is bounded
// anyway.  Polls that acquire and stores that release, not relaxed ones with
// fences: a fence waits about a microsecond in either place (32^3, base 8, 64
// steps: 401 us with a fence at both ends, 380 without).
// OWN: the manager also reports (64 workers, where a CTA has no room for
// the reporter warp).
template <bool OWN>
__device__ void manager_tickets(const RegionArgs &a, const TablesDev *s_tabs, SimDev *s_sd, RegionInfo *s_ri,
                                const GroupSync &y, bool prefetch)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long limit = a.ctl->wait_limit_ns;
    const int epoch = *(volatile int *)a.epoch;
    int seq = 0, reported = 0;  // handoffs made; OWN, lane 0: regions reported
    // lane 0 waits for the worker to have finished n regions (and for the last but
    // two of them to be reported: there are four id slots); false: it is stuck
    auto finished = [&](int n) {
        unsigned long long t0 = 0;
        for (unsigned spin = 0;; ++spin) {
            if (OWN)
                reported += report_next(a, epoch, y, reported);
            if (OWN ? reported >= n
                    : ld_acquire_cta_shared(y.done) >= n && ld_acquire_cta_shared(y.reported) >= n - 2)
                return true;
            if ((spin & 63u) == 63u) {
                if (t0 == 0) t0 = globaltimer_ns();
                if (globaltimer_ns() - t0 > 4 * limit) {
                    atomicCAS(&a.ctl->error, 0, kDevTimeout);
                    return false;
                }
            }
        }
    };
    for (;;) {
        // the descriptor slot of the region before the current one
        bool stop = false;
        unsigned t = 0;
        if (lane == 0) {
            stop = !finished(seq - 1);
            if (!stop) t = atomicAdd(&a.ctl->head, 1u);
        }
        stop = __shfl_sync(0xffffffffu, stop, 0);
        t = __shfl_sync(0xffffffffu, t, 0);
        int next = stop ? -2 : -1;  // region handed over; -1: no more, -2: stop
        if (!stop && t < a.total) {
            const RegionInfo ni = decode_ticket(a, t, &next);
            const int slot = (seq + 1) & 1;
            const int4 *src = reinterpret_cast<const int4 *>(a.sims + ni.sim);
            int4 *dst = reinterpret_cast<int4 *>(s_sd + slot);
            if (lane < (int)(sizeof(SimDev) / 16)) dst[lane] = src[lane];
            if (lane == 0) s_ri[slot] = ni;
            __syncwarp();
            const SimDev &nsd = s_sd[slot];
            const TablesDev &T = s_tabs[nsd.tab_index];
            const int *f0 = pred_flag(a, nsd, T, ni, lane), *f1 = pred_flag(a, nsd, T, ni, lane + 32);
            const unsigned long long t0 = globaltimer_ns();
            for (unsigned spin = 0;; ++spin) {
                if (f0 && ld_acquire_gpu(f0) == epoch) f0 = nullptr;
                if (f1 && ld_acquire_gpu(f1) == epoch) f1 = nullptr;
                const bool ok = !f0 && !f1;
                if (__all_sync(0xffffffffu, ok)) break;
                if (OWN && lane == 0) reported += report_next(a, epoch, y, reported);
                if ((spin & 15u) == 15u) {
                    if (lane == 0) {
                        if (ld_relaxed_gpu(&a.ctl->error) != 0) {
                            stop = true;
                        } else if (globaltimer_ns() - t0 > limit) {
                            atomicCAS(&a.ctl->error, 0, kDevTimeout);
                            atomicExch(&a.ctl->error_info, (int)t);
                            stop = true;
                        }
                    }
                    stop = __shfl_sync(0xffffffffu, stop, 0);
                    if (stop) {
                        next = -2;
                        break;
                    }
                }
                // The polls share the SM's issue slots and L2 with the working groups, and
                // an acquire empties L1 (32^3, base 4, 64 steps: 642 us at 100 ns, 562 at
                // 300, 565 at 500; 48^3, base 8: 521, 456, 454; 545 and 444 at 300 since a
                // lane leaves out what it has seen).
                __nanosleep(300);
            }
            __syncwarp();  // every lane's acquire before lane 0's release below
        }
        if (lane == 0) {
            y.slot[(seq + 1) & 3] = next;
            if (next < 0) st_release_cta_shared(y.last, seq);
            st_release_cta_shared(y.handoff, seq + 1);
        }
        if (next < 0) {
            if (OWN && lane == 0) finished(seq);
            break;
        }
        ++seq;
        if (prefetch) {
            const SimDev &nsd = s_sd[seq & 1];
            prefetch_region_l2(nsd, s_tabs[nsd.tab_index].type[s_ri[seq & 1].S], s_ri[seq & 1], lane);
        }
    }
}

// Reporter warp of a CTA: lane g sets the done flag of each region that group g
// has finished.  A warp of its own, so that a flag waits for no manager's staging
// or poll (48^3, base 8, 64 steps: 488 us with reporting managers, 455).
__device__ void report_regions(const RegionArgs &a, int groups, const GroupSync &y)
{
    const int lane = threadIdx.x & 31;
    const int epoch = *(volatile int *)a.epoch;
    const unsigned long long limit = 16 * a.ctl->wait_limit_ns;
    unsigned long long t0 = globaltimer_ns();
    int seq = 0;  // regions reported
    bool live = lane < groups;
    for (unsigned spin = 0; __any_sync(0xffffffffu, live); ++spin) {
        if (live) {
            const int last = ld_acquire_cta_shared(y.last);
            if (report_next(a, epoch, y, seq)) {
                st_release_cta_shared(y.reported, ++seq);
                t0 = globaltimer_ns();
            } else if (last >= 0 && seq >= last) {
                live = false;
            } else if ((spin & 255u) == 255u &&
                       ((last >= 0 && ld_relaxed_gpu(&a.ctl->error) != 0) || globaltimer_ns() - t0 > limit)) {
                live = false;  // the launch has failed
            }
        }
    }
}

// One instantiation per worker count NW, with the region base BB fixed at
// compile time (16: index arithmetic in shifts, stencil offsets as immediates;
// measured 1.5 % faster) or, for BB = 0, taken from the descriptor (bases 4
// and 8, whose several CTAs per SM favour the smaller code: the fixed-base
// build measured 1.4 % slower there).  A launch holds simulations of one base.
// A CTA hosts `groups` regions at a time, each a group of a manager warp and NW
// workers with its own buffers and named barrier, which share the tables and
// import lists (base 8: 10.8 KB beside 25.3 KB a region, so eight regions fit
// an SM where six CTAs did).  Bound by latency, not by a pipe: a
// region is a chain of requesting its base (0.8 us at base 16), waiting for it
// (0.4) and its levels (0.6 us each, imports, barrier, indices, update, exports),
// in which every instruction counts: 40 % of the issue slots and 28 % of DRAM are
// used (base 8: 62 and 34 %).  So the tables hold what a level reads in three wide
// loads (128^3, base 16, 128 steps 3.60 to 3.50 ms), quotients are a multiply and
// a shift (3.46), and a thread takes one cell at a time (two interleaved: 3.46,
// one 3.41; the shorter code also leaves registers).  On a small grid the hop from
// a region to its successor adds 2 us.  With the ready queue, and six CTAs at
// base 8, against this: 256^3, base 8, 8 steps 3.18 and 2.85 ms; 32^3, 64 steps 618
// and 300 us; 192^3, base 16, 64 steps 6.35 and 5.55 ms; 64^3 540 and 386 us.
template <int NW, int BB>
__global__ void __launch_bounds__(region_max_threads(NW), 1) region_kernel(RegionArgs a, int max_P_launch)
{
    const int max_P = BB ? BB + 2 : max_P_launch;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // Static, apart from the buffers, so that no store to a buffer can alias it.
    // One region per CTA: a variable each at a constant address (as members of
    // one struct they are 2.5 % slower at base 16); several: one struct each
    // (an array of each member is 11 % slower at base 8, a base register more
    // per array).
    constexpr int G = region_max_groups(NW);
    constexpr bool one = G == 1;
    __shared__ GroupShared g_shared[G];
    __shared__ int x_slot[4], x_handoff, x_done, x_reported, x_last, x_abort;
    __shared__ SimDev x_sd[2];
    __shared__ RegionInfo x_ri[2];
    __shared__ float2 *x_mb[64];
    const int groups = one ? 1 : blockDim.x / (NW + 32);  // and the reporter warp
    const int group = one ? 0 : threadIdx.x / (NW + 32), tid = threadIdx.x - group * (NW + 32);
    const int kWorkerBarrier = 1 + group;
    const int P3 = max_P * max_P * max_P, B3 = (max_P - 2) * (max_P - 2) * (max_P - 2);
    // one region: its buffers at constant offsets, then the tables; several: the tables first
    TablesDev *s_tabs = reinterpret_cast<TablesDev *>(smem_raw + (one ? region_group_bytes(max_P - 2) : 0));
    unsigned char *const mine =
        smem_raw + (one ? 0 : (size_t)a.n_tabs * sizeof(TablesDev) + (size_t)group * region_group_bytes(max_P - 2));
    float2 *phi_buf0 = reinterpret_cast<float2 *>(mine);
    float2 *phi_buf1 = phi_buf0 + P3;
    float4 *pc_s = reinterpret_cast<float4 *>(phi_buf1 + P3);
    LevelCoef *s_coef = reinterpret_cast<LevelCoef *>(pc_s + B3);
    {  // the launch's tables, once
        const int4 *src = reinterpret_cast<const int4 *>(a.tabs);
        int4 *dst = reinterpret_cast<int4 *>(s_tabs);
        const int nt = a.n_tabs * (int)(sizeof(TablesDev) / 16);
        for (int i = threadIdx.x; i < nt; i += blockDim.x) dst[i] = src[i];
    }
    __syncthreads();
    unsigned short *s_imp = reinterpret_cast<unsigned short *>(smem_raw + (size_t)a.n_tabs * sizeof(TablesDev) +
                                                               (size_t)groups * region_group_bytes(max_P - 2));
    for (int t = threadIdx.x; t < kTypes * a.n_tabs; t += blockDim.x) {  // the shortest runs that give each worker one
        TypeMeta &m = s_tabs[t / kTypes].type[t % kTypes];
        const int w2 = m.base_phi.hi[2] - m.base_phi.lo[2];
        int len = 1;
        while (len < kBaseRun && m.base_cols * ((w2 + len - 1) / len) > NW) ++len;
        m.base_len = len;
        m.base_runs = (w2 + len - 1) / len;
    }
    for (int t = 0; t < a.n_tabs; ++t) {  // every import list of the launch, once
        const int4 *src = reinterpret_cast<const int4 *>(s_tabs[t].imp);
        int4 *dst = reinterpret_cast<int4 *>(s_imp + s_tabs[t].imp_smem);
        for (int i = threadIdx.x; i < s_tabs[t].imp_n / 8; i += blockDim.x) dst[i] = src[i];
    }
    const bool reporter = region_reporter(NW) && threadIdx.x >= groups * (NW + 32);
    GroupShared &gs = g_shared[reporter ? min(threadIdx.x & 31, groups - 1) : group];  // the reporter's lanes: a group each
    int *const s_slot = one ? x_slot : gs.slot;
    int &s_handoff = one ? x_handoff : gs.handoff, &s_done = one ? x_done : gs.done, &s_abort = one ? x_abort : gs.abort;
    SimDev *const s_sd = one ? x_sd : gs.sd;
    RegionInfo *const s_ri = one ? x_ri : gs.ri;
    float2 **const s_mb = one ? x_mb : gs.mb;
    if (tid == 0) {
        s_handoff = 0;
        s_done = 0;
        (one ? x_reported : gs.reported) = 0;
        (one ? x_last : gs.last) = -1;
    }
    __syncthreads();
    const GroupSync sync = {s_slot, &s_handoff, &s_done, one ? &x_reported : &gs.reported, one ? &x_last : &gs.last};
    if (reporter) {
        if (a.flags) report_regions(a, groups, sync);
        return;
    }
    if (tid < 32) {
        if (a.flags)
            manager_tickets<region_reporter(NW) == 0>(a, s_tabs, s_sd, s_ri, sync, BB == 16);
        else
            manager_loop(a, s_tabs, s_slot, s_sd, s_ri, &s_handoff, &s_done, BB == 16);
        return;
    }
    const int wt = tid - 32;  // worker thread index
    // Its index with the warps in reverse, for the exports: the cells of a level and
    // its full imports are dealt out from worker 0, the exports and the phi-only
    // imports from the last one, so that no warp is last with all of them (128^3,
    // base 16, 128 steps 3.71 ms with every list from worker 0, 3.60 so; 3.68 with
    // each list starting where the one before ended).
    const int wr = NW - 32 - (wt & ~31) + (wt & 31);
    for (int seq = 1;; ++seq) {
        if (wt == 0) {
            // bounded wait for the manager's handoff (a shared-memory poll: the
            // handoff normally follows within a microsecond)
            s_abort = 0;
            unsigned long long t0 = 0;
            for (unsigned spin = 0; ld_acquire_cta_shared(&s_handoff) < seq; ++spin) {
                if ((spin & 63u) == 63u) {
                    if (t0 == 0) t0 = globaltimer_ns();
                    if (globaltimer_ns() - t0 > 8 * a.ctl->wait_limit_ns) {
                        atomicCAS(&a.ctl->error, 0, kDevTimeout);
                        s_abort = 1;
                        break;
                    }
                }
            }
        }
        named_barrier(kWorkerBarrier, NW);
        if (s_abort) break;
        const int g = s_slot[seq & 3];
        if (g < 0) break;
        if (a.trace && wt == 0) a.trace[2 * (size_t)g] = globaltimer_ns();

        const RegionInfo r = s_ri[seq & 1];  // decoded by the manager at the handoff
        const SimDev &sd = s_sd[seq & 1];
        const TablesDev &T = s_tabs[sd.tab_index];
        const TypeMeta &M = T.type[r.S];
        const int S = r.S, band = r.band, jl = r.jl;
        const int B = BB ? BB : sd.B, H = B / 2, P = B + 2, PP = P * P;  // sd.B == BB when BB is fixed
        int gbase[3];  // global coordinate of local u = 0 along each axis
        for (int d = 0; d < 3; ++d) gbase[d] = (band & 1) * H + r.j[d] * B - (((S >> d) & 1) ? H + 1 : 1);
        const int nx = sd.n[0], ny = sd.n[1], nz = sd.n[2];
        const long long nxy = (long long)nx * ny;
        const long long slot = (long long)(band & 1) * sd.mb_slot;
        if (wt < 64) {
            // mailbox of the consumer with this code, if the code names one
            const int Sc = wt & 7, eb = wt >> 3;
            int jc = 0, mul = 1;
            for (int d = 0; d < 3; ++d) {
                int v = r.j[d] + ((eb >> d) & 1);
                v -= (v >= sd.J[d]) ? sd.J[d] : 0;
                jc += v * mul;
                mul *= sd.J[d];
            }
            s_mb[wt] = sd.mbox + slot + sd.mb_type_off[Sc] + (long long)jc * T.type[Sc].mb_size;
        }

        // ---- group 0: the band base (tops of the previous band) + coefficients ----
        // Work units are (run of base_len cells along z, column), columns fastest:
        // every worker gets a similar share whatever the box's shape, and
        // consecutive threads read consecutive cells along x.  A run's cells are
        // independent straight-line code: of the first microsecond of a region
        // most was one warp's chain through runs of four while others had none
        // (base 16, types 3 5 6 7: 0.68 us to the last request).
        {
            if (wt < H) cp_async16(s_coef + wt, sd.coef + band * H + wt);
            const Box3 bp = M.base_phi;
            const Box3 bc = M.base_pc;
            const int w0 = bp.hi[0] - bp.lo[0];
            const int ncol = M.base_cols, len = M.base_len, units = ncol * M.base_runs;
            for (int u = wt; u < units; u += NW) {
                const int run = mdiv(u, M.mul_cols);
                const int i = u - run * ncol;
                const int t1 = mdiv(i, M.mul_w0);
                const int ux = bp.lo[0] + i - t1 * w0;
                const int uy = bp.lo[1] + t1;
                const int oxy = (ux < bc.lo[0] || ux >= bc.hi[0]) + (uy < bc.lo[1] || uy >= bc.hi[1]);
                const long long gxy =
                    (long long)wrap_axis(gbase[0] + ux, nx) + (long long)nx * wrap_axis(gbase[1] + uy, ny);
                const int z0 = bp.lo[2] + len * run;
#pragma unroll
                for (int e = 0; e < kBaseRun; ++e) {
                    const int uz = z0 + e;
                    // out > 1: not a 7-point neighbour of A(1)
                    const int out = oxy + (uz < bc.lo[2] || uz >= bc.hi[2]);
                    const long long gi = gxy + nxy * wrap_axis(gbase[2] + uz, nz);
                    if (e < len && uz < bp.hi[2] && out <= 1) {
                        cp_async8(phi_buf0 + (uz * P + uy) * P + ux, sd.phi + gi);
                        if (out == 0) cp_async16(pc_s + pc_slot_of(ux, uy, uz, B), sd.pc + gi);
                    }
                }
            }
            cp_async_commit();
        }
        // ---- sloped initial surface: level L lands as copy group L, issued one
        // level ahead (level 1 now, level k+1 at the start of level k) ----
        const float2 *mb_self = sd.mbox + slot + sd.mb_type_off[S] + (long long)jl * M.mb_size;
        const unsigned short *s_imp_t = s_imp + T.imp_smem;
        auto issue_level = [&](int L) {
            if (L <= H - 1) {
                const LevelLists l = M.lists[L];
                if (l.full_n + l.phi_n > 0)
                    import_level<NW>(mb_self + l.mb_off, l.full_n, l.phi_n, s_imp_t + l.imp_off,
                                     s_imp_t + l.imp_off + l.full_n, (L & 1) ? phi_buf1 : phi_buf0, pc_s, B, P, wt);
            }
            cp_async_commit();  // one group per level, empty or not
        };
        issue_level(1);

        const int nlev = M.levels;
        const PhysConst q = sd.q;
        int2 pre[kExportPrefetch];
        for (int k = 1; k <= nlev; ++k) {
            const float2 *__restrict__ prev_buf = (k & 1) ? phi_buf0 : phi_buf1;
            float2 *__restrict__ cur = (k & 1) ? phi_buf1 : phi_buf0;
            issue_level(k + 1);  // lands in buffer (k+1) & 1 outside what level k reads
            // export entries of level k-1, loaded now, used after the compute
            const LevelExports ex = M.exps[k - 1];  // none at level 0
            const int ne = ex.n;
            const int2 *el = T.exp + ex.off;
            prefetch_entries<NW>(el, ne, pre, wr);
            cp_async_wait_pending(2);  // groups 0..k-1 (base, coefficients, levels < k) have landed
            named_barrier(kWorkerBarrier, NW);
            // ---- evolve the cells of level k ----
            const LevelCoef co = s_coef[k - 1];
            const LevelBox L = M.box[k];
            for (int i = wt; i < L.cnt; i += NW) evolve_cell(i, L, P, PP, B, prev_buf, cur, pc_s, co, q);
            // ---- final surface of level k-1 (read-only data of level k-1) ----
            if (ne > 0) export_entries<NW>(el, ne, pre, s_mb, prev_buf, pc_s, wr);
        }
        const float2 *last = (nlev & 1) ? phi_buf1 : phi_buf0;
        if (nlev <= H - 1) {
            // ---- final surface of the last level ----
            const int ne = M.exps[nlev].n;
            const int2 *el = T.exp + M.exps[nlev].off;
            prefetch_entries<NW>(el, ne, pre, wr);
            named_barrier(kWorkerBarrier, NW);
            export_entries<NW>(el, ne, pre, s_mb, last, pc_s, wr);
        } else {
            named_barrier(kWorkerBarrier, NW);
            // ---- tops of the inverted pyramid: the next band's base ----
            const int lgB = 31 - __clz(B), share = B * B * B / NW;
            const int len = share >= 4 ? 4 : share >= 2 ? 2 : 1;  // cells of a unit along z
            for (int u = wt; u < B * B * B / len; u += NW) {
                const int ux = 1 + (u & (B - 1));
                const int uy = 1 + ((u >> lgB) & (B - 1));
                const int z0 = 1 + len * (u >> (2 * lgB));
                const long long gxy =
                    (long long)wrap_axis(gbase[0] + ux, nx) + (long long)nx * wrap_axis(gbase[1] + uy, ny);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int uz = z0 + e;
                    const long long gi = gxy + nxy * wrap_axis(gbase[2] + uz, nz);
                    if (e < len) {
                        __stcg(sd.phi + gi, last[(uz * P + uy) * P + ux]);
                        __stcg(sd.pc + gi, pc_s[pc_slot_of(ux, uy, uz, B)]);
                    }
                }
            }
        }
        named_barrier(kWorkerBarrier, NW);
        if (wt == 0) {
            if (a.trace) a.trace[2 * (size_t)g + 1] = globaltimer_ns();
            st_release_cta_shared(&s_done, seq);
        }
    }
}

// ------------------------------------------------------------ sweep kernel
// One level of the whole grid: block 32 x 4 over (x, y), each thread marches
// a chunk of z keeping phi(z-1), phi(z), phi(z+1) in registers; x and y
// neighbours come through L1.  48 bytes per site-update: bound by DRAM beyond
// L2, by L2 and the chain of its round trips below.  Ten blocks of 128 threads
// per SM (48 registers): 512 x 512 x 128 249.5 us, 128^3 10.7 us; the same
// threads as five blocks of 32 x 8 253.4 and 11.0 us, and at 40 registers, six
// blocks, 259 and 12.0 us.
constexpr int kSweepY = 4, kSweepPerSm = 10;
__global__ void __launch_bounds__(32 * kSweepY, kSweepPerSm)
    sweep_kernel(const float2 *__restrict__ phi_in, float2 *__restrict__ phi_out, float4 *__restrict__ pc, int nx, int ny,
                 int nz, int zchunk, const LevelCoef *__restrict__ coef, int lvl, PhysConst q)
{
    const int x = blockIdx.x * 32 + threadIdx.x;
    const int y = blockIdx.y * kSweepY + threadIdx.y;
    if (x >= nx || y >= ny) return;
    const int z0 = blockIdx.z * zchunk;
    const int z1 = min(z0 + zchunk, nz);
    const int xm = x == 0 ? nx - 1 : x - 1, xp = x == nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
    const LevelCoef co = coef[lvl];
    const long long plane = (long long)nx * ny;
    const int zb = z0 == 0 ? nz - 1 : z0 - 1;
    float2 zprev = phi_in[zb * plane + (long long)y * nx + x];
    float2 zcur = phi_in[z0 * plane + (long long)y * nx + x];
    for (int z = z0; z < z1; ++z) {
        const int zn = z == nz - 1 ? 0 : z + 1;
        const float2 znext = phi_in[zn * plane + (long long)y * nx + x];
        const long long zo = z * plane;
        const long long row = zo + (long long)y * nx;
        const float4 v = pc[row + x];
        float2 p = make_float2(v.x, v.y), cc = make_float2(v.z, v.w);
        const float2 out = site_update(zcur, phi_in[row + xm], phi_in[row + xp], phi_in[zo + (long long)ym * nx + x],
                                       phi_in[zo + (long long)yp * nx + x], zprev, znext, p, cc, co, q);
        phi_out[row + x] = out;
        pc[row + x] = make_float4(p.x, p.y, cc.x, cc.y);
        zprev = zcur;
        zcur = znext;
    }
}

// ------------------------------------------------------------ region features
// The 16 inputs of the region cost model, per region of a launch, from its
// descriptor and from the state at the start of the call (the footprint of
// the region's own cells, sampled on a 2 x 2 x 2 lattice):
//   0-2  inverted axes of the region type (x, y, z);  3  |S| / 3 (phase);
//   4    B / 16;  5  log2(sites) / 24;  6  nu / 2;  7  a^2 lambda at the band's
//   first level;  8  band / bands;  9  (4 band + |S|) / (4 bands);
//   10, 11  mean and max |phi|^2;  12  mean |pi|^2;  13  fraction of sampled
//   xy plaquettes with nonzero winding;  14  mean |phi(x+1) - phi(x)|^2 / dx^2;
//   15  the region's measured time in the previous traced call (us / 20), or 0.
// simf[s] = (B / 16, log2(sites) / 24, nu / 2, 0) of simulation s.
__global__ void __launch_bounds__(128) feature_kernel(RegionArgs a, const float4 *__restrict__ simf,
                                                      const unsigned long long *__restrict__ prev_trace,
                                                      float *__restrict__ X)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= (int)a.total) return;
    const RegionInfo r = decode_region(a.sims, a.n_sims, g);
    const SimDev &sd = a.sims[r.sim];
    const float4 sf = simf[r.sim];
    const int S = r.S, B = sd.B, H = sd.H, nb = sd.nbands;
    const int ns = (S & 1) + ((S >> 1) & 1) + ((S >> 2) & 1);
    float f[16];
    f[0] = (float)(S & 1);
    f[1] = (float)((S >> 1) & 1);
    f[2] = (float)((S >> 2) & 1);
    f[3] = ns / 3.0f;
    f[4] = sf.x;
    f[5] = sf.y;
    f[6] = sf.z;
    f[7] = sd.coef[r.band * H].m;
    f[8] = (float)r.band / (float)nb;
    f[9] = (float)(4 * r.band + ns) / (float)(4 * nb);
    int gb[3];
    for (int d = 0; d < 3; ++d) gb[d] = (r.band & 1) * H + r.j[d] * B - (((S >> d) & 1) ? H + 1 : 1);
    const int nx = sd.n[0], ny = sd.n[1], nz = sd.n[2];
    const int stride = B / 2;
    double sphi = 0.0, spi = 0.0, sgrad = 0.0;
    float mphi = 0.0f;
    int pierced = 0;
    for (int m = 0; m < 8; ++m) {
        const int x = wrap_axis(gb[0] + 1 + stride * (m & 1), nx);
        const int y = wrap_axis(gb[1] + 1 + stride * ((m >> 1) & 1), ny);
        const int z = wrap_axis(gb[2] + 1 + stride * (m >> 2), nz);
        const int x1 = x + 1 == nx ? 0 : x + 1, y1 = y + 1 == ny ? 0 : y + 1;
        const long long row = (long long)nx * (y + (long long)ny * z), row1 = (long long)nx * (y1 + (long long)ny * z);
        const float2 p0 = sd.phi[row + x], p1 = sd.phi[row + x1], p2 = sd.phi[row1 + x1], p3 = sd.phi[row1 + x];
        const float4 pc = sd.pc[row + x];
        const float a2 = p0.x * p0.x + p0.y * p0.y;
        sphi += a2;
        mphi = fmaxf(mphi, a2);
        spi += (double)(pc.x * pc.x + pc.y * pc.y);
        const float dx = p1.x - p0.x, dy = p1.y - p0.y;
        sgrad += (double)(dx * dx + dy * dy);
        pierced += (crossing(p0, p1) + crossing(p1, p2) + crossing(p2, p3) + crossing(p3, p0)) != 0;
    }
    f[10] = (float)(sphi / 8.0);
    f[11] = mphi;
    f[12] = (float)(spi / 8.0);
    f[13] = pierced / 8.0f;
    f[14] = (float)(sgrad / 8.0) * sd.q.inv_dx2;
    f[15] = 0.0f;
    if (prev_trace) {
        const unsigned long long t0 = prev_trace[2 * (size_t)g], t1 = prev_trace[2 * (size_t)g + 1];
        if (t1 > t0) f[15] = (float)((double)(t1 - t0) * 1e-3 / 20.0);
    }
    float4 *o = reinterpret_cast<float4 *>(X + 16 * (size_t)g);
    for (int q = 0; q < 4; ++q) o[q] = make_float4(f[4 * q], f[4 * q + 1], f[4 * q + 2], f[4 * q + 3]);
}

cudaError_t launch_features(const RegionArgs &a, const float4 *simf, const unsigned long long *prev_trace, float *X,
                            cudaStream_t st)
{
    if (a.total == 0) return cudaSuccess;
    feature_kernel<<<(a.total + 127) / 128, 128, 0, st>>>(a, simf, prev_trace, X);
    return cudaGetLastError();
}

cudaError_t launch_reset(const RegionArgs &a, cudaStream_t st)
{
    if (a.flags) {
        ticket_reset_kernel<<<1, 1, 0, st>>>(a.ctl, a.epoch);
        return cudaGetLastError();
    }
    const unsigned blocks = (a.total + 255) / 256;
    reset_kernel<<<blocks ? blocks : 1, 256, 0, st>>>(a);
    if (a.prio && a.n_seed > 0) {
        seed_count_kernel<<<(a.n_seed + 255) / 256, 256, 0, st>>>(a);
        seed_kernel<<<(a.n_seed + 255) / 256, 256, 0, st>>>(a);
    }
    return cudaGetLastError();
}

static const void *region_fn(int threads, int B)
{
    const bool b16 = B == 16;
    if (B != 4 && B != 8 && B != 16) return nullptr;
    switch (threads) {
#define SP_REGION(NW) \
    case NW:          \
        return b16 ? (const void *)region_kernel<NW, 16> : (const void *)region_kernel<NW, 0>;
        SP_REGION(64)
        SP_REGION(128)
        SP_REGION(256)
        SP_REGION(320)
        SP_REGION(384)
        SP_REGION(480)
        SP_REGION(512)
        SP_REGION(768)
#undef SP_REGION
    default:
        return nullptr;
    }
}

// threads = worker threads per region (its manager warp comes on top)
cudaError_t region_config(int threads, int B, int imp_units, RegionConfig *c)
{
    *c = RegionConfig();
    const void *f = region_fn(threads, B);
    if (!f) return cudaErrorInvalidValue;
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    // the number of regions per CTA that leaves the most of them on an SM
    for (int g = 1; g <= region_max_groups(threads); ++g) {
        const size_t smem = sizeof(TablesDev) + (size_t)imp_units * sizeof(unsigned short) + g * region_group_bytes(B);
        if (smem + fa.sharedSizeBytes > 227 * 1024) break;
        int ctas = 0;
        e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, f, g * (threads + 32) + region_reporter(threads), smem);
        if (e != cudaSuccess) return e;
        if (ctas * g >= c->ctas_per_sm * c->groups) {
            c->groups = g;
            c->ctas_per_sm = ctas;
            c->smem = smem;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_region(const RegionArgs &a, int threads, int B, int groups, size_t smem, int grid, cudaStream_t st)
{
    const void *f = region_fn(threads, B);
    if (!f) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int P = B + 2;
    void *args[2] = {const_cast<RegionArgs *>(&a), &P};
    e = cudaLaunchKernel(f, dim3((unsigned)grid), dim3((unsigned)(groups * (threads + 32) + region_reporter(threads))), args, smem, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_sweep(const float2 *phi_in, float2 *phi_out, float4 *pc, const int n[3],
                         const LevelCoef *coef, int lvl, PhysConst q, cudaStream_t st)
{
    // Planes a block marches through.  A grid of few blocks takes one plane
    // per block (the march is a chain of L2 round trips: 48 x 40 x 36 takes 3.93
    // us a level at eight planes, 1.81 at one), and more as that makes one full
    // wave of resident blocks (64^3: 4.14 us at eight planes, 2.86 at two).
    // Beyond six planes a wave, chunks of four keep the last wave small (150 x
    // 77 x 131: 10.4 us at eight planes, 9.1 at four; 128^3: 11.4 and 10.7),
    // until the waves are so many that the two extra planes a chunk reads weigh
    // more (512 x 512 x 128: 249.5 us at eight, 249.9 at four).
    const dim3 block(32, kSweepY, 1);
    dim3 grid((n[0] + 31) / 32, (n[1] + kSweepY - 1) / kSweepY, 1);
    constexpr long long kWave = 152ll * kSweepPerSm;
    const long long waves = ((long long)grid.x * grid.y * n[2] + kWave - 1) / kWave;
    const int zchunk = waves <= 6 ? (int)waves : waves <= 64 ? 4 : 8;
    grid.z = (n[2] + zchunk - 1) / zchunk;
    sweep_kernel<<<grid, block, 0, st>>>(phi_in, phi_out, pc, n[0], n[1], n[2], zchunk, coef, lvl, q);
    return cudaGetLastError();
}

}  // namespace sp
