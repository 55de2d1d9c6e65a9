// sp_lattice.cu -- the persistent kernel of the 4-cube lattice regions
// (paper Sec. 2, Figs. 2-5; geometry, tables and the in-place data flow in
// lattice.h).
//
// Every region is a translate of one 4-cube of 16 s^4 site-updates over 4s
// levels, whose cells and halo fit a few tens of KB of shared memory (s = 4:
// 1278 phi slots in each of two parity buffers and 878 (pi, c) slots, 34.5
// KB), so several regions run on one SM: as groups of threads of one CTA that
// shares the cell list (lattice_kernel, up to edge 20; five at s = 4), or one
// per CTA (lattice_ring_kernel: edge 24, whose list does not fit, and the worker
// counts and short calls of lattice_ring_faster and lattice_ring_brief).  A region
//   1. waits until its four predecessors (layer L - 1) have reported done,
//   2. copies in the values it does not compute (cp.async: phi of the halo
//      and the whole state of cells entering the region), straight from the
//      state arrays, all at its start and in address order (every one is
//      final by then and stays in place until the region is done; lattice.h),
//      a phi value as the 16-byte pair of sites around it where the pair's
//      other slot may take it,
//   3. evolves level by level in shared memory (the site update of
//      sp_update.h), writing every value another region needs (a per-cell
//      flag of the tables) straight into the state arrays,
//   4. reports done with a release store of its layer number.
// The per-level cell lists and the import list (lattice.h) are the same for
// every region.  A site index follows from the cell's slot and row through the
// row's wrapped y + n1 z, which is refilled for each region, without a branch.
//
// Regions are handed out by ticket in layer order (one atomic per region, taken
// a region ahead).  In lattice_kernel a region's flag is set by a releasing store
// and the next region's flags are read by acquiring loads, both while the next
// region's imports are on their way; in lattice_ring_kernel the flags are read
// early, relaxed, and one fence per region serves as the release of its writes
// and the acquire of those reads.  A ticket's predecessors hold smaller tickets,
// and a group holding a ticket is running or will run it next, so the waits
// always end; each is bounded anyway.  The manager of the paper (Sec. 4) is thus
// reduced to a counter and one flag per region.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "lattice.h"
#include "sp_device.cuh"
#include "sp_kernels.h"

namespace sp {

namespace {

// Per-row record in shared memory (16 bytes): byte offsets, from a cell's phi
// slot, of its y - 1 / y + 1 neighbours (dy: low / high 16 bits, signed) and
// z - 1 / z + 1 neighbours (dz); the byte offset of its (pi, c) slot minus
// 16 x its phi slot; and, for the region being evolved, the row's y + n1 z
// (both wrapped into the grid).
struct alignas(16) LatRow {
    int dy, dz, dpc;
    unsigned yz;
};

// Shared-memory layout of one region (bytes): (pi, c) slots, the two phi
// buffers (an even number of slots each, so that every even slot starts a
// 16-byte pair), the row records and a ring of two levels' cell entries
// (every cp.async16 destination on a 16-byte boundary).
struct LatSmem {
    size_t pc, ph0, ph1, row, ring, total;
    __host__ __device__ LatSmem(int n_slots, int n_foot, int W, int max_cell_n)
    {
        const size_t nb = 8 * (((size_t)n_slots + 1) & ~(size_t)1);
        pc = 0;
        ph0 = 16 * (size_t)n_foot;
        ph1 = ph0 + nb;
        row = ph1 + nb;
        ring = row + 16 * (size_t)W * W;
        total = ring + 2 * 4 * (size_t)max_cell_n;
    }
};

struct LatRegion {
    int sim, L, Labs, tau_b, k_lo, k_hi;
    int c[3];        // centre, cells
    unsigned t, j;   // ticket, region within the layer (all simulations)
    long long id;    // trace / fault-injection id
    int pred[4];     // predecessors' flag indices (-1: none)
};

// Decode ticket t (no waiting).  Returns false when the tickets are exhausted.
__device__ bool lat_decode(const LatArgs &a, unsigned t, int epoch, LatRegion *out)
{
    if (t >= a.total) return false;
    const unsigned li = t / a.per_layer_all;
    const unsigned j = t - li * a.per_layer_all;
    int sim = 0;
    while (sim + 1 < a.n_sims && (long long)j >= a.sims[sim + 1].region_base) ++sim;
    const LatSimDev &sd = a.sims[sim];
    const int idx = (int)((long long)j - sd.region_base);  // < 2^31 regions per layer of one simulation
    LatGeom g;
    g.s = a.s;
    g.M[0] = sd.M[0], g.M[1] = sd.M[1], g.M[2] = sd.M[2];
    const int L = lat_min_layer() + (int)li;
    int ctr[3];
    lat_centre(g, L, idx, ctr);
    LatRegion &r = *out;
    r.sim = sim;
    r.L = L;
    r.Labs = epoch + (int)li;
    r.tau_b = 1 + a.s * L;
    r.k_lo = r.tau_b < 1 ? 1 - r.tau_b : 0;
    r.k_hi = min(a.K - 1, a.T - r.tau_b);
    for (int d = 0; d < 3; ++d) r.c[d] = a.s * ctr[d];
    r.t = t;
    r.j = j;
    r.id = sd.trace_base + (long long)li * sd.per_layer + idx;
    const long long base = (long long)((r.Labs - 1) & 3) * a.per_layer_all + sd.region_base;
    for (int i = 0; i < 4; ++i) r.pred[i] = li > 0 ? (int)(base + lat_pred_of<int>(g, ctr, i)) : -1;
    return true;
}

// Control thread: bounded wait until every predecessor of r has reported done
// (acquire).  False (and the error word set) when a wait gave up or another
// CTA failed.
__device__ bool lat_wait(const LatArgs &a, const LatRegion &r)
{
    const int need = r.Labs - 1;
    const unsigned long long t0 = globaltimer_ns();
    const unsigned long long limit = a.ctl->wait_limit_ns;
    for (int i = 0; i < 4; ++i) {
        if (r.pred[i] < 0) continue;
        unsigned spins = 0;
        while (ld_acquire_gpu(a.flags + r.pred[i]) < need) {
            if ((++spins & 63u) == 0) {
                if (ld_relaxed_gpu(&a.ctl->error) != 0) return false;
                if (globaltimer_ns() - t0 > limit) {
                    if (atomicCAS(&a.ctl->error, 0, (int)kDevTimeout) == 0) a.ctl->error_info = (int)r.t;
                    return false;
                }
            }
            __nanosleep(100);
        }
    }
    return true;
}

// Site index of the cell at x offset rx (plus 2s) in a row with wrapped index
// yz = y + n1 z: x = (centre x - 2s) + rx, wrapped once (branch-free; regions
// are narrower than the grid, so one wrap suffices).
__device__ __forceinline__ unsigned long long lat_site(int rx, unsigned yz, int cx, int n0)
{
    int x = cx + rx;
    x += x < 0 ? n0 : 0;
    x -= x >= n0 ? n0 : 0;
    return (unsigned long long)yz * (unsigned)n0 + (unsigned)x;
}

// A region's imports: the list of all of them (imp_run, in address order),
// loaded in batches, of which a thread loads lat_imp_batch entries before using
// any, so the entry reads overlap in one round of L2 latency: 12 cover a whole
// region of edge 16 with 128 workers (1370 entries), 19 one of edge 20 with 256
// (4609; 240^3, 32 steps 4079 us with 12 in two rounds, 3832 so; 160^3, 4 steps 331
// and 301).  More than a size needs costs code: edge 16 with 20 is 5 % slower.
template <int NW>
__host__ __device__ constexpr int lat_imp_batch()
{
    return NW == 64 ? 6 : NW == 192 ? 8 : NW == 256 ? 19 : 12;
}

// One batch of import entries, i0 + u NW (padding: first level 255).
template <int NW>
__device__ __forceinline__ void load_import_batch(uint2 (&ie)[lat_imp_batch<NW>()], const uint2 *__restrict__ imp_run,
                                                  int n, int i0)
{
#pragma unroll
    for (int u = 0; u < lat_imp_batch<NW>(); ++u)
        ie[u] = i0 + u * NW < n ? __ldg(imp_run + i0 + u * NW) : make_uint2(0u, ~0u);
}

// cp.async of one batch of imports of levels k_lo..k_hi: phi of one level
// into its buffer, and the (pi, c) of full imports.  pair_bit: a phi import
// whose entry has this bit (kLatImpPair for a region that loads nothing else
// into its phi buffers at its start, kLatImpPairRow for one cut by the call's
// first level, lattice.h) and whose slot and site have the same parity copies
// the aligned 16-byte site pair into the aligned slot pair (L2 only): the
// other slot of the pair then receives the same bytes any other load of it
// does, or is written by the region only at a later level, and an 8-byte copy
// would have to allocate in L1.  PAIRS: the list holds the two imports of a
// slot pair as one entry, which then share the copy, the row record and the
// address arithmetic (edge 16 at 240^3: 1.293e11 site-updates/s with an
// entry per import, 1.311e11 so; the test for it costs the sizes without such
// entries 7 %, hence the two forms).
template <int NW, bool PAIRS, int YS>
__device__ __forceinline__ void issue_import_batch(const uint2 (&ie)[lat_imp_batch<NW>()], int k_lo, int k_hi, int cx,
                                                   int n0, const unsigned *s_yz, char *pcb, char *ph0, char *ph1,
                                                   const float2 *g0, const float2 *g1, const float4 *gpc, uint32_t pair_bit,
                                                   bool aligned)
{
#pragma unroll
    for (int u = 0; u < lat_imp_batch<NW>(); ++u) {
        const uint32_t w = ie[u].y;
        if (lat_run_last(w) < k_lo || lat_run_first(w) > k_hi) continue;  // (also the padding)
        const uint32_t e = ie[u].x;
        const int sl = lat_slot(e), row = lat_row(e);
        const bool b = (e & kLatImpBuf) != 0;  // phi buffer (k - 1) & 1; g0 / g1 are its arrays
        const unsigned yz = s_yz[row * YS];
        const unsigned long long g = lat_site(lat_rx2s(e), yz, cx, n0);
        char *dst = (b ? ph1 : ph0) + (sl << 3);
        const float2 *src = (b ? g1 : g0) + g;
        const bool same = aligned && ((sl ^ (int)g) & 1) == 0;  // slot and site parity, and phi on 16 bytes
        const bool both = PAIRS && (w & kLatRunPair);
        if (same && (both || (e & pair_bit)))
            cp_async16(dst - ((sl & 1) << 3), src - (g & 1));
        else
            cp_async8(dst, src);
        char *const pc = pcb + ((sl + lat_run_pc(w)) << 4);
        if (e & kLatImpFull) cp_async16(pc, gpc + g);
        if (both) {
            const unsigned long long g2 = same ? g + 1 : lat_site(lat_rx2s(e) + 1, yz, cx, n0);
            if (!same) cp_async8(dst + 8, (b ? g1 : g0) + g2);
            if (w & kLatRunFull2) cp_async16(pc + 16, gpc + g2);
        }
    }
}

// cp.async of the cell entries of one level (16-byte chunks; lists are padded)
template <int NW>
__device__ __forceinline__ void copy_entries(uint32_t *ring, const uint32_t *__restrict__ tab, int off, int n)
{
    const int n4 = (n + 3) & ~3;
    for (int i = 4 * (int)threadIdx.x; i < n4; i += 4 * NW) cp_async16(ring + i, tab + off + i);
}

__device__ __forceinline__ float2 ld_f2(const char *base, int off) { return *reinterpret_cast<const float2 *>(base + off); }

// ---- the kernel for sizes whose cell list fits shared memory (up to edge 20) ----

// Most threads of a CTA: sets the register budget (64, 102, 68 and 128
// registers for 64, 128, 192 and 256 workers a region).
template <int NW>
constexpr int lat_max_threads()
{
    return NW == 64 ? 1024 : NW == 128 ? 640 : NW == 192 ? 960 : 512;
}

constexpr int kLatMaxGroups = 15;  // one named barrier per region of a CTA, and barrier 0

// Shared memory: of the CTA, the wide cell entries of all levels and the rows'
// first slots; of each of its regions, the (pi, c) slots, the two phi buffers
// (an even number of slots each, so that every even slot starts a 16-byte
// pair) and the rows' wrapped y + n1 z.
struct LatResident {
    size_t row_x0, region, pc, ph0, ph1, yz, stride;
    __host__ __device__ LatResident(int n_cell, int n_slots, int n_foot, int W)
    {
        const size_t nb = 8 * (((size_t)n_slots + 1) & ~(size_t)1), rows = (4 * (size_t)W * W + 15) & ~(size_t)15;
        row_x0 = 8 * (size_t)n_cell;
        region = row_x0 + rows;
        pc = 0;
        ph0 = 16 * (size_t)n_foot;
        ph1 = ph0 + nb;
        yz = ph1 + nb;
        stride = yz + rows;
    }
    __host__ __device__ size_t total(int groups) const { return region + groups * stride; }
};

// The next region of a group: none, its predecessors not all done, ready.
enum { kLatNone, kLatWait, kLatReady };

__device__ __forceinline__ int sext8(uint32_t w, int byte) { return (int)(w << (24 - 8 * byte)) >> 24; }

// A CTA hosts several regions, each a group of NW threads with a barrier of its
// own, which share the cell list: it is read into shared memory once a launch,
// a cell's entry is one coalesced 8-byte read with everything its update needs
// (the kernel with a ring of levels reads a 4-byte entry and, through it, a
// 16-byte row record at a random bank, and copies the list anew for every
// region), and a level waits for nothing but the barrier.  What bounds it at
// edge 16 is the L1 data pipe (76 % busy, 43 wavefronts per 32 site-updates) and
// the five regions that fit an SM: 1.384e11 site-updates/s at 240^3, 1.329e11
// with the ring (1.449e11 since a region follows the one before without a wait); 2, 3 or 2 interleaved cells a step 1.31, 1.30, 1.28e11; 160 or
// 192 workers 1.35, 1.21e11.  Smaller regions gain most, as sharing the list
// fits more of them: edge 12 0.785 to 1.05e11, edge 8 0.361 to 0.536e11.
template <int NW>
__global__ void __launch_bounds__(lat_max_threads<NW>(), 1) lattice_kernel(const LatArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_cell_off[4 * kLatMaxS + 1], s_cell_n[4 * kLatMaxS];
    __shared__ LatRegion s_regs[kLatMaxGroups];
    __shared__ int s_stops[kLatMaxGroups], s_nexts[kLatMaxGroups];
    const int group = threadIdx.x / NW, tid = threadIdx.x - group * NW;
    const int R = 2 * a.s, W = 4 * a.s + 1, WW = W * W;
    const LatResident L(a.n_cell, a.n_slots, a.n_foot, W);
    uint2 *const s_cell = reinterpret_cast<uint2 *>(smem);
    int *const s_row_x0 = reinterpret_cast<int *>(smem + L.row_x0);
    unsigned char *const mine = smem + L.region + (size_t)group * L.stride;
    char *const s_pcb = reinterpret_cast<char *>(mine + L.pc);
    char *const s_ph0 = reinterpret_cast<char *>(mine + L.ph0);
    char *const s_ph1 = reinterpret_cast<char *>(mine + L.ph1);
    unsigned *const s_yz = reinterpret_cast<unsigned *>(mine + L.yz);
    LatRegion &s_reg = s_regs[group];
    volatile int &s_stop = s_stops[group], &s_next = s_nexts[group];
    // the list by asynchronous copies, all on their way at once (an even number of
    // 8-byte entries)
    for (int i = 2 * threadIdx.x; i < a.n_cell; i += 2 * blockDim.x) cp_async16(s_cell + i, a.cell_wide + i);
    cp_async_commit();
    for (int i = threadIdx.x; i < WW; i += blockDim.x) s_row_x0[i] = a.row_x0[i];
    for (int i = threadIdx.x; i <= a.K; i += blockDim.x) {
        s_cell_off[i] = a.cell_off[i];
        if (i < a.K) s_cell_n[i] = a.cell_n[i];
    }
    // The control thread of a region is its last one: cells are dealt out from
    // thread 0, so it has the least evolution work at every level.  Its state:
    // the next ticket and the finished region whose flag is still to be set.  While
    // a region's imports are on their way it sets that flag, decodes the region of
    // the next ticket and, with three other threads of its warp, reads its
    // predecessors' flags; if they are done, which is the rule once a layer has more
    // regions than the GPU holds, the region follows without a wait, a fence or a
    // barrier of its own (with a fence, the flag and the early reads' check between
    // two regions: edge 16 1.390e11 site-updates/s at 240^3, now 1.449e11; edge 8
    // 0.534 and 0.588e11; edge 20 1.121 and 1.205e11, with imports in two rounds).
    const int ctl = NW - 1;
    const bool ctl_warp = tid >= NW - 32;
    unsigned next = 0;
    int epoch = 0;
    int *unset = nullptr, unset_to = 0;  // flag of the finished region
    cp_async_wait_all();
    __syncthreads();  // the shared lists; a region waits only after it: another group of the CTA may hold its predecessor
    const int bar = 1 + group;
    if (tid == ctl) {
        epoch = *(volatile int *)&a.ctl->epoch;
        s_stop = 0;
        // First tickets go round the CTAs, one group of each after the other, so that
        // a small grid's layers spread over the SMs (edge 16, 64 x 64 x 64, 100 steps:
        // 591 us with all groups at once, 486).  A group takes its turn after a
        // few microseconds in any case: only groups that run hold tickets.
        const unsigned turn = (unsigned)group * gridDim.x;
        const unsigned long long t0 = globaltimer_ns();
        while (ld_relaxed_gpu_u(&a.ctl->head) < turn && globaltimer_ns() - t0 < 4000) {}
        const unsigned t = atomicAdd(&a.ctl->head, 1u);
        if (!lat_decode(a, t, epoch, &s_reg) || !lat_wait(a, s_reg)) s_stop = 1;
    }
    named_barrier(bar, NW);
    const int ya = 8 * a.bank_a, zb = 8 * a.bank_b;  // byte steps of the residues
    while (!s_stop) {
        const LatRegion r = s_reg;
        if (tid == ctl) next = atomicAdd(&a.ctl->head, 1u);
        const LatSimDev &sdr = a.sims[r.sim];
        const int n0 = sdr.n[0], cx = r.c[0] - R;
        // the first batch of import entries (their loads overlap the row set-up)
        uint2 ie[lat_imp_batch<NW>()];
        load_import_batch<NW>(ie, a.imp_run, a.n_imp_run, tid);
        // the rows' wrapped y + n1 z for this region (row = (y + 2s) W + z + 2s)
        {
            const int n1 = sdr.n[1], n2 = sdr.n[2];
            const unsigned wdiv = lat_row_div(a.s);
            for (int i = tid; i < WW; i += NW) {
                const int y2s = lat_row_y2s(i, wdiv);
                int y = r.c[1] + y2s - R, z = r.c[2] + (i - y2s * W) - R;
                y += y < 0 ? n1 : 0;
                y -= y >= n1 ? n1 : 0;
                z += z < 0 ? n2 : 0;
                z -= z >= n2 ? n2 : 0;
                s_yz[i] = (unsigned)y + (unsigned)n1 * (unsigned)z;
            }
        }
        const PhysConst q = sdr.q;
        const LevelCoef *__restrict__ coef = sdr.coef;
        float2 *const g_even = sdr.phi0;
        float2 *const g_odd = sdr.phi1;
        float4 *const gpc = sdr.pc;
        unsigned long long t_start = 0;
        if (tid == ctl && a.trace) t_start = globaltimer_ns();
        const int par0 = r.tau_b & 1;  // level k of the region is global parity par0 ^ (k & 1)
        named_barrier(bar, NW);  // row indices written

        // a region cut by the call's first level: its own cells of level k_lo - 1, whole
        if (r.k_lo > 0) {
            const int kb = r.k_lo - 1;
            char *phb = (kb & 1) ? s_ph1 : s_ph0;
            const float2 *gp = (par0 ^ (kb & 1)) ? g_odd : g_even;
            const uint2 *const ent = s_cell + s_cell_off[kb];
            const int n = s_cell_n[kb];
            for (int i = tid; i < n; i += NW) {
                const uint32_t e = ent[i].x;
                const int sl = (int)(e & kLatWideSlotMask), row = (int)((e >> kLatWideRowShift) & kLatRowMask);
                const unsigned long long g = lat_site(sl - s_row_x0[row], s_yz[row], cx, n0);
                cp_async8(phb + (sl << 3), gp + g);
                cp_async16(s_pcb + (sl << 4) + (sext8(e, 3) << 8), gpc + g);
            }
        }
        // every import of the region's levels; buffer b holds values of local
        // levels of parity b, global parity par0 ^ b
        const float2 *const g0 = par0 ? g_odd : g_even, *const g1 = par0 ? g_even : g_odd;
        const uint32_t pair_bit = r.k_lo == 0 ? kLatImpPair : kLatImpPairRow;
        const bool aligned = (((uintptr_t)g_even | (uintptr_t)g_odd) & 15) == 0;  // the caller's phi may not be
        for (int i0 = tid;;) {
            if (a.run_pairs)
                issue_import_batch<NW, true, 1>(ie, r.k_lo, r.k_hi, cx, n0, s_yz, s_pcb, s_ph0, s_ph1, g0, g1, gpc, pair_bit,
                                                   aligned);
            else
                issue_import_batch<NW, false, 1>(ie, r.k_lo, r.k_hi, cx, n0, s_yz, s_pcb, s_ph0, s_ph1, g0, g1, gpc, pair_bit,
                                                   aligned);
            i0 += lat_imp_batch<NW>() * NW;
            if (i0 - tid >= a.n_imp_run) break;
            load_import_batch<NW>(ie, a.imp_run, a.n_imp_run, i0);
        }
        LevelCoef co = coef[r.tau_b + r.k_lo - 1];
        cp_async_commit();
        if (ctl_warp) {
            int more = 0;
            if (tid == ctl) {
                if (unset) st_release_gpu(unset, unset_to);
                unset = nullptr;
                more = lat_decode(a, next, epoch, &s_reg);  // every thread has copied the descriptor
            }
            __syncwarp();  // the descriptor
            more = __shfl_sync(0xffffffffu, more, 31);
            const int p = tid & 31;
            bool ok = true;
            if (more && p < 4 && s_reg.pred[p] >= 0) ok = ld_acquire_gpu(a.flags + s_reg.pred[p]) >= s_reg.Labs - 1;
            ok = __all_sync(0xffffffffu, ok);
            if (tid == ctl) s_next = !more ? kLatNone : ok ? kLatReady : kLatWait;
        }
        cp_async_wait_all();
        named_barrier(bar, NW);
        for (int k = r.k_lo; k <= r.k_hi; ++k) {
            const int odd = k & 1;
            const char *rd = odd ? s_ph0 : s_ph1;
            char *wr = odd ? s_ph1 : s_ph0;
            LevelCoef co_next = co;
            if (k < r.k_hi) co_next = coef[r.tau_b + k];
            float2 *gout = (par0 ^ odd) ? g_odd : g_even;
            const uint32_t exp_phi = k == r.k_hi ? ~0u : kLatWideExpPhi;  // the call's last level: export all
            const uint32_t exp_pc = k == r.k_hi ? ~0u : kLatWideExpPc;
            const int n = s_cell_n[k];
            const uint2 *ent = s_cell + s_cell_off[k];
#pragma unroll 1
            for (int i = tid; i < n; i += NW) {
                const uint2 e = ent[i];
                const int own = (int)(e.x & kLatWideSlotMask) << 3;
                const int pcoff = 2 * own + (sext8(e.x, 3) << 8);
                const float4 v = *reinterpret_cast<const float4 *>(s_pcb + pcoff);
                float2 pi = make_float2(v.x, v.y), cc = make_float2(v.z, v.w);
                const float2 out = site_update(ld_f2(rd, own), ld_f2(rd, own - 8), ld_f2(rd, own + 8),
                                               ld_f2(rd, own - ya + (sext8(e.y, 0) << 7)), ld_f2(rd, own + ya + (sext8(e.y, 1) << 7)),
                                               ld_f2(rd, own - zb + (sext8(e.y, 2) << 7)), ld_f2(rd, own + zb + (sext8(e.y, 3) << 7)),
                                               pi, cc, co, q);
                *reinterpret_cast<float2 *>(wr + own) = out;
                const float4 pcv = make_float4(pi.x, pi.y, cc.x, cc.y);
                *reinterpret_cast<float4 *>(s_pcb + pcoff) = pcv;
                if (e.x & (exp_phi | exp_pc)) {
                    const int row = (int)((e.x >> kLatWideRowShift) & kLatRowMask);
                    const unsigned long long g = lat_site((own >> 3) - s_row_x0[row], s_yz[row], cx, n0);
                    if (e.x & exp_phi) __stcg(gout + g, out);  // L2 only: read by other SMs
                    if (e.x & exp_pc) __stcg(gpc + g, pcv);
                }
            }
            named_barrier(bar, NW);
            co = co_next;
        }
        if (tid == ctl) {
            if (a.trace) {
                a.trace[2 * r.id] = t_start;
                a.trace[2 * r.id + 1] = globaltimer_ns();
            }
            if (r.id != a.fault_drop) {
                unset = a.flags + (size_t)((r.Labs & 3) * a.per_layer_all) + r.j;
                unset_to = r.Labs;
            }
        }
        if (s_next == kLatReady) continue;
        if (tid == ctl) {
            if (unset) st_release_gpu(unset, unset_to);
            unset = nullptr;
            if (s_next == kLatNone || !lat_wait(a, s_reg)) s_stop = 1;
        }
        named_barrier(bar, NW);
    }
}

// ---- the kernel with a region per CTA and a ring of two levels' entries ----
// (a level's cell entries are copied into shared memory a level ahead; a cell's
// neighbours, (pi, c) slot and site index follow from its slot and a 16-byte
// record of its row)

// CTAs per SM the register budget is set for (shared memory allows 5 regions
// of edge 16 per SM, 2 of edge 20; measured at 240^3 with all imports at the
// region's start: 128 workers at 5 per SM 1.226e11 site-updates/s, 160 at 5
// per SM 1.204e11, 192 at 5 per SM (56 registers) 1.182e11, at 4 per SM
// (72 registers) 1.020e11).
template <int NW>
constexpr int lat_min_blocks()
{
    return NW <= 64 ? 8 : NW <= 192 ? 5 : NW <= 256 ? 2 : 1;
}

template <int NW>
__global__ void __launch_bounds__(NW, lat_min_blocks<NW>())
    lattice_ring_kernel(const LatArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_cell_off[4 * kLatMaxS + 1], s_cell_n[4 * kLatMaxS];
    __shared__ LatRegion s_reg;
    __shared__ int s_stop;
    const int tid = threadIdx.x;
    const int R = 2 * a.s, W = 4 * a.s + 1, WW = W * W;
    const int max_cell_n = a.max_cell_n;
    const LatSmem L(a.n_slots, a.n_foot, W, max_cell_n);
    char *s_pcb = reinterpret_cast<char *>(smem + L.pc);
    char *s_ph0 = reinterpret_cast<char *>(smem + L.ph0);
    char *s_ph1 = reinterpret_cast<char *>(smem + L.ph1);
    LatRow *s_row = reinterpret_cast<LatRow *>(smem + L.row);
    uint32_t *s_ring = reinterpret_cast<uint32_t *>(smem + L.ring);
    const uint32_t *__restrict__ g_cell = a.cell;
    if (tid <= a.K) {
        s_cell_off[tid] = a.cell_off[tid];
        if (tid < a.K) s_cell_n[tid] = a.cell_n[tid];
    }
    for (int i = tid; i < WW; i += NW) {
        const uint64_t nb = a.row_nb[i];
        LatRow r;
        r.dy = (lat_dym(nb) * 8 & 0xffff) | (lat_dyp(nb) * 8) << 16;
        r.dz = (lat_dzm(nb) * 8 & 0xffff) | (lat_dzp(nb) * 8) << 16;
        r.dpc = a.row_pc[i] * 16;
        r.yz = 0;
        s_row[i] = r;
    }
    // The control thread is the last one: cells are dealt out from thread 0,
    // so it has the least evolution work at every level.  Its state: the next
    // ticket, and early (relaxed) reads of the flags of the region that
    // ticket names.
    const int ctl = NW - 1;
    unsigned next = 0;
    int epoch = 0;
    int fv[4] = {0, 0, 0, 0};
    bool early = false;
    if (tid == ctl) {
        epoch = *(volatile int *)&a.ctl->epoch;
        s_stop = 0;
        const unsigned t = atomicAdd(&a.ctl->head, 1u);
        if (!lat_decode(a, t, epoch, &s_reg) || !lat_wait(a, s_reg))
            s_stop = 1;
        else
            next = atomicAdd(&a.ctl->head, 1u);
    }
    __syncthreads();
    while (!s_stop) {
        const LatRegion r = s_reg;
        const LatSimDev &sdr = a.sims[r.sim];
        const int n0 = sdr.n[0], cx = r.c[0] - R;
        // the first batch of import entries (their loads overlap the row set-up)
        uint2 ie[lat_imp_batch<NW>()];
        load_import_batch<NW>(ie, a.imp_run, a.n_imp_run, tid);
        // the rows' wrapped y + n1 z for this region (row = (y + 2s) W + z + 2s)
        {
            const int n1 = sdr.n[1], n2 = sdr.n[2];
            const unsigned wdiv = lat_row_div(a.s);
            for (int i = tid; i < WW; i += NW) {
                const int y2s = lat_row_y2s(i, wdiv);
                int y = r.c[1] + y2s - R, z = r.c[2] + (i - y2s * W) - R;
                y += y < 0 ? n1 : 0;
                y -= y >= n1 ? n1 : 0;
                z += z < 0 ? n2 : 0;
                z -= z >= n2 ? n2 : 0;
                s_row[i].yz = (unsigned)y + (unsigned)n1 * (unsigned)z;
            }
        }
        const PhysConst q = sdr.q;
        const LevelCoef *__restrict__ coef = sdr.coef;
        float2 *const g_even = sdr.phi0;
        float2 *const g_odd = sdr.phi1;
        float4 *const gpc = sdr.pc;
        unsigned long long t_start = 0;
        if (tid == ctl && a.trace) t_start = globaltimer_ns();
        const int par0 = r.tau_b & 1;  // level k of the region is global parity par0 ^ (k & 1)
        __syncthreads();  // row indices written

        // a region cut by the call's first level: its own cells of level k_lo - 1, whole
        if (r.k_lo > 0) {
            const int kb = r.k_lo - 1;
            char *phb = (kb & 1) ? s_ph1 : s_ph0;
            const float2 *gp = (par0 ^ (kb & 1)) ? g_odd : g_even;
            const int off = s_cell_off[kb], n = s_cell_n[kb];
            for (int i = tid; i < n; i += NW) {
                const uint32_t e = __ldg(g_cell + off + i);
                const int sl = lat_slot(e), row = lat_row(e);
                const LatRow rr = s_row[row];
                const unsigned long long g = lat_site(lat_rx2s(e), rr.yz, cx, n0);
                cp_async8(phb + (sl << 3), gp + g);
                cp_async16(s_pcb + (sl << 4) + rr.dpc, gpc + g);
            }
        }
        copy_entries<NW>(s_ring + (r.k_lo & 1) * max_cell_n, g_cell, s_cell_off[r.k_lo], s_cell_n[r.k_lo]);
        // every import of the region's levels; buffer b holds values of local
        // levels of parity b, global parity par0 ^ b
        for (int i0 = tid;;) {
            const float2 *const g0 = par0 ? g_odd : g_even, *const g1 = par0 ? g_even : g_odd;
            const uint32_t pair_bit = r.k_lo == 0 ? kLatImpPair : kLatImpPairRow;
            const bool aligned = (((uintptr_t)g_even | (uintptr_t)g_odd) & 15) == 0;  // the caller's phi may not be
            if (a.run_pairs)
                issue_import_batch<NW, true, 4>(ie, r.k_lo, r.k_hi, cx, n0, &s_row->yz, s_pcb, s_ph0, s_ph1, g0, g1, gpc, pair_bit,
                                                   aligned);
            else
                issue_import_batch<NW, false, 4>(ie, r.k_lo, r.k_hi, cx, n0, &s_row->yz, s_pcb, s_ph0, s_ph1, g0, g1, gpc, pair_bit,
                                                   aligned);
            i0 += lat_imp_batch<NW>() * NW;
            if (i0 >= a.n_imp_run) break;
            load_import_batch<NW>(ie, a.imp_run, a.n_imp_run, i0);
        }
        LevelCoef co = coef[r.tau_b + r.k_lo - 1];
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        for (int k = r.k_lo; k <= r.k_hi; ++k) {
            const int odd = k & 1;
            const char *rd = odd ? s_ph0 : s_ph1;
            char *wr = odd ? s_ph1 : s_ph0;
            LevelCoef co_next = co;
            if (k < r.k_hi) {
                // the cell entries of level k + 1
                copy_entries<NW>(s_ring + ((k + 1) & 1) * max_cell_n, g_cell, s_cell_off[k + 1], s_cell_n[k + 1]);
                cp_async_commit();
                co_next = coef[r.tau_b + k];
            }
            if (tid == ctl && k == r.k_lo) {
                // every thread has copied the descriptor: decode the next
                // region into it and read its predecessors' flags early
                early = lat_decode(a, next, epoch, &s_reg);
                if (early)
                    for (int i = 0; i < 4; ++i)
                        fv[i] = s_reg.pred[i] >= 0 ? ld_relaxed_gpu(a.flags + s_reg.pred[i]) : 0x7fffffff;
            }
            float2 *gout = (par0 ^ odd) ? g_odd : g_even;
            const uint32_t exp_phi = k == r.k_hi ? ~0u : kLatExpPhi;  // the call's last level: export all
            const uint32_t exp_pc = k == r.k_hi ? ~0u : kLatExpPc;
            const int n = s_cell_n[k];
            const uint32_t *ent = s_ring + odd * max_cell_n;
#pragma unroll 1  // measured: unrolling 2, 3 or 4 cells per step is slower
            for (int i = tid; i < n; i += NW) {
                const uint32_t e = ent[i];
                const int sl = lat_slot(e), row = lat_row(e);
                const LatRow rr = s_row[row];
                const int own = sl << 3;
                const int pcoff = (sl << 4) + rr.dpc;
                const float4 v = *reinterpret_cast<const float4 *>(s_pcb + pcoff);
                float2 pi = make_float2(v.x, v.y), cc = make_float2(v.z, v.w);
                const float2 out = site_update(ld_f2(rd, own), ld_f2(rd, own - 8), ld_f2(rd, own + 8),
                                               ld_f2(rd, own + (int)(short)rr.dy), ld_f2(rd, own + (rr.dy >> 16)),
                                               ld_f2(rd, own + (int)(short)rr.dz), ld_f2(rd, own + (rr.dz >> 16)), pi,
                                               cc, co, q);
                *reinterpret_cast<float2 *>(wr + own) = out;
                const float4 pcv = make_float4(pi.x, pi.y, cc.x, cc.y);
                *reinterpret_cast<float4 *>(s_pcb + pcoff) = pcv;
                if (e & (exp_phi | exp_pc)) {
                    const unsigned long long g = lat_site(lat_rx2s(e), rr.yz, cx, n0);
                    if (e & exp_phi) __stcg(gout + g, out);  // L2 only: read by other SMs
                    if (e & exp_pc) __stcg(gpc + g, pcv);
                }
            }
            cp_async_wait_all();
            __syncthreads();
            co = co_next;
        }
        if (tid == ctl) {
            if (a.trace) {
                a.trace[2 * r.id] = t_start;
                a.trace[2 * r.id + 1] = globaltimer_ns();
            }
            // One fence: release of this region's writes (made before the
            // barrier above by every thread) to the flag store after it, and
            // acquire for the early flag reads before it.
            fence_acq_rel_gpu();
            if (r.id != a.fault_drop) st_relaxed_gpu(a.flags + (size_t)((r.Labs & 3) * a.per_layer_all) + r.j, r.Labs);
            if (!early) {
                s_stop = 1;
            } else {
                const int need = s_reg.Labs - 1;
                bool ready = true;
                for (int i = 0; i < 4; ++i) ready = ready && fv[i] >= need;
                if (!ready && !lat_wait(a, s_reg)) s_stop = 1;
                if (!s_stop) next = atomicAdd(&a.ctl->head, 1u);
            }
        }
        __syncthreads();
    }
}

// Before every lattice call: a fresh ticket counter and error word, and the
// call's layers numbered above every done flag written before.
__global__ void lattice_reset_kernel(Ctl *ctl, int layers)
{
    ctl->head = 0;
    ctl->error = 0;
    ctl->error_info = 0;
    lat_next_epoch(&ctl->last_layer, layers, &ctl->epoch);
}

// The kernel of a size: resident list (several regions per CTA) or the ring.
const void *lattice_fn(int threads, bool resident)
{
    switch (threads) {
#define SP_LAT(NW) \
    case NW:       \
        return resident ? (const void *)lattice_kernel<NW> : (const void *)lattice_ring_kernel<NW>;
        SP_LAT(64)
        SP_LAT(128)
        SP_LAT(192)
        SP_LAT(256)
        SP_LAT(512)
#undef SP_LAT
    default:
        return nullptr;
    }
}

int lattice_max_groups(int threads)
{
    const int t = threads == 64    ? lat_max_threads<64>()
                  : threads == 128 ? lat_max_threads<128>()
                  : threads == 192 ? lat_max_threads<192>()
                  : threads == 256 ? lat_max_threads<256>()
                                   : lat_max_threads<512>();
    return std::min(kLatMaxGroups, t / threads);
}

}  // namespace

bool lattice_valid_threads(int threads) { return lattice_fn(threads, false) != nullptr; }

// Whether a region per CTA with a ring of levels is the faster kernel although
// the whole list fits: 64 workers at edges 16 and 20, whose 64 registers (16
// regions of 64 threads would have to fit) cost the resident kernel more than the
// shared list gives, at edge 12 up to 12 regions of a layer per SM, and 192 at edge 20,
// where the list leaves room for two regions instead of three (32 steps, us,
// resident / ring: edge 16, 64 workers, 128^3 728 / 641, 240^3 4601 / 4176; edge
// 20, 64 workers, 160^3 2531 / 2229, 192 workers 1514 / 1441; edge 12, 64 workers,
// 48^3 260 / 238, 84^3, 91 steps 799 / 703, 240^3 4350 / 4939).  None of them is a
// default.
bool lattice_ring_faster(int s, int threads, bool few)
{
    return (threads == 64 && (s >= 4 || (s == 3 && few))) || (threads == 192 && s >= 5);
}

// The same for a call of few steps with 64 (s = 3: 128) workers: where a layer's
// regions about fit the SMs, more of them are resident as CTAs of their own, and
// no group waits its turn for a first ticket (resident / ring, us: edge 4, 32^3, 1
// step 63 / 59, 8 steps 128 / 125; edge 8, 64^3, 1 step 69 / 63, 4 steps 87 / 82,
// 8 steps 116 / 114, 56^3, 8 steps 106 / 95, 48^3, 6 steps 84 / 84, 16^3, 4 steps 49 / 58; edge 12, 72^3, 1 step 66 / 59, 8 steps
// 102 / 97, 16 steps 144 / 139, 24^3, 8 steps 64 / 68, 96^3, 3 steps 104 / 98, 16
// steps 237 / 242; beyond 14 regions per SM edge 4, 240^3 64 / 86 ms in 32 steps).
bool lattice_ring_brief(int s, long long n_steps, long long per_layer, int sms)
{
    if (per_layer > 14ll * sms) return false;
    if (s == 1) return n_steps <= 8;
    if (per_layer <= 2ll * sms) return false;
    return s == 2 ? n_steps <= (per_layer <= 6ll * sms ? 4 : 8) : s == 3 && n_steps <= (per_layer <= 7ll * sms ? 16 : 8);
}

cudaError_t lattice_config(const LatticeTables &t, int threads, bool ring, LatConfig *c)
{
    *c = LatConfig();
    if (!lattice_valid_threads(threads)) return cudaErrorInvalidValue;
    constexpr size_t kMost = 227 * 1024 - 2048;  // dynamic: the static arrays take up to 2 KB
    const bool resident = !t.cell_wide.empty() && !ring;
    const LatResident L((int)t.cell.size(), t.n_slots, t.n_foot, t.rb_side);
    const void *f = lattice_fn(threads, resident);
    // the number of regions per CTA that leaves the most of them on an SM
    for (int g = 1; g <= (resident ? lattice_max_groups(threads) : 1); ++g) {
        const size_t smem = resident ? L.total(g) : LatSmem(t.n_slots, t.n_foot, t.rb_side, t.max_cell_n).total;
        if (smem > kMost) break;
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int ctas = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, f, threads * g, smem);
        if (e != cudaSuccess) return e;
        if (ctas * g >= c->ctas_per_sm * c->groups) {
            c->resident = resident;
            c->groups = g;
            c->smem = smem;
            c->ctas_per_sm = ctas;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_lattice_reset(Ctl *ctl, int layers, cudaStream_t st)
{
    lattice_reset_kernel<<<1, 1, 0, st>>>(ctl, layers);
    return cudaGetLastError();
}

cudaError_t launch_lattice(const LatArgs &a, int threads, size_t smem, int grid, cudaStream_t st)
{
    const void *f = lattice_fn(threads, a.cell_wide != nullptr);
    if (!f) return cudaErrorInvalidValue;
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    void *args[1] = {const_cast<LatArgs *>(&a)};
    e = cudaLaunchKernel(f, dim3((unsigned)grid), dim3((unsigned)(threads * a.groups)), args, smem, st);
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace sp
