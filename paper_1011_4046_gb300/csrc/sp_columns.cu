// sp_columns.cu -- two levels of the whole-grid sweep in one pass over memory.
//
// What bounds it: DRAM.  One level at a time moves 48 B per site-update (24
// read, 24 written); two levels a pass read and write the state half as often,
// 24 B per site-update and a little for the halo rows that miss L2 (measured
// 25.5 B).  At 512^3 a pass takes 1.08 ms (2.50e11 site-updates/s, 6.4 TB/s
// of DRAM traffic, 0.94 of the measured copy rate) against 2 x 1.02 ms for
// two one-level passes (1.32e11).
//
// A CTA owns a tile of 60 x 26 columns and marches along z through a chunk of
// planes.  It reads the state with a halo of two cells around the tile (the
// domain of dependence of two levels), so tiles need nothing from each other
// during a pass and write to a second copy of the state.  At step p it takes
// in plane p, computes level 1 of plane p - 1 and level 2 of plane p - 2: the
// z neighbour above is always the value computed just before, and one barrier
// per plane orders everything else.
//
// A warp holds two rows of 64 sites, two sites of each row per lane.  Of level
// 1 a thread keeps the planes p - 1 .. p - 3 of phi and p - 1, p - 2 of (pi, c)
// in registers; x neighbours come by shuffles, the rows above and below the
// warp's two through shared memory.  Input planes arrive by cp.async two steps
// ahead.  Why this tile: 15 warps of two rows use 124 registers a thread and
// 200 KB of shared memory, one CTA per SM; at 512^3 other shapes measured
// 1.12 ms (32 rows), 1.13 (two CTAs of 16 rows), 1.18 (24), 1.23 (24 rows, one
// row per warp).  Three and four levels a pass move less but spill or leave
// too few warps for the longer chain: 1.63 ms (three levels, 2.47e11) and 2.44
// ms (four levels, 2.20e11).
#include <cuda_runtime.h>
#include <stdint.h>

#include "sp_device.cuh"
#include "sp_kernels.h"

namespace sp {

namespace {

constexpr int kColRows = 30;                // rows of a tile with its halo
constexpr int kColWarps = kColRows / 2;     // two rows per warp
constexpr int kColHalo = 2;                 // one cell per level
constexpr int kColX = 64 - 2 * kColHalo;    // own columns of a tile along x
constexpr int kColY = kColRows - 2 * kColHalo;
constexpr int kColAhead = 2;                // planes requested ahead of the march
constexpr int kColPhiSlots = kColAhead + 3; // in flight, and planes p, p - 1, p - 2
constexpr int kColPcSlots = kColAhead + 1;
constexpr int kRowB = 64 * 8;               // bytes of a row of phi
constexpr int kPlaneB = kColRows * kRowB;   // a plane of phi; (pi, c) takes twice as much
// shared memory: a row before the first (read by lanes whose result is halo),
// the phi slots, two level-1 planes, the (pi, c) slots
constexpr size_t kColSmem = kRowB + (size_t)(kColPhiSlots + 2 + 2 * kColPcSlots) * kPlaneB;
constexpr int kColSlots = 4;                // planes whose registers a step touches

struct ColArgs {
    const float2 *phi_in;
    const float4 *pc_in;
    float2 *phi_out;
    float4 *pc_out;
    const LevelCoef *coef;  // of the pass's first level
    PhysConst q;
    int nx, ny, nz;
    int vx, vy, zc;  // own columns of a tile, planes of a chunk
    int vec;         // a lane's two sites are one aligned pair of phi and of (pi, c)
};

__device__ __forceinline__ int wrap_mod(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// (pi, c) of two neighbouring sites, 32-byte aligned
__device__ __forceinline__ void store_pair(float4 *p, float4 u, float4 v)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(u.x), "f"(u.y), "f"(u.z),
                 "f"(u.w), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                 : "memory");
}

struct Pair {  // a lane's two sites of a row
    float2 a, b;
};

__device__ __forceinline__ Pair load_pair(const char *s)
{
    const float4 v = *reinterpret_cast<const float4 *>(s);
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

// One level of a row: mid and its six neighbours, (pi, c) updated in place.
__device__ __forceinline__ Pair update_pair(const Pair &mid, const Pair &ym, const Pair &yp, const Pair &zm, const Pair &zp,
                                            float4 &p0, float4 &p1, const LevelCoef &co, const PhysConst &q)
{
    const float2 xl = make_float2(__shfl_up_sync(~0u, mid.b.x, 1), __shfl_up_sync(~0u, mid.b.y, 1));
    const float2 xr = make_float2(__shfl_down_sync(~0u, mid.a.x, 1), __shfl_down_sync(~0u, mid.a.y, 1));
    float2 pi0 = make_float2(p0.x, p0.y), c0 = make_float2(p0.z, p0.w);
    float2 pi1 = make_float2(p1.x, p1.y), c1 = make_float2(p1.z, p1.w);
    const Pair out = {site_update(mid.a, xl, mid.b, ym.a, yp.a, zm.a, zp.a, pi0, c0, co, q),
                      site_update(mid.b, mid.a, xr, ym.b, yp.b, zm.b, zp.b, pi1, c1, co, q)};
    p0 = make_float4(pi0.x, pi0.y, c0.x, c0.y);
    p1 = make_float4(pi1.x, pi1.y, c1.x, c1.y);
    return out;
}

__global__ void __launch_bounds__(32 * kColWarps, 1) column_kernel(const ColArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ LevelCoef s_coef[2];
    const int lane = threadIdx.x, row = 2 * threadIdx.y;
    char *const phi_ring = reinterpret_cast<char *>(smem) + kRowB;
    char *const lev = phi_ring + kColPhiSlots * kPlaneB;
    char *const pc_ring = lev + 2 * kPlaneB;
    const int own = row * kRowB + lane * 16;
    if (row == 0 && lane < 2) s_coef[lane] = a.coef[lane];

    const int x0 = blockIdx.x * a.vx, y0 = blockIdx.y * a.vy, z0 = blockIdx.z * a.zc;
    const int z1 = min(z0 + a.zc, a.nz);
    const int xb = x0 - kColHalo, lx = 2 * lane - kColHalo;
    // site offsets within a plane: of the lane's pair (a, and b = a + db), and
    // of the (pi, c) values it copies (lane and lane + 32 of the row)
    const int xa = wrap_mod(xb + 2 * lane, a.nx), db = wrap_mod(xb + 2 * lane + 1, a.nx) - xa;
    unsigned oa[2], oc[2], od[2];
    bool mine[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const unsigned oy = (unsigned)wrap_mod(y0 - kColHalo + row + j, a.ny) * (unsigned)a.nx;
        oa[j] = oy + (unsigned)xa;
        oc[j] = oy + (unsigned)wrap_mod(xb + lane, a.nx);
        od[j] = oy + (unsigned)wrap_mod(xb + lane + 32, a.nx);
        const int ly = row + j - kColHalo;
        mine[j] = ly >= 0 && ly < a.vy && y0 + ly < a.ny;
    }
    const bool mine_a = lx >= 0 && lx < a.vx && x0 + lx < a.nx;
    const bool mine_b = lx + 1 >= 0 && lx + 1 < a.vx && x0 + lx + 1 < a.nx;
    const size_t plane = (size_t)a.nx * a.ny;
    const PhysConst q = a.q;
    // Site s of a row of (pi, c) sits at position s ^ (bit 3 of s): the copies
    // (consecutive sites) and the reads (every second site) of eight lanes then
    // hit eight different 16-byte bank groups.
    const int pc_w = (lane ^ ((lane >> 3) & 1)) * 16;
    const int pc_r = ((2 * lane) ^ ((lane >> 2) & 1)) * 16;

    // request plane p of phi and plane p - 1 of (pi, c), p = z0 - 2, z0 - 1, ...
    int z_phi = wrap_mod(z0 - kColHalo, a.nz), z_pc = wrap_mod(z0 - kColHalo - 1, a.nz);
    int w_phi = 0, w_pc = 0;
    auto request = [&]() {
        char *f = phi_ring + w_phi * kPlaneB + row * kRowB;
        char *c = pc_ring + w_pc * 2 * kPlaneB + row * 2 * kRowB + pc_w;
        const float2 *gf = a.phi_in + plane * (size_t)z_phi;
        const float4 *gc = a.pc_in + plane * (size_t)z_pc;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            if (a.vec) {
                cp_async16(f + j * kRowB + lane * 16, gf + oa[j]);
            } else {
                cp_async8(f + j * kRowB + lane * 8, gf + oc[j]);
                cp_async8(f + j * kRowB + lane * 8 + kRowB / 2, gf + od[j]);
            }
            cp_async16(c + j * 2 * kRowB, gc + oc[j]);
            cp_async16(c + j * 2 * kRowB + kRowB, gc + od[j]);
        }
        z_pc = z_phi;
        z_phi = z_phi + 1 == a.nz ? 0 : z_phi + 1;
        w_phi = w_phi + 1 == kColPhiSlots ? 0 : w_phi + 1;
        w_pc = w_pc + 1 == kColPcSlots ? 0 : w_pc + 1;
    };

    // Registers of a plane, in slot (p mod 4): level 1 of phi, and (pi, c),
    // which both levels update in place.
    Pair f1[kColSlots][2] = {};
    float4 pc[kColSlots][2][2] = {};
    int p = z0 - kColHalo;
    const int p_end = z1 + kColHalo;
    for (int i = 0; i < kColAhead; ++i) {
        if (p + i < p_end) request();
        cp_async_commit();
    }
    int r_phi = 0, r_pc = 0;
    char *l_rd = lev + own, *l_wr = lev + kPlaneB + own;  // level 1 of planes p - 2 and p - 1
    const char *f_dn = phi_ring + own, *f_mid = f_dn, *f_up = f_dn;  // phi of planes p - 2, p - 1, p
    __syncthreads();
    for (;;) {
#pragma unroll
        for (int r = 0; r < kColSlots; ++r, ++p) {
            if (p >= p_end) return;
            if (p + kColAhead < p_end) request();
            cp_async_commit();
            cp_async_wait_pending(kColAhead);
            __syncwarp();  // lanes read (pi, c) that other lanes of the warp copied
            f_dn = f_mid;
            f_mid = f_up;
            f_up = phi_ring + r_phi * kPlaneB + own;
            r_phi = r_phi + 1 == kColPhiSlots ? 0 : r_phi + 1;
            const char *const c_row = pc_ring + r_pc * 2 * kPlaneB + row * 2 * kRowB;
            r_pc = r_pc + 1 == kColPcSlots ? 0 : r_pc + 1;
            constexpr int M = kColSlots;
            const int s1 = (r + M - 1) % M, s2 = (r + M - 2) % M, s3 = (r + M - 3) % M;  // planes p - 1, p - 2, p - 3
            if (p >= z0) {
                // level 1 of plane p - 1
                const LevelCoef co = s_coef[0];
                Pair ym = load_pair(f_mid - kRowB), mid = load_pair(f_mid);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    const Pair yp = load_pair(f_mid + (j + 1) * kRowB);
                    pc[s1][j][0] = *reinterpret_cast<const float4 *>(c_row + j * 2 * kRowB + pc_r);
                    pc[s1][j][1] = *reinterpret_cast<const float4 *>(c_row + j * 2 * kRowB + (pc_r ^ 16));
                    f1[s1][j] = update_pair(mid, ym, yp, load_pair(f_dn + j * kRowB), load_pair(f_up + j * kRowB),
                                            pc[s1][j][0], pc[s1][j][1], co, q);
                    *reinterpret_cast<float4 *>(l_wr + j * kRowB) =
                        make_float4(f1[s1][j].a.x, f1[s1][j].a.y, f1[s1][j].b.x, f1[s1][j].b.y);
                    ym = mid;
                    mid = yp;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 2; ++j) {  // nothing carried into the march
                    f1[s1][j] = {};
                    pc[s1][j][0] = pc[s1][j][1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
            }
            if (p >= z0 + kColHalo) {
                // level 2 of plane p - 2
                const LevelCoef co = s_coef[1];
                const Pair ym = load_pair(l_rd - kRowB), yp = load_pair(l_rd + 2 * kRowB);
                float2 *const gf = a.phi_out + plane * (size_t)(p - kColHalo);
                float4 *const gc = a.pc_out + plane * (size_t)(p - kColHalo);
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float4 p0 = pc[s2][j][0], p1 = pc[s2][j][1];
                    const Pair u = update_pair(f1[s2][j], j ? f1[s2][0] : ym, j ? yp : f1[s2][1], f1[s3][j], f1[s1][j], p0, p1,
                                               co, q);
                    if (!mine[j]) continue;
                    if (mine_a && mine_b && a.vec) {
                        *reinterpret_cast<float4 *>(gf + oa[j]) = make_float4(u.a.x, u.a.y, u.b.x, u.b.y);
                        store_pair(gc + oa[j], p0, p1);
                    } else {
                        if (mine_a) {
                            gf[oa[j]] = u.a;
                            gc[oa[j]] = p0;
                        }
                        if (mine_b) {
                            gf[(int)oa[j] + db] = u.b;
                            gc[(int)oa[j] + db] = p1;
                        }
                    }
                }
            }
            char *const t = l_rd;
            l_rd = l_wr;
            l_wr = t;
            __syncthreads();
        }
    }
}

}  // namespace

namespace {

// Tiles (of even width, evenly cut) and chunks of planes for a grid.  A chunk
// takes 2 x halo steps more than its planes, and the SMs take the chunks in
// waves; the fewest steps over all waves wins.  Returns those steps.
long long plan_columns(const int n[3], int sm_count, ColArgs *a)
{
    const int tx = (n[0] + kColX - 1) / kColX, ty = (n[1] + kColY - 1) / kColY;
    a->vx = ((n[0] + tx - 1) / tx + 1) & ~1;
    a->vy = (n[1] + ty - 1) / ty;
    const long long tiles = (long long)((n[0] + a->vx - 1) / a->vx) * ((n[1] + a->vy - 1) / a->vy);
    long long best = 0;
    for (int chunks = 1; chunks <= n[2]; ++chunks) {
        const int zc = (n[2] + chunks - 1) / chunks;
        const long long ctas = tiles * ((n[2] + zc - 1) / zc);
        const long long steps = ((ctas + sm_count - 1) / sm_count) * (zc + 2 * kColHalo);
        if (best == 0 || steps < best) best = steps, a->zc = zc;
        if (ctas > 32ll * sm_count) break;
    }
    return best;
}

// Whether a lane's two sites are one aligned pair of phi and of (pi, c).
bool columns_vec(int nx, const void *phi_a, const void *phi_b, const void *pc_a, const void *pc_b)
{
    return (nx & 1) == 0 && (((uintptr_t)phi_a | (uintptr_t)phi_b) & 15) == 0 && (((uintptr_t)pc_a | (uintptr_t)pc_b) & 31) == 0;
}

}  // namespace

// Whether a pass of two levels beats two one-level sweeps.  The pass takes its
// steps over all waves times 1.5 us (1.8 where the rows are no aligned pairs),
// whatever part of a tile the grid fills: a thin grid, one just over a tile's
// width or one of few planes pays for whole tiles and halos (1024 x 4 x 1024: 185
// us, two levels one at a time 68; 20 x 512 x 512: 122 and 99; 137^3: 39 and 33).
// The one-level sweep takes 16 us per 1e6 sites for two levels beyond L2, 11.5
// where part of the state and its phi copy (32 B a site) still hits it, up to half
// as much again where lanes of its 32-wide blocks stay idle, and always wins where
// all of the state hits (128^3: 11.4 us a level against 13.2).  Over 249 grids of
// 2.5e6 to 1e8 sites, sides 4 to 16384, the side it takes is within 2 % of the
// better one (level pairs beyond 2.5e6 sites, whatever the shape: up to 2.7 times
// slower).
bool columns_pay(const float2 *phi, const float4 *pc, const int n[3], int sm_count)
{
    const double sites = (double)n[0] * n[1] * n[2];
    if (sites < 2500000.0) return false;
    ColArgs a = {};
    const double pass = (double)plan_columns(n, sm_count, &a) * (columns_vec(n[0], phi, nullptr, pc, nullptr) ? 1.5 : 1.8);
    const double idle = 1.0 - n[0] / (32.0 * ((n[0] + 31) / 32));
    return pass <= 1e-6 * sites * (sites < 2800000.0 ? 11.5 : 16.0) * (1.0 + 0.5 * idle);
}

cudaError_t launch_columns(const float2 *phi_in, const float4 *pc_in, float2 *phi_out, float4 *pc_out, const int n[3],
                           const LevelCoef *coef, PhysConst q, int sm_count, cudaStream_t st)
{
    ColArgs a{phi_in, pc_in, phi_out, pc_out, coef, q, n[0], n[1], n[2], 0, 0, 0, 0};
    plan_columns(n, sm_count, &a);
    a.vec = columns_vec(n[0], phi_in, phi_out, pc_in, pc_out);
    cudaError_t e = cudaFuncSetAttribute(column_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kColSmem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((n[0] + a.vx - 1) / a.vx), (unsigned)((n[1] + a.vy - 1) / a.vy),
                    (unsigned)((n[2] + a.zc - 1) / a.zc));
    column_kernel<<<grid, dim3(32, kColWarps), kColSmem, st>>>(a);
    return cudaGetLastError();
}

}  // namespace sp
