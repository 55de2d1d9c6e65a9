// sp_diag.cu -- energy terms and winding numbers of a stored state.
//
// One pass reads the state once (24 B per site) and gives the three energy
// terms and the winding counts; the winding map alone reads phi (8 B) and
// writes three bytes.  A thread marches along z through a chunk of planes with
// the four corners of its cell's face in registers, so a plane costs four
// loads of phi and seven edge tests instead of thirteen loads and twelve tests.
//
// FP64 arithmetic was the bound before (84 % of that pipe, two operations per
// clock and SM: 10.6 ms of energy and 17.3 ms of winding at 512^3).  The edge
// tests are exact in FP32 but for ties (sp_crossing.cuh).  The energy terms are
// kept as sums of three FP32 words: a difference, sum or square of FP32 values
// is a rounded value plus an FP32 error (two-sum, Knuth; two-product by fused
// multiply-add, Dekker), and the errors are summed with their own errors (two
// words measured 1e-15 off, FP64 1e-16; three words are good to 2^-70, below
// the rounding of the FP64 sums that follow).  Warps combine their lanes the
// same way, then one FP64 sum per warp, all in a fixed order (deterministic).
// A thread whose sums leave the range in which FP32 products and their errors
// are exact (tiny, huge, infinite or NaN values) sums its column again in FP64.
#include <cuda_runtime.h>
#include <stdint.h>

#include "sp_crossing.cuh"
#include "sp_device.cuh"
#include "sp_kernels.h"

namespace sp {

namespace {

constexpr int kDiagY = 8, kDiagThreads = 32 * kDiagY;
constexpr int kDiagPlanes = 64;  // most planes of a thread's march

struct DiagArgs {
    const float2 *phi;
    const float4 *pc;
    int nx, ny, nz, zc;
    int flat;  // a block's threads are consecutive sites of a plane, not a 32 x 8 tile
    double eta2;
    float eta_w[3];  // eta^2 = eta_w[0] + [1] + [2], rounded words
    int fast;        // eta^2 in the range of the FP32 pairs
    double *energy;  // per block: kinetic, gradient, potential sums (no factors), each [blocks]
    long long *count;  // per block: pierced by normal axis, sum |w|, sum w by normal axis, each [blocks]
    signed char *map;  // [3][sites], or unused
};

__device__ __forceinline__ float two_sum(float a, float b, float &err)
{
    const float s = a + b, bb = s - a;
    err = (a - (s - bb)) + (b - bb);
    return s;
}

__device__ __forceinline__ float2 neg2(float2 a) { return __fmul2_rn(make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(make_float2(-1.0f, -1.0f), b, a); }

// a + b and its error, both parts at once
__device__ __forceinline__ float2 two_sum2(float2 a, float2 b, float2 &err)
{
    const float2 s = __fadd2_rn(a, b), bb = sub2(s, a);
    err = __fadd2_rn(sub2(a, sub2(s, bb)), sub2(b, bb));
    return s;
}

// A running sum of three words.
struct Sum3 {
    float2 s, e, g;
    __device__ __forceinline__ void add(float2 h, float2 t, float2 tiny)  // h + t + tiny, each far below the last
    {
        float2 e1, e2, e3;
        s = two_sum2(s, h, e1);
        e = two_sum2(e, two_sum2(e1, t, e2), e3);
        g = __fadd2_rn(g, __fadd2_rn(__fadd2_rn(e2, e3), tiny));
    }
};

// d^2 into a running sum
__device__ __forceinline__ void add_square(Sum3 &acc, float2 d)
{
    const float2 h = __fmul2_rn(d, d);
    acc.add(h, __ffma2_rn(d, d, neg2(h)), make_float2(0.0f, 0.0f));
}

// (d + e)^2 into a running sum, e the error of d: d^2 + 2 d e + e^2
__device__ __forceinline__ void add_square(Sum3 &acc, float2 d, float2 e)
{
    const float2 h = __fmul2_rn(d, d), l = __ffma2_rn(d, d, neg2(h));
    const float2 d2 = __fadd2_rn(d, d), p = __fmul2_rn(d2, e);
    float2 tiny;
    const float2 t = two_sum2(l, p, tiny);
    acc.add(h, t, __fadd2_rn(tiny, __ffma2_rn(e, e, __ffma2_rn(d2, e, neg2(p)))));
}

// |phi|^2 - eta^2 as a rounded value, its error and the error of that
__device__ __forceinline__ float off_vacuum(float2 f, const float *eta_w, float &low, float &lower)
{
    const float hr = f.x * f.x, hi = f.y * f.y;
    const float lr = __fmaf_rn(f.x, f.x, -hr), li = __fmaf_rn(f.y, f.y, -hi);
    float a1, a2, c1, c2, c3, c4, m;
    const float s2 = two_sum(two_sum(hr, hi, a1), -eta_w[0], a2);
    const float b1 = two_sum(lr, li, c1), b2 = two_sum(a1, a2, c2);
    const float b4 = two_sum(b2, two_sum(b1, -eta_w[1], c3), c4);
    const float t = two_sum(s2, b4, m);
    float r1;
    const float r = two_sum(m, ((c1 + c2) + (c3 + c4)) - eta_w[2], r1);
    const float v = t + r;
    const float w = r - (v - t);  // |r| is at most an ulp of t unless t is zero: exact
    low = w + r1;
    lower = r1 - (low - w);
    return v;
}

__device__ __forceinline__ unsigned bits_of(float2 a) { return __float_as_uint(a.x) | __float_as_uint(a.y); }

// Whether a sum of squares is one the FP32 pairs give: finite and not so small
// that errors fell below the FP32 range (unless every value was zero).
__device__ __forceinline__ bool in_range(float s, float e, unsigned bits)
{
    return s < 0x1p100f && fabsf(e) < 0x1p100f && (s >= 0x1p-80f || (bits & 0x7fffffffu) == 0);
}

// The same sums of one column in FP64.
__device__ __noinline__ void column_fp64(const DiagArgs &a, unsigned oa, unsigned ob, unsigned od, int z0, int z1,
                                         double *out)
{
    const size_t plane = (size_t)a.nx * a.ny;
    double kin = 0.0, grad = 0.0, pot = 0.0;
    for (int z = z0; z < z1; ++z) {
        const float2 *p = a.phi + plane * (size_t)z, *pn = a.phi + plane * (size_t)(z + 1 == a.nz ? 0 : z + 1);
        const float4 v = a.pc[plane * (size_t)z + oa];
        const float2 f = p[oa];
        const double fr = f.x, fi = f.y;
        kin = __dadd_rn(kin, __dadd_rn(__dmul_rn((double)v.x, (double)v.x), __dmul_rn((double)v.y, (double)v.y)));
        const float2 nb[3] = {p[ob], p[od], pn[oa]};
        for (int k = 0; k < 3; ++k) {
            const double dr = __dsub_rn((double)nb[k].x, fr), di = __dsub_rn((double)nb[k].y, fi);
            grad = __dadd_rn(grad, __dadd_rn(__dmul_rn(dr, dr), __dmul_rn(di, di)));
        }
        const double m2 = __dsub_rn(__dadd_rn(__dmul_rn(fr, fr), __dmul_rn(fi, fi)), a.eta2);
        pot = __dadd_rn(pot, __dmul_rn(m2, m2));
    }
    out[0] = kin;
    out[1] = grad;
    out[2] = pot;
}

// ENERGY: energy sums and winding counts; else the winding map.  Bound by
// instruction issue (485 a site with the energies; 64 % of issue slots before,
// and 3.3 of 5.0 stall cycles on loads, which the step-ahead loads hide): 2.26
// ms at 512^3, 2.56 without the loads ahead, 2.40 at four blocks per SM (64
// registers, spilling).
template <bool ENERGY>
__global__ void __launch_bounds__(kDiagThreads, 3) diag_kernel(const DiagArgs a)
{
    __shared__ double s_en[kDiagY][3];
    __shared__ int s_cnt[kDiagY][7];
    int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * kDiagY + threadIdx.y;
    if (a.flat) {
        x += (int)(blockIdx.x * (kDiagThreads - 32) + threadIdx.y * 32);
        y = x / a.nx;
        x -= y * a.nx;
    }
    const int z0 = blockIdx.z * a.zc, z1 = min(z0 + a.zc, a.nz);
    const size_t plane = (size_t)a.nx * a.ny;
    const size_t sites = plane * a.nz;
    const bool inside = x < a.nx && y < a.ny;
    int cnt[7] = {0, 0, 0, 0, 0, 0, 0};
    Sum3 kin = {}, grad = {};
    float ps = 0.0f, pe = 0.0f, pg = 0.0f;
    unsigned kin_bits = 0, grad_bits = 0, pot_bits = 0;
    double en[3] = {0.0, 0.0, 0.0};
    bool slow = false;
    if (inside) {
        const int x1 = x + 1 == a.nx ? 0 : x + 1, y1 = y + 1 == a.ny ? 0 : y + 1;
        const unsigned ya = (unsigned)y * (unsigned)a.nx, yd = (unsigned)y1 * (unsigned)a.nx;
        const unsigned oa = ya + x, ob = ya + x1, oc = yd + x1, od = yd + x;
        const float2 *p = a.phi + plane * (size_t)z0;
        float2 A = __ldg(p + oa), B = __ldg(p + ob), C = __ldg(p + oc), D = __ldg(p + od);
        int ab = crossing(A, B), ad = crossing(A, D), bc = crossing(B, C), dc = crossing(D, C);
        // the next plane's corners and this plane's (pi, c), a step ahead
        p = a.phi + plane * (size_t)(z0 + 1 == a.nz ? 0 : z0 + 1);
        float2 An = __ldg(p + oa), Bn = __ldg(p + ob), Cn = __ldg(p + oc), Dn = __ldg(p + od);
        float4 vn = {};
        if (ENERGY) vn = __ldg(a.pc + plane * (size_t)z0 + oa);
        for (int z = z0; z < z1; ++z) {
            const float2 A1 = An, B1 = Bn, C1 = Cn, D1 = Dn;
            const float4 v = vn;
            if (z + 1 < z1) {
                p = a.phi + plane * (size_t)(z + 2 == a.nz ? 0 : z + 2);
                An = __ldg(p + oa), Bn = __ldg(p + ob), Cn = __ldg(p + oc), Dn = __ldg(p + od);
                if (ENERGY) vn = __ldg(a.pc + plane * (size_t)(z + 1) + oa);
            }
            if (ENERGY) {
                const float2 pi = make_float2(v.x, v.y);
                add_square(kin, pi);
                kin_bits |= bits_of(pi);
                const float2 nA = neg2(A);
                float2 e;
                float2 d = two_sum2(B, nA, e);
                add_square(grad, d, e);
                grad_bits |= bits_of(d);
                d = two_sum2(D, nA, e);
                add_square(grad, d, e);
                grad_bits |= bits_of(d);
                d = two_sum2(A1, nA, e);
                add_square(grad, d, e);
                grad_bits |= bits_of(d);
                float low, lower, e1, e2, e3, e4;
                const float m = off_vacuum(A, a.eta_w, low, lower);
                const float h = m * m, m2 = m + m, q = m2 * low;
                const float l = two_sum(__fmaf_rn(m, m, -h), q, e1);
                e1 += __fmaf_rn(low, low, __fmaf_rn(m2, lower, __fmaf_rn(m2, low, -q)));
                ps = two_sum(ps, h, e2);
                pe = two_sum(pe, two_sum(e2, l, e3), e4);
                pg += (e3 + e4) + e1;
                pot_bits |= __float_as_uint(m);
            }
            bool unsure = false;
            int ab1 = crossing_fp32(A1, B1, unsure), ad1 = crossing_fp32(A1, D1, unsure);
            int bc1 = crossing_fp32(B1, C1, unsure), dc1 = crossing_fp32(D1, C1, unsure);
            int va = crossing_fp32(A, A1, unsure), vb = crossing_fp32(B, B1, unsure), vd = crossing_fp32(D, D1, unsure);
            if (unsure) {
                ab1 = crossing(A1, B1), ad1 = crossing(A1, D1), bc1 = crossing(B1, C1), dc1 = crossing(D1, C1);
                va = crossing(A, A1), vb = crossing(B, B1), vd = crossing(D, D1);
            }
            const int w[3] = {ad + vd - ad1 - va, va + ab1 - vb - ab, ab + bc - dc - ad};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                if (ENERGY) {
                    cnt[k] += w[k] != 0;
                    cnt[3] += abs(w[k]);
                    cnt[4 + k] += w[k];
                } else {
                    a.map[k * sites + plane * (size_t)z + oa] = (signed char)w[k];
                }
            }
            A = A1, B = B1, C = C1, D = D1;
            ab = ab1, ad = ad1, bc = bc1, dc = dc1;
        }
        if (ENERGY) {
            const float ks = kin.s.x + kin.s.y, gs = grad.s.x + grad.s.y;
            // without a vacuum value |phi|^2 can fall below the FP32 range and leave
            // m = 0 where phi is not: a zero sum then says nothing
            if (a.eta2 == 0.0) pot_bits = 1u;
            slow = !(a.fast && in_range(ks, kin.e.x + kin.e.y, kin_bits) &&
                     in_range(gs, grad.e.x + grad.e.y, grad_bits) && in_range(ps, pe, pot_bits));
            if (slow) column_fp64(a, oa, ob, od, z0, z1, en);
        }
    }
    if (!ENERGY) return;
    // lanes to one sum of three words per warp
    float s[3], e[3], g[3], e1, e2;
    s[0] = two_sum(kin.s.x, kin.s.y, e1);
    e[0] = two_sum(kin.e.x, kin.e.y, e2);
    e[0] = two_sum(e[0], e1, e1);
    g[0] = (kin.g.x + kin.g.y) + (e1 + e2);
    s[1] = two_sum(grad.s.x, grad.s.y, e1);
    e[1] = two_sum(grad.e.x, grad.e.y, e2);
    e[1] = two_sum(e[1], e1, e1);
    g[1] = (grad.g.x + grad.g.y) + (e1 + e2);
    s[2] = ps, e[2] = pe, g[2] = pg;
    const bool any_slow = __any_sync(~0u, slow);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        if (slow) s[q] = e[q] = g[q] = 0.0f;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {  // lane 0 ends with the sum
            const float so = __shfl_down_sync(~0u, s[q], o), eo = __shfl_down_sync(~0u, e[q], o);
            const float go = __shfl_down_sync(~0u, g[q], o);
            float r1, r2, r3;
            s[q] = two_sum(s[q], so, r1);
            e[q] = two_sum(two_sum(e[q], eo, r2), r1, r3);
            g[q] = (g[q] + go) + (r2 + r3);
        }
        if (any_slow)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) en[q] = __dadd_rn(en[q], __shfl_down_sync(~0u, en[q], o));
        if (threadIdx.x == 0)
            s_en[threadIdx.y][q] = __dadd_rn(__dadd_rn((double)s[q], __dadd_rn((double)e[q], (double)g[q])), en[q]);
    }
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        const int c = __reduce_add_sync(~0u, cnt[k]);
        if (threadIdx.x == 0) s_cnt[threadIdx.y][k] = c;
    }
    __syncthreads();
    const int t = threadIdx.y * 32 + threadIdx.x;
    const size_t blocks = (size_t)gridDim.x * gridDim.y * gridDim.z;
    const size_t b = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    if (t < 3) {
        double v = 0.0;
        for (int k = 0; k < kDiagY; ++k) v = __dadd_rn(v, s_en[k][t]);
        a.energy[t * blocks + b] = v;
    } else if (t >= 32 && t < 39) {
        long long v = 0;
        for (int k = 0; k < kDiagY; ++k) v += s_cnt[k][t - 32];
        a.count[(t - 32) * blocks + b] = v;
    }
}

// Block q sums quantity q over the blocks of the pass, in a fixed order, and
// applies the factor of its term.
__global__ void __launch_bounds__(256)
    diag_final_kernel(const double *__restrict__ energy, const long long *__restrict__ count, int blocks, double inv_dx2,
                      double half_lambda_a2, DiagOut *__restrict__ out)
{
    __shared__ double sd[256];
    __shared__ long long sl[256];
    const int q = blockIdx.x, t = threadIdx.x;
    double d = 0.0;
    long long l = 0;
    if (q < 3)
        for (int b = t; b < blocks; b += 256) d = __dadd_rn(d, energy[(size_t)q * blocks + b]);
    else
        for (int b = t; b < blocks; b += 256) l += count[(size_t)(q - 3) * blocks + b];
    sd[t] = d;
    sl[t] = l;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (t < w) {
            if (q < 3)
                sd[t] = __dadd_rn(sd[t], sd[t + w]);
            else
                sl[t] += sl[t + w];
        }
        __syncthreads();
    }
    if (t != 0) return;
    if (q < 3)
        out->energy[q] = q == 1 ? __dmul_rn(sd[0], inv_dx2) : q == 2 ? __dmul_rn(sd[0], half_lambda_a2) : sd[0];
    else
        out->winding[q - 3] = sl[0];
}

// Rows narrower than a warp would leave its lanes idle, of which a field that
// needs the FP64 sums has none to spare: there a plane's sites go to the threads
// one after the other (4 x 1024 x 1024, us, in tiles / so: 620 / 125, below the FP32
// range 5530 / 1010; 16 x 512 x 512 199 / 124, 1856 / 954).
bool diag_flat(int nx) { return nx < 32; }

dim3 diag_grid(const int n[3], int *zc)
{
    dim3 g((n[0] + 31) / 32, (n[1] + kDiagY - 1) / kDiagY, 1);
    if (diag_flat(n[0])) g = dim3((n[0] * n[1] + kDiagThreads - 1) / kDiagThreads, 1, 1);
    // as many planes a thread as leave four blocks for every SM
    const long long cols = (long long)g.x * g.y;
    long long z = cols * n[2] / (4 * 152);
    z = z < 1 ? 1 : z > kDiagPlanes ? kDiagPlanes : z;
    *zc = (int)z;
    g.z = (n[2] + *zc - 1) / *zc;
    return g;
}

}  // namespace

size_t diag_scratch_bytes(const int n[3])
{
    int zc;
    const dim3 g = diag_grid(n, &zc);
    return 10 * sizeof(double) * (size_t)g.x * g.y * g.z;
}

cudaError_t launch_diag(const float2 *phi, const float4 *pc, const int n[3], double inv_dx2, double eta2,
                        double half_lambda_a2, void *scratch, DiagOut *out, cudaStream_t st)
{
    DiagArgs a = {};
    const dim3 g = diag_grid(n, &a.zc);
    const size_t blocks = (size_t)g.x * g.y * g.z;
    a.phi = phi;
    a.pc = pc;
    a.nx = n[0], a.ny = n[1], a.nz = n[2];
    a.flat = diag_flat(n[0]);
    a.eta2 = eta2;
    a.fast = eta2 == 0.0 || (eta2 >= 0x1p-40 && eta2 <= 0x1p50);
    double r = a.fast ? eta2 : 0.0;
    for (int i = 0; i < 3; ++i) {
        a.eta_w[i] = (float)r;
        r -= (double)a.eta_w[i];
    }
    a.energy = static_cast<double *>(scratch);
    a.count = reinterpret_cast<long long *>(a.energy + 3 * blocks);
    diag_kernel<true><<<g, dim3(32, kDiagY), 0, st>>>(a);
    diag_final_kernel<<<10, 256, 0, st>>>(a.energy, a.count, (int)blocks, inv_dx2, half_lambda_a2, out);
    return cudaGetLastError();
}

cudaError_t launch_winding_map(const float2 *phi, const int n[3], signed char *map, cudaStream_t st)
{
    DiagArgs a = {};
    const dim3 g = diag_grid(n, &a.zc);
    a.phi = phi;
    a.nx = n[0], a.ny = n[1], a.nz = n[2];
    a.flat = diag_flat(n[0]);
    a.map = map;
    diag_kernel<false><<<g, dim3(32, kDiagY), 0, st>>>(a);
    return cudaGetLastError();
}

}  // namespace sp
