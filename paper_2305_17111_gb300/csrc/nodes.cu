// Projections of dense event lists through energy nodes.
//
// The single-scatter part of an event's row is a sum of Gaussians in the
// recorded energy, a_j[q] = sum_{p,w} C_p(b_j) omega_{qpw} g(E_j; E'_{qpw}),
// g(E; E') = exp(-(E - E')^2 / (2 sigma^2(E'))), and the projections are
// linear in it, so neither needs the rows themselves.  With the energy axis in
// units of the local resolution, t(E) = 2 sqrt(E) / kappa (sigma = kappa
// sqrt(E)), g is smooth on the scale 1 in both of its arguments, and local
// Lagrange interpolation in each turns the sums into (the idea of the fast
// Gauss transform, Greengard & Strain 1991, with local polynomials):
//
//   forward   D[p][l]  = sum_{q,w} lambda_q omega_{qpw} L_l(E'_{qpw}),
//             DB[b][l] = sum_p C_p(b) D[p][l]                                k_node_spread
//             F[b][k]  = sum_l G[l][k] DB[b][l]                              k_node_values
//             y_j      = sum_k L_k(E_j) F[b_j][k] + unscattered part         k_node_y, k_node_cells
//   back      V[b][k]  = sum_{j in cell b} r_j L_k(E_j)                      k_node_cells
//             VG[b][l] = sum_k G[l][k] V[b][k]                               k_node_unvalues
//             PHI[p][l] = sum_b C_p(b) VG[b][l],
//             out[q]   = sum_{p,w} omega_{qpw} sum_l L_l(E'_{qpw}) PHI[p][l] k_node_gather
//
// per detector angle, with l over the nodes of the scattered energies (16 per
// unit of t, 7 taps), k over those of the recorded energies (8 per unit, 12
// taps) and G[l][k] = g(E_k; E_l).  A path (q, p, w, angle) is visited once per
// projection whatever the number of events, where the rows take one
// exponential per event and path in reach.  Interpolation error of a term,
// relative to the term: 4e-10 (1e-8, 1e-6) for an energy 0 (4, 6) sigma from
// E', below the FP32 rounding of the sums for every energy the lines produce;
// everything is FP32 with fixed-order sums, the voxel sums FP64.
//
// omega = 2^-nlh and E' (sigma = sqrt(log2(e)/2) / sr) come from the path
// tables of the row kernel, so both routes evaluate the same paths.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "lmmew_internal.cuh"

namespace lmmew {
namespace {

constexpr int kTapsL = 7;          // taps of the scattered-energy nodes
constexpr int kPerUnitL = 16;      // nodes per unit of t
constexpr int kTapsK = 12;         // taps of the recorded-energy nodes
constexpr int kPerUnitK = 8;
constexpr double kBandSigmas = 9.0;   // G kept within this many sigma (reach 8 plus the stencils)
constexpr int kSpreadWarpsMax = 4;
constexpr int kStageRows = 16;     // voxels per copy of the spread kernel
constexpr uint32_t kStageBytes = kStageRows * kPC * 4u;   // one component of a stage
constexpr int kGatherThreads = 256;
constexpr int kValueRows = 8;      // (angle, bin) rows per block of k_node_values / _unvalues
constexpr int kCellWarps = 2;

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcpf(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ f32x2 pk1(float v) { return pk(v, v); }

// Two paths' scattered energies on their line's nodes, u = c1 / sr in node
// units: the local index of the first of the 7 taps (clamped into the line's
// nodes) and the distance from the centre tap, in [-1/2, 1/2].  c1 comes in
// two parts and the reciprocal's error is taken out to first order, so the
// distance carries sr's own rounding only (u's rounding would shift a path by
// 4e-6 sigma).  Absent paths (sr = 0) carry weight 0 and land on the last taps.
__device__ __forceinline__ f32x2 node_pos2(float sr0, float sr1, float c1, float c1_lo, int first,
                                           unsigned last, unsigned& i0, unsigned& i1) {
    const float x0 = fmaxf(sr0, 1e-6f), x1 = fmaxf(sr1, 1e-6f);
    const f32x2 r = pk(rcpf(x0), rcpf(x1));
    const f32x2 me = fma2(pk(x0, x1), r, pk1(-1.f));        // x r - 1
    const f32x2 big = fma2(pk1(c1), r, pk1(12582912.f));     // 1.5 2^23: rounds to the nearest integer
    const f32x2 mj = fma2(big, pk1(-1.f), pk1(12582912.f));  // -(nearest node)
    f32x2 s = fma2(pk1(c1), r, mj);
    s = fma2(pk1(c1_lo), r, s);
    s = fma2(mul2(pk1(-c1), r), me, s);
    float b0, b1;
    upk(big, b0, b1);
    i0 = min((unsigned)(__float_as_int(b0) - 0x4B400000 - first), last);
    i1 = min((unsigned)(__float_as_int(b1) - 0x4B400000 - first), last);
    return s;
}

// The 7 Lagrange weights of two paths at distance s, times wt.
__device__ __forceinline__ void lagrange7(f32x2 s, f32x2 wt, f32x2 (&w)[7]) {
    const f32x2 q = mul2(s, s);
    const f32x2 a1 = add2(q, pk1(-1.f)), a2 = add2(q, pk1(-4.f)), a3 = add2(q, pk1(-9.f));
    const f32x2 sw = mul2(s, wt), a12 = mul2(a1, a2);
    const f32x2 m1 = mul2(mul2(sw, mul2(a2, a3)), pk1(1.f / 48.f));
    const f32x2 m2 = mul2(mul2(sw, mul2(a1, a3)), pk1(-1.f / 120.f));
    const f32x2 m3 = mul2(mul2(sw, a12), pk1(1.f / 720.f));
    const f32x2 t1 = mul2(m1, s), t2 = mul2(m2, s), t3 = mul2(m3, s);
    w[3] = mul2(mul2(a12, a3), mul2(wt, pk1(-1.f / 36.f)));
    w[4] = add2(t1, m1);
    w[2] = fma2(m1, pk1(-1.f), t1);
    w[5] = fma2(m2, pk1(2.f), t2);
    w[1] = fma2(m2, pk1(-2.f), t2);
    w[6] = fma2(m3, pk1(3.f), t3);
    w[0] = fma2(m3, pk1(-3.f), t3);
}

// The 12 Lagrange weights at position f in [0, 1) between nodes 5 and 6,
// normalised to sum 1 (their common rounding cancels).
__device__ __forceinline__ void lagrange12(float f, float (&w)[12]) {
    // nodes at +-1/2, +-3/2, .. +-11/2 from the middle, x = f - 1/2;
    // 1 / prod_{j != i} (x_i - x_j) for the pair at +-(i + 1/2)
    constexpr float c[6] = {-1.f / 86400.f, 1.f / 120960.f,   -1.f / 241920.f,
                            1.f / 725760.f, -1.f / 3628800.f, 1.f / 39916800.f};
    const float x = f - 0.5f, q = x * x;
    float a[6], pre[6], suf[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) a[i] = q - (i + 0.5f) * (i + 0.5f);
    pre[0] = 1.f;
    suf[5] = 1.f;
#pragma unroll
    for (int i = 1; i < 6; ++i) pre[i] = pre[i - 1] * a[i - 1];
#pragma unroll
    for (int i = 4; i >= 0; --i) suf[i] = suf[i + 1] * a[i + 1];
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const float m = pre[i] * suf[i] * c[i], n = m * (i + 0.5f);
        w[6 + i] = fmaf(m, x, n);        // node at +(i + 1/2): factor (x + (i + 1/2))
        w[5 - i] = -fmaf(m, x, -n);
        sum += w[6 + i] + w[5 - i];
    }
    const float inv = 1.f / sum;
#pragma unroll
    for (int i = 0; i < 12; ++i) w[i] *= inv;
}

// Position of a recorded energy on its nodes, u = ck sqrt(E): first of its 12
// taps (local index) and the fraction.  ck comes in two parts and the square
// root's rounding is taken out to first order: the fraction is good to its
// own FP32 rounding, where u's would shift the event by 4e-6 sigma.
__device__ __forceinline__ float energy_pos(const NodeConst& N, float e, int* k) {
    const float r = sqrtf(e);
    const float j = floorf(N.ck * r);
    const float lo = e > 0.f ? 0.5f * fmaf(-r, r, e) / r : 0.f;
    *k = min(max((int)j - 5 - N.k_first, 0), N.nk - kTapsK);
    return fmaf(N.ck, r, -j) + fmaf(N.ck_lo, r, N.ck * lo);
}
__device__ __forceinline__ bool in_reach(const NodeConst& N, float e) {
    bool in = false;
    for (int w = 0; w < N.W; ++w) in |= e >= N.reach_lo[w] && e <= N.reach_hi[w];
    return in;
}

__global__ void k_node_matrix(const NodeConst N, double kappa, float* g, float* gt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N.nl * N.nk_pad) return;
    const int l = i / N.nk_pad, k = i % N.nk_pad;
    int w = 0;
    while (w + 1 < N.W && l >= N.l_off[w + 1]) ++w;
    const double xl = 0.5 * kappa * (N.l_first[w] + (l - N.l_off[w])) / kPerUnitL;   // sqrt(E')
    const double xk = 0.5 * kappa * (N.k_first + k) / kPerUnitK;
    const double d = (xk * xk - xl * xl) / (kappa * xl);
    const float v = k < N.nk && fabs(d) <= kBandSigmas ? (float)exp(-0.5 * d * d) : 0.f;
    g[(size_t)l * N.nk_pad + k] = v;
    gt[(size_t)k * N.nl_pad + l] = v;
}

struct NodeParams {
    NodeConst N;
    const float* tab;        // path tables; angle i of the launch in slot slot0 + i slot_step
    int slot0, slot_step;
    int a0, a_step, angles;  // angle i of the launch: a0 + i a_step
    int B, nq, nqt, npc, nq_pad;
    const float* g;          // [nl][nk_pad] Gaussians
    const float* gt;         // [nk][nl_pad] their transpose
    const int2* k_of_l;      // [nl] recorded-energy nodes in reach of node l
    const int2* l_of_k;      // [W][nk_pad] nodes of line w in reach of k
    const int2* chunk_bins;  // [A][npc] bins a chunk of 32 scatter points reaches
    const float* cs;         // [A][npc][B][kCPad]
    const int2* crange;      // [A][B]
    const float* cv;         // [A][B][nq]
    const float* prim;       // [A][W][nq]
    const float* lam;        // [nq]
    float* dbp;              // [angles][npc][nb_max][nl_pad]: DB's part of each chunk
    float* F;                // [angles][B][nk_pad]
    float* Pr;               // [angles][B][W] unscattered sums
    const float* V;          // [angles][B][nk_pad]
    const float* PV;         // [angles][B][W]
    float* VG;               // [angles][B][nl_pad]
    float* part;             // [angles][npc][W][nq_pad]
    float* part_prim;        // [angles][nq_pad]
    int* status;
};

// One CTA per (angle, 32 scatter points, line).  Each warp takes every
// warps-th run of 16 voxels, a lane per scatter point, and adds each path to
// the 7 nodes around its scattered energy in the warp's own sums [node][point]
// in shared memory (a lane only touches its own column: no conflicts between
// lanes or banks).  The tables of a run (nlh and sr, 2 KiB each) arrive by
// bulk copies, double buffered per warp.  The warps' sums are added in warp
// order and contracted with the collimator rows of the bins the 32 points
// reach, so only the bins' node sums leave the SM.
__global__ void __launch_bounds__(32 * kSpreadWarpsMax) k_node_spread(const NodeParams P) {
    extern __shared__ __align__(128) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int W = P.N.W, warps = P.N.spread_warps;
    const int w = blockIdx.x % W, pc = (blockIdx.x / W) % P.npc, ai = blockIdx.x / (W * P.npc);
    const int nlw = P.N.l_count[w];
    float* stages = reinterpret_cast<float*>(smem);
    float* stage0 = stages + warp * (4 * kStageRows * kPC);
    float* sums = stages + warps * (4 * kStageRows * kPC);
    float* mine = sums + (size_t)warp * nlw * kPC + lane;
    __shared__ __align__(8) uint64_t bars[2 * kSpreadWarpsMax];
    const uint32_t bar0 = smem_addr(&bars[2 * warp]);
    if (lane == 0) {
        mbar_init(bar0, 1);
        mbar_init(bar0 + 8, 1);
        mbar_fence_init();
    }
    __syncwarp();
    const size_t block = (size_t)3 * W * kQT * kPC;
    const float* tab = P.tab + ((size_t)(P.slot0 + ai * P.slot_step) * P.nqt * P.npc + pc) * block +
                       (size_t)w * kQT * kPC;
    const int runs = (P.nq + kStageRows - 1) / kStageRows;
    const int nt = runs > warp ? (runs - warp + warps - 1) / warps : 0;
    auto issue = [&](int it) {
        const int run = warp + it * warps;
        const float* src = tab + (size_t)(run / (kQT / kStageRows)) * P.npc * block +
                           (size_t)(run % (kQT / kStageRows)) * (kStageRows * kPC);
        float* dst = stage0 + (it & 1) * (2 * kStageRows * kPC);
        const uint32_t bar = bar0 + 8 * (it & 1);
        mbar_expect_tx(bar, 2 * kStageBytes);
        bulk_g2s(smem_addr(dst), src, kStageBytes, bar);
        bulk_g2s(smem_addr(dst + kStageRows * kPC), src + (size_t)W * kQT * kPC, kStageBytes, bar);
    };
    if (lane == 0) {
        if (nt > 0) issue(0);
        if (nt > 1) issue(1);
    }
    for (int l = 0; l < nlw; ++l) mine[l * kPC] = 0.f;
    const int first = P.N.l_first[w] + 3;
    const unsigned last = (unsigned)(nlw - kTapsL);
    const float c1 = P.N.cl, c1_lo = P.N.cl_lo;
    for (int it = 0; it < nt; ++it) {
        const int q0 = (warp + it * warps) * kStageRows;
        const float lam_l = lane < kStageRows && q0 + lane < P.nq ? P.lam[q0 + lane] : 0.f;
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar0 + 8 * (it & 1), (it >> 1) & 1))) {
            if (lane == 0) {
                atomicOr(P.status, kStatusTimeout);
                // the copies still in flight land before the CTA goes on
                mbar_wait_bounded(bar0 + 8 * (it & 1), (it >> 1) & 1);
                if (it + 1 < nt) mbar_wait_bounded(bar0 + 8 * ((it + 1) & 1), ((it + 1) >> 1) & 1);
            }
            break;
        }
        // the whole stage into registers first: the sums' stores below could
        // alias it as far as the compiler knows, which would keep every load
        // and all arithmetic of a path behind the stores of the one before
        const float* st = stage0 + (it & 1) * (2 * kStageRows * kPC) + lane;
        float nl[kStageRows], sr[kStageRows];
#pragma unroll
        for (int r = 0; r < kStageRows; ++r) {
            nl[r] = st[r * kPC];
            sr[r] = st[(kStageRows + r) * kPC];
        }
        __syncwarp();
        if (lane == 0 && it + 2 < nt) issue(it + 2);
#pragma unroll
        for (int r = 0; r < kStageRows; r += 2) {
            const f32x2 lam = pk(__shfl_sync(0xffffffffu, lam_l, r), __shfl_sync(0xffffffffu, lam_l, r + 1));
            const f32x2 wt = mul2(pk(ex2f(-nl[r]), ex2f(-nl[r + 1])), lam);
            unsigned i0, i1;
            const f32x2 s = node_pos2(sr[r], sr[r + 1], c1, c1_lo, first, last, i0, i1);
            f32x2 c[7];
            lagrange7(s, wt, c);
            float x[7], y[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) upk(c[k], x[k], y[k]);
            float* d = mine + i0 * kPC;
            float v[7];
#pragma unroll
            for (int k = 0; k < 7; ++k) v[k] = d[k * kPC];
#pragma unroll
            for (int k = 0; k < 7; ++k) d[k * kPC] = v[k] + x[k];
            d = mine + i1 * kPC;
#pragma unroll
            for (int k = 0; k < 7; ++k) v[k] = d[k * kPC];
#pragma unroll
            for (int k = 0; k < 7; ++k) d[k * kPC] = v[k] + y[k];
        }
    }
    __syncthreads();
    const int T = blockDim.x;
    for (int i = threadIdx.x; i < nlw * kPC / 4; i += T) {
        float4 a = reinterpret_cast<const float4*>(sums)[i];
        for (int k = 1; k < warps; ++k) {
            const float4 b = reinterpret_cast<const float4*>(sums + (size_t)k * nlw * kPC)[i];
            a.x += b.x;
            a.y += b.y;
            a.z += b.z;
            a.w += b.w;
        }
        reinterpret_cast<float4*>(sums)[i] = a;
    }
    // the bins' sums over the 32 points: a thread per node, 4 bins at a time;
    // the points in quads, rotated by the lane (no bank conflicts)
    const int a = P.a0 + ai * P.a_step;
    const int2 br = P.chunk_bins[(size_t)a * P.npc + pc];
    const float* cr = P.cs + (((size_t)a * P.npc + pc) * P.B + br.x) * kCPad;
    float* out = P.dbp + (((size_t)ai * P.npc + pc) * P.N.nb_max) * P.N.nl_pad + P.N.l_off[w];
    const int nb = br.y - br.x;
    constexpr int kBinsStaged = 64;   // collimator rows staged at a time (8 KiB, in the copy buffers)
    for (int s0 = 0; s0 < nb; s0 += kBinsStaged) {
        const int ns = min(kBinsStaged, nb - s0);
        __syncthreads();
        for (int i = threadIdx.x; i < ((ns + 3) & ~3) * (kPC / 4); i += T) {
            const int b = i >> 3, c = i & 7;
            reinterpret_cast<float4*>(stages)[i] =
                b < ns ? *reinterpret_cast<const float4*>(cr + (size_t)(s0 + b) * kCPad + 4 * c)
                       : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        __syncthreads();
        for (int l = threadIdx.x; l < nlw; l += T) {
            const float4* dl = reinterpret_cast<const float4*>(sums + (size_t)l * kPC);
            for (int b = 0; b < ns; b += 4) {
                const float4* cb = reinterpret_cast<const float4*>(stages) + b * (kPC / 4);
                f32x2 acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
                for (int i = 0; i < kPC / 4; ++i) {
                    const int p = (i + lane) & 7;
                    const float4 d = dl[p];
                    const f32x2 d0 = pk(d.x, d.y), d1 = pk(d.z, d.w);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const float4 c = cb[k * (kPC / 4) + p];
                        acc[k] = fma2(d0, pk(c.x, c.y), acc[k]);
                        acc[k] = fma2(d1, pk(c.z, c.w), acc[k]);
                    }
                }
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (b + k < ns) {
                        float x, y;
                        upk(acc[k], x, y);
                        out[(size_t)(s0 + b + k) * P.N.nl_pad + l] = x + y;
                    }
            }
        }
    }
}

// 8 (angle, bin) rows per block: a row's sums over the chunks of its run of
// scatter points, then the Gaussians onto the recorded-energy nodes, a thread
// per node; the blocks past those form the unscattered sums, a warp per
// (row, line).  Sums run over 32 nodes at a time, then over those.
__global__ void __launch_bounds__(384) k_node_values(const NodeParams P) {
    extern __shared__ __align__(16) float db[];   // [nl][8]
    const int t = threadIdx.x, T = blockDim.x, W = P.N.W;
    const int rows = P.angles * P.B, n_row_blocks = (rows + kValueRows - 1) / kValueRows;
    if ((int)blockIdx.x >= n_row_blocks) {
        const int i = (blockIdx.x - n_row_blocks) * (T >> 5) + (t >> 5);
        if (i >= rows * W) return;
        const int row = i / W, w = i % W;
        const int a = P.a0 + (row / P.B) * P.a_step;
        const float* cv = P.cv + ((size_t)a * P.B + row % P.B) * P.nq;
        const float* pr = P.prim + ((size_t)a * W + w) * P.nq;
        float s = 0.f;
#pragma unroll 4
        for (int q = t & 31; q < P.nq; q += 32) s = fmaf(cv[q] * pr[q], P.lam[q], s);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 31) == 0) P.Pr[i] = s;
        return;
    }
    const int r0 = blockIdx.x * kValueRows;
    for (int i = 0; i < kValueRows; ++i) {
        const int row = r0 + i;
        const int ai = row / P.B, b = row % P.B, a = P.a0 + ai * P.a_step;
        const int2 run = row < rows ? P.crange[(size_t)a * P.B + b] : make_int2(0, 0);
        const int c0 = run.x / kPC, c1 = run.y > run.x ? (run.y + kPC - 1) / kPC : c0;
        for (int l = t; l < P.N.nl; l += T) {
            float s = 0.f;
#pragma unroll 4
            for (int pc = c0; pc < c1; ++pc) {
                const int b0 = P.chunk_bins[(size_t)a * P.npc + pc].x;
                s += P.dbp[(((size_t)ai * P.npc + pc) * P.N.nb_max + (b - b0)) * P.N.nl_pad + l];
            }
            db[l * kValueRows + i] = s;
        }
    }
    __syncthreads();
    for (int k = t; (k & ~31) < P.N.nk; k += T) {
        f32x2 f[kValueRows / 2] = {0ull, 0ull, 0ull, 0ull};
        for (int w = 0; w < W; ++w) {
            // the warp's nodes l: from its first node's reach to its last's
            const int2 r = P.l_of_k[(size_t)w * P.N.nk_pad + min(k, P.N.nk - 1)];
            const int lo = __reduce_min_sync(0xffffffffu, r.y > r.x ? r.x : 0x7fffffff);
            const int hi = __reduce_max_sync(0xffffffffu, r.y);
            for (int l0 = lo; l0 < hi; l0 += 32) {
                f32x2 s[kValueRows / 2] = {0ull, 0ull, 0ull, 0ull};
                const int l1 = min(l0 + 32, hi);
    #pragma unroll 8
                for (int l = l0; l < l1; ++l) {
                    const float g = P.g[(size_t)l * P.N.nk_pad + k];
                    const float4 d0 = *reinterpret_cast<const float4*>(db + l * kValueRows);
                    const float4 d1 = *reinterpret_cast<const float4*>(db + l * kValueRows + 4);
                    const f32x2 g2 = pk1(g);
                    s[0] = fma2(g2, pk(d0.x, d0.y), s[0]);
                    s[1] = fma2(g2, pk(d0.z, d0.w), s[1]);
                    s[2] = fma2(g2, pk(d1.x, d1.y), s[2]);
                    s[3] = fma2(g2, pk(d1.z, d1.w), s[3]);
                }
    #pragma unroll
                for (int i = 0; i < kValueRows / 2; ++i) f[i] = add2(f[i], s[i]);
            }
        }
    #pragma unroll
        for (int i = 0; i < kValueRows / 2; ++i) {
            float x, y;
            upk(f[i], x, y);
            if (r0 + 2 * i < rows) P.F[(size_t)(r0 + 2 * i) * P.N.nk_pad + k] = x;
            if (r0 + 2 * i + 1 < rows) P.F[(size_t)(r0 + 2 * i + 1) * P.N.nk_pad + k] = y;
        }
    }
}

// Transposed: the Gaussians from the recorded-energy nodes onto the scattered-
// energy nodes, 8 (angle, bin) rows per block, a thread per node; the blocks
// past those form the unscattered part of the back projection, a thread per
// voxel.
__global__ void __launch_bounds__(256) k_node_unvalues(const NodeParams P) {
    extern __shared__ __align__(16) float vb[];   // [nk][8]
    const int t = threadIdx.x, W = P.N.W;
    const int rows = P.angles * P.B;
    const int lt = (P.N.nl + 255) / 256;
    const int n_row_blocks = (rows + kValueRows - 1) / kValueRows * lt;
    if ((int)blockIdx.x >= n_row_blocks) {
        const int qb = (P.nq + 255) / 256;
        const int ai = (blockIdx.x - n_row_blocks) / qb;
        const int q = ((blockIdx.x - n_row_blocks) % qb) * 256 + t;
        if (q >= P.nq) return;
        const int a = P.a0 + ai * P.a_step;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        const float* cv = P.cv + (size_t)a * P.B * P.nq + q;
        const float* pv = P.PV + (size_t)ai * P.B * W;
#pragma unroll 8
        for (int b = 0; b < P.B; ++b) {
            const float c = cv[(size_t)b * P.nq];
#pragma unroll
            for (int w = 0; w < 4; ++w)
                if (w < W) s[w] = fmaf(c, pv[b * W + w], s[w]);
        }
        float o = 0.f;
#pragma unroll
        for (int w = 0; w < 4; ++w)
            if (w < W) o = fmaf(P.prim[((size_t)a * W + w) * P.nq + q], s[w], o);
        P.part_prim[(size_t)ai * P.nq_pad + q] = o;
        return;
    }
    const int r0 = (blockIdx.x / lt) * kValueRows;
    for (int i = 0; i < kValueRows; ++i)
        for (int k = t; k < P.N.nk; k += 256)
            vb[k * kValueRows + i] = r0 + i < rows ? P.V[(size_t)(r0 + i) * P.N.nk_pad + k] : 0.f;
    __syncthreads();
    const int l = (blockIdx.x % lt) * 256 + t;
    if ((l & ~31) >= P.N.nl) return;
    const int2 r = P.k_of_l[min(l, P.N.nl - 1)];
    const int lo = __reduce_min_sync(0xffffffffu, r.y > r.x ? r.x : 0x7fffffff);
    const int hi = __reduce_max_sync(0xffffffffu, r.y);
    f32x2 f[kValueRows / 2] = {0ull, 0ull, 0ull, 0ull};
    for (int k0 = lo; k0 < hi; k0 += 32) {
        f32x2 s[kValueRows / 2] = {0ull, 0ull, 0ull, 0ull};
        const int k1 = min(k0 + 32, hi);
#pragma unroll 8
        for (int k = k0; k < k1; ++k) {
            const float g = P.gt[(size_t)k * P.N.nl_pad + l];
            const float4 d0 = *reinterpret_cast<const float4*>(vb + k * kValueRows);
            const float4 d1 = *reinterpret_cast<const float4*>(vb + k * kValueRows + 4);
            const f32x2 g2 = pk1(g);
            s[0] = fma2(g2, pk(d0.x, d0.y), s[0]);
            s[1] = fma2(g2, pk(d0.z, d0.w), s[1]);
            s[2] = fma2(g2, pk(d1.x, d1.y), s[2]);
            s[3] = fma2(g2, pk(d1.z, d1.w), s[3]);
        }
#pragma unroll
        for (int i = 0; i < kValueRows / 2; ++i) f[i] = add2(f[i], s[i]);
    }
#pragma unroll
    for (int i = 0; i < kValueRows / 2; ++i) {
        float x, y;
        upk(f[i], x, y);
        if (r0 + 2 * i < rows) P.VG[(size_t)(r0 + 2 * i) * P.N.nl_pad + l] = x;
        if (r0 + 2 * i + 1 < rows) P.VG[(size_t)(r0 + 2 * i + 1) * P.N.nl_pad + l] = y;
    }
}

// One CTA per (angle, 32 scatter points, line): PHI of the 32 points [node]
// [point] in shared memory, then every voxel's sum over the 32 points, a lane
// per point, each warp every 8th tile of 32 voxels (8 at a time: loads in
// flight together, the lanes' values added by a butterfly that leaves voxel r
// in lanes 4 r .. 4 r + 3).
__global__ void __launch_bounds__(kGatherThreads) k_node_gather(const NodeParams P) {
    extern __shared__ __align__(16) float phi[];   // [node][32]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int kWarps = kGatherThreads / 32;
    const int W = P.N.W;
    const int w = blockIdx.x % W, pc = (blockIdx.x / W) % P.npc, ai = blockIdx.x / (W * P.npc);
    const int a = P.a0 + ai * P.a_step;
    const int nlw = P.N.l_count[w];
    const int2 br = P.chunk_bins[(size_t)a * P.npc + pc];
    {
        const float* cr = P.cs + (((size_t)a * P.npc + pc) * P.B) * kCPad + lane;
        const float* vg = P.VG + (size_t)ai * P.B * P.N.nl_pad + P.N.l_off[w];
        for (int l0 = warp * 8; l0 < nlw; l0 += kWarps * 8) {
            float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
            for (int b = br.x; b < br.y; ++b) {
                const float c = cr[(size_t)b * kCPad];
                const float* v = vg + (size_t)b * P.N.nl_pad + l0;
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    if (l0 + i < nlw) acc[i] = fmaf(c, v[i], acc[i]);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (l0 + i < nlw) phi[(l0 + i) * kPC + lane] = acc[i];
        }
    }
    __syncthreads();
    const size_t block = (size_t)3 * W * kQT * kPC;
    const float* tab = P.tab + ((size_t)(P.slot0 + ai * P.slot_step) * P.nqt * P.npc + pc) * block +
                       (size_t)w * kQT * kPC + lane;
    const float* col = phi + lane;
    float* out = P.part + (size_t)blockIdx.x * P.nq_pad;
    const int first = P.N.l_first[w] + 3;
    const unsigned last = (unsigned)(nlw - kTapsL);
    const float c1 = P.N.cl, c1_lo = P.N.cl_lo;
    for (int qt = warp; qt < P.nqt; qt += kWarps) {
        const float* src = tab + (size_t)qt * P.npc * block;
#pragma unroll 1
        for (int r0 = 0; r0 < kQT; r0 += 8) {
            float nl[8], sr[8], v[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                nl[r] = src[(r0 + r) * kPC];
                sr[r] = src[(size_t)W * kQT * kPC + (r0 + r) * kPC];
            }
#pragma unroll
            for (int r = 0; r < 8; r += 2) {
                unsigned i0, i1;
                const f32x2 s = node_pos2(sr[r], sr[r + 1], c1, c1_lo, first, last, i0, i1);
                f32x2 c[7];
                lagrange7(s, pk(ex2f(-nl[r]), ex2f(-nl[r + 1])), c);
                const float *d0 = col + i0 * kPC, *d1 = col + i1 * kPC;
                f32x2 acc = mul2(c[0], pk(d0[0], d1[0]));
#pragma unroll
                for (int k = 1; k < 7; ++k) acc = fma2(c[k], pk(d0[k * kPC], d1[k * kPC]), acc);
                upk(acc, v[r], v[r + 1]);
            }
            // lanes' sums: after the three exchanges lane keeps voxel (lane >> 2)
            const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
            float u[4], x[2], z;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float give = h16 ? v[i] : v[i + 4], keep = h16 ? v[i + 4] : v[i];
                u[i] = keep + __shfl_xor_sync(0xffffffffu, give, 16);
            }
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const float give = h8 ? u[i] : u[i + 2], keep = h8 ? u[i + 2] : u[i];
                x[i] = keep + __shfl_xor_sync(0xffffffffu, give, 8);
            }
            {
                const float give = h4 ? x[0] : x[1], keep = h4 ? x[1] : x[0];
                z = keep + __shfl_xor_sync(0xffffffffu, give, 4);
            }
            z += __shfl_xor_sync(0xffffffffu, z, 2);
            z += __shfl_xor_sync(0xffffffffu, z, 1);
            if ((lane & 3) == 0) out[qt * kQT + r0 + (lane >> 2)] = z;
        }
    }
}

struct EventParams {
    NodeConst N;
    LineConst lc;
    const float* F;        // [angles][B][nk_pad]
    const float* Pr;       // [angles][B][W]
    int B;
};

// Unscattered part of one event: sum over lines of its response at the line
// times the cell's sum; g[w] the responses.
__device__ __forceinline__ float line_response(const EventParams& P, float e, int w) {
    const float d = e - P.lc.e[w];
    return P.lc.norm[w] * ex2f(P.lc.nk[w] * d * d);
}

// Forward values in the caller's event order, for the events of angles
// a0 .. a0 + angles - 1 (every angle: all events).  Events outside the model
// get NaN and set the status word (in the pass that holds angle 0).
__global__ void __launch_bounds__(256) k_node_y(const EventParams P, const uint16_t* angle,
                                                const uint16_t* bin, const float* energy,
                                                int64_t n, int A, int n_win, const NodeWindows win,
                                                int a0, int angles, float* out, int* status) {
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int a = angle[j], b = bin[j];
    const float e = energy[j];
    bool in = false;
    for (int k = 0; k < n_win; ++k) in |= e >= win.lo[k] && e < win.hi[k];
    if (!(a < A && b < P.B && isfinite(e) && in)) {
        if (a0 == 0) {
            out[j] = __int_as_float(0x7fc00000);
            atomicOr(status, kStatusOutOfRange);
        }
        return;
    }
    const int ai = a - a0;
    if (ai < 0 || ai >= angles) return;
    const size_t cell = (size_t)ai * P.B + b;
    float y = 0.f;
    for (int w = 0; w < P.N.W; ++w) y = fmaf(P.Pr[cell * P.N.W + w], line_response(P, e, w), y);
    if (in_reach(P.N, e)) {
        const float* F = P.F + cell * P.N.nk_pad;
        int k;
        float wt[12];
        lagrange12(energy_pos(P.N, e, &k), wt);
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int i = 0; i < 12; i += 2) {
            s0 = fmaf(wt[i], F[k + i], s0);
            s1 = fmaf(wt[i + 1], F[k + i + 1], s1);
        }
        y += s0 + s1;
    }
    out[j] = y;
}

// One block per (angle, bin) cell of sorted events.  With F: the cell's
// forward values, the ratios r_j = 1 / y_j (0 where y_j <= 0) and, when ll is
// set, the cell's FP64 sum of log y_j; else r_j = the caller's weights.  Then
// the cell's node weights V = sum_j r_j L(E_j) and unscattered weights PV.  A
// lane forms the values of one event; the events' 12 taps are then added one
// event per half-warp at a time into the half-warp's own row, 12 lanes one tap
// each.  The rows are emptied into second sums every 256 events of a warp.
__global__ void __launch_bounds__(32 * kCellWarps) k_node_cells(
    const EventParams P, const int* cell_start, int cell0, const float* energy, const float* weight,
    const uint32_t* perm, float* V, float* PV, double* ll) {
    extern __shared__ float sh[];
    constexpr int kRows = 2 * kCellWarps;
    const int nkp = P.N.nk_pad, W = P.N.W;
    float* Fs = sh;                          // [nk_pad]
    float* acc = Fs + nkp;                   // [kRows][nk_pad]
    float* tot = acc + kRows * nkp;          // [kRows][nk_pad]
    __shared__ float wts[kCellWarps][32][13];
    __shared__ int kpos[kCellWarps][32];
    __shared__ float pv_s[kCellWarps][4];
    __shared__ double ll_s[kCellWarps];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const size_t cell = blockIdx.x;
    const int e0 = cell_start[cell0 + blockIdx.x], e1 = cell_start[cell0 + blockIdx.x + 1];
    float* out = V + cell * nkp;
    if (e0 == e1) {
        for (int k = t; k < nkp; k += 32 * kCellWarps) out[k] = 0.f;
        if (t < W) PV[cell * W + t] = 0.f;
        if (ll && t == 0) ll[cell] = 0.0;
        return;
    }
    for (int k = t; k < nkp; k += 32 * kCellWarps) {
        if (P.F) Fs[k] = P.F[cell * nkp + k];
        for (int i = 0; i < kRows; ++i) acc[i * nkp + k] = tot[i * nkp + k] = 0.f;
    }
    __syncthreads();
    float pv[4] = {0.f, 0.f, 0.f, 0.f};
    double lsum = 0.0;
    float* mine = acc + (2 * warp + (lane >> 4)) * nkp;
    const int tap = lane & 15;
    int batches = 0;
    for (int b0 = e0 + 32 * warp; b0 < e1; b0 += 32 * kCellWarps) {
        const int j = b0 + lane;
        float r = 0.f, wt[12];
        int k = 0;
        bool reach = false;
        if (j < e1) {
            const float e = energy[j];
            float g[4];
            float y = 0.f;
#pragma unroll
            for (int w = 0; w < 4; ++w)
                if (w < W) {
                    g[w] = line_response(P, e, w);
                    if (P.F) y = fmaf(P.Pr[cell * W + w], g[w], y);
                }
            reach = in_reach(P.N, e);
            if (reach) lagrange12(energy_pos(P.N, e, &k), wt);
            if (P.F) {
                if (reach) {
                    float s0 = 0.f, s1 = 0.f;
#pragma unroll
                    for (int i = 0; i < 12; i += 2) {
                        s0 = fmaf(wt[i], Fs[k + i], s0);
                        s1 = fmaf(wt[i + 1], Fs[k + i + 1], s1);
                    }
                    y += s0 + s1;
                }
                if (y > 0.f) {
                    r = 1.0f / y;
                    if (ll) lsum += log((double)y);
                }
            } else {
                r = weight[perm[j]];
            }
#pragma unroll
            for (int w = 0; w < 4; ++w)
                if (w < W) pv[w] = fmaf(r, g[w], pv[w]);
        }
        kpos[warp][lane] = k;
#pragma unroll
        for (int i = 0; i < 12; ++i) wts[warp][lane][i] = reach ? r * wt[i] : 0.f;
        __syncwarp();
        const int n_here = min(32, e1 - b0);
        const int h0 = (lane >> 4) * 16;
        for (int i = 0; i < 16; ++i) {
            const int ev = h0 + i;
            if (ev < n_here && tap < kTapsK) mine[kpos[warp][ev] + tap] += wts[warp][ev][tap];
            __syncwarp();
        }
        if ((++batches & 7) == 0) {
            for (int k2 = tap; k2 < nkp; k2 += 16) {
                tot[mine - acc + k2] += mine[k2];
                mine[k2] = 0.f;
            }
            __syncwarp();
        }
    }
#pragma unroll
    for (int w = 0; w < 4; ++w) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pv[w] += __shfl_xor_sync(0xffffffffu, pv[w], o);
        if (lane == 0) pv_s[warp][w] = pv[w];
    }
    if (ll) {
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0) ll_s[warp] = lsum;
    }
    __syncthreads();
    for (int k = t; k < nkp; k += 32 * kCellWarps) {
        float s = 0.f;
        for (int i = 0; i < kRows; ++i) s += tot[i * nkp + k] + acc[i * nkp + k];
        out[k] = s;
    }
    if (t < W) {
        float s = 0.f;
        for (int i = 0; i < kCellWarps; ++i) s += pv_s[i][t];
        PV[cell * W + t] = s;
    }
    if (ll && t == 0) {
        double s = 0.0;
        for (int i = 0; i < kCellWarps; ++i) s += ll_s[i];
        ll[cell] = s;
    }
}

// Voxel sums over the parts (FP64, 32 strands in fixed order) and, with sens,
// the multiplicative update of lam; else the sums go to num.  One block per
// 32 voxels.
__global__ void __launch_bounds__(1024) k_node_update(const float* part, int64_t n_part,
                                                      const float* part_prim, int n_prim,
                                                      int nq, int nq_pad, const double* sens,
                                                      float* lam, double* num) {
    __shared__ double red[32][33];
    const int lane = threadIdx.x & 31, strand = threadIdx.x >> 5;
    const int q = blockIdx.x * 32 + lane;
    double s = 0.0;
    if (q < nq) {
#pragma unroll 4
        for (int64_t i = strand; i < n_part; i += 32) s += (double)part[(size_t)i * nq_pad + q];
        for (int i = strand; i < n_prim; i += 32) s += (double)part_prim[(size_t)i * nq_pad + q];
    }
    red[strand][lane] = s;
    __syncthreads();
    if (strand == 0 && q < nq) {
        double v = 0.0;
        for (int i = 0; i < 32; ++i) v += red[i][lane];
        if (sens)
            lam[q] = sens[q] > 0.0 ? (float)((double)lam[q] * v / sens[q]) : 0.f;
        else
            num[q] = v;
    }
}

// Log-likelihood at the incoming image: the cells' log sums minus sum lam sens.
__global__ void __launch_bounds__(1024) k_node_loglik(const double* ll, int n_ll, const float* lam,
                                                      const double* sens, int nq, double* out) {
    __shared__ double red[1024];
    const int t = threadIdx.x;
    double s = 0.0;
    for (int i = t; i < n_ll; i += 1024) s += ll[i];
    for (int q = t; q < nq; q += 1024) s -= (double)lam[q] * sens[q];
    red[t] = s;
    __syncthreads();
    for (int off = 512; off > 0; off >>= 1) {
        if (t < off) red[t] += red[t + off];
        __syncthreads();
    }
    if (t == 0) *out = red[0];
}

// Bins a chunk of 32 scatter points reaches: those whose run overlaps it.
__global__ void k_chunk_bins(const int2* crange, int B, int npc, int2* chunk_bins, int* most) {
    const int a = blockIdx.y, pc = blockIdx.x * blockDim.x + threadIdx.x;
    if (pc >= npc) return;
    int lo = B, hi = 0;
    for (int b = 0; b < B; ++b) {
        const int2 r = crange[(size_t)a * B + b];
        if (r.y > r.x && r.x < (pc + 1) * kPC && r.y > pc * kPC) {
            lo = min(lo, b);
            hi = b + 1;
        }
    }
    chunk_bins[(size_t)a * npc + pc] = lo < hi ? make_int2(lo, hi) : make_int2(0, 0);
    atomicMax(most, max(hi - lo, 0));
}

// Shared-memory opt-in of the node kernels, once per device.
int node_kernel_attrs() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0, cap = 0;
    LMMEW_CUDA(cudaGetDevice(&dev));
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load() & bit) return LMMEW_OK;
    LMMEW_CUDA(cudaDeviceGetAttribute(&cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    cudaFuncAttributes fa;
    LMMEW_CUDA(cudaFuncGetAttributes(&fa, k_node_spread));
    LMMEW_CUDA(cudaFuncSetAttribute(k_node_spread, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    cap - (int)fa.sharedSizeBytes));
    LMMEW_CUDA(cudaFuncSetAttribute(k_node_gather, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    cap - 1024));
    LMMEW_CUDA(cudaFuncSetAttribute(k_node_values, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    cap - 1024));
    LMMEW_CUDA(cudaFuncSetAttribute(k_node_unvalues, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    cap - 1024));
    LMMEW_CUDA(cudaFuncSetAttribute(k_node_cells, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    64 * 1024));
    done.fetch_or(bit);
    return LMMEW_OK;
}

}  // namespace

// Nodes of the model's energies and the Gaussians between them.  The route
// exists for the square-root energy resolution, with energy classes on, when
// the node sums of 32 scatter points fit shared memory and one angle's sums
// the static scratch of lm_forward_noalloc (so that call takes the same route).
int build_nodes(lm_handle* h) {
    const ModelConst& m = h->mc;
    NodeConst& N = h->nodes;
    h->node_route = 0;
    N = NodeConst{};
    if (m.np == 0 || m.W > 4 || m.expo != -0.5) return LMMEW_OK;
    const double f2s = 1.0 / (2.0 * sqrt(2.0 * log(2.0)));
    const double kappa = m.fwhm_frac * sqrt(m.e_ref) * f2s;   // sigma = kappa sqrt(E)
    auto t_of = [&](double e) { return 2.0 * sqrt(e) / kappa; };
    N.W = m.W;
    const double cl = kPerUnitL * 2.0 * sqrt(0.5 * 1.4426950408889634) / (kappa * kappa);
    const double ck = kPerUnitK * 2.0 / kappa;
    N.cl = (float)cl;
    N.cl_lo = (float)(cl - (double)N.cl);
    N.ck = (float)ck;
    N.ck_lo = (float)(ck - (double)N.ck);
    double e_lo = 1e300, e_hi = 0.0;
    for (int k = 0; k < m.n_win; ++k) {
        e_lo = std::min(e_lo, std::max(m.win_lo[k], 0.0));
        e_hi = std::max(e_hi, m.win_hi[k]);
    }
    const double t_hi = t_of(e_hi) * kPerUnitK;
    if (!(t_hi < 8192.0)) return LMMEW_OK;
    N.k_first = (int)floor(t_of(e_lo) * kPerUnitK) - 6;
    N.nk = (int)floor(t_hi) + 7 - N.k_first + 1;
    N.nk_pad = (N.nk + 31) & ~31;
    int most = 0;
    for (int w = 0; w < m.W; ++w) {
        const double eb = m.line_e[w] / (1.0 + 2.0 * m.line_e[w] / 510.99895);
        const double u0 = t_of(eb) * kPerUnitL, u1 = t_of(m.line_e[w]) * kPerUnitL;
        if (!(u1 < 1.0e6)) return LMMEW_OK;
        N.l_first[w] = (int)floor(u0) - 4;
        N.l_count[w] = (int)ceil(u1) + 4 - N.l_first[w] + 1;
        if (N.l_first[w] < 1) return LMMEW_OK;
        N.l_off[w] = N.nl;
        N.nl += N.l_count[w];
        most = std::max(most, N.l_count[w]);
    }
    N.nl_pad = (N.nl + 31) & ~31;
    int dev = 0, max_smem = 0;
    LMMEW_CUDA(cudaGetDevice(&dev));
    LMMEW_CUDA(cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    const size_t per_warp = 4 * kStageBytes + (size_t)most * kPC * 4;
    N.spread_warps = (int)std::min<size_t>(kSpreadWarpsMax, (size_t)(max_smem - 1024) / per_warp);
    N.spread_smem = (int)(N.spread_warps * per_warp);
    N.gather_smem = most * kPC * 4;
    if (N.spread_warps < 1 || N.gather_smem > 200 * 1024 || N.nl > 6000 || N.nk > 1024) return LMMEW_OK;
    LMMEW_CUDA(cudaMalloc(&h->d_chunk_bins, sizeof(int2) * ((size_t)m.A * m.npc + 1)));
    int* d_most = reinterpret_cast<int*>(h->d_chunk_bins + (size_t)m.A * m.npc);
    LMMEW_CUDA(cudaMemset(d_most, 0, sizeof(int)));
    k_chunk_bins<<<dim3((m.npc + 31) / 32, m.A), 32>>>(h->d_crange, m.B, m.npc, h->d_chunk_bins, d_most);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    LMMEW_CUDA(cudaMemcpy(&N.nb_max, d_most, sizeof(int), cudaMemcpyDeviceToHost));
    if (N.nb_max < 1) return LMMEW_OK;
    // one angle (with the voxel values) fits lm_forward_noalloc's array
    if (node_angle_bytes(h) + sizeof(float) * (size_t)m.nq + 4096 > (size_t(16) << 20)) return LMMEW_OK;
    for (int w = 0; w < m.W; ++w) line_reach(h, w, &N.reach_lo[w], &N.reach_hi[w]);
    // bands of the Gaussian matrix
    auto e_l = [&](int w, int i) { const double x = 0.5 * kappa * (N.l_first[w] + i) / kPerUnitL; return x * x; };
    auto e_k = [&](int k) { const double x = 0.5 * kappa * (N.k_first + k) / kPerUnitK; return x * x; };
    std::vector<int2> bands((size_t)N.nl + (size_t)m.W * N.nk_pad, make_int2(0, 0));
    int2* k_of_l = bands.data();
    int2* l_of_k = k_of_l + N.nl;
    for (int w = 0; w < m.W; ++w)
        for (int i = 0; i < N.l_count[w]; ++i) {
            const double e = e_l(w, i), s = kBandSigmas * kappa * sqrt(e);
            int2 r = make_int2(N.nk, 0);
            for (int k = 0; k < N.nk; ++k)
                if (fabs(e_k(k) - e) <= s) {
                    r.x = std::min(r.x, k);
                    r.y = k + 1;
                    int2& q = l_of_k[(size_t)w * N.nk_pad + k];
                    if (q.y == 0) q.x = N.l_off[w] + i;
                    q.y = N.l_off[w] + i + 1;
                }
            if (r.y == 0) r.x = 0;
            k_of_l[N.l_off[w] + i] = r;
        }
    const size_t gm = (size_t)N.nl_pad * N.nk_pad;
    if (cudaMalloc(&h->d_node_g, 2 * gm * sizeof(float)) != cudaSuccess ||
        cudaMalloc(&h->d_node_band, bands.size() * sizeof(int2)) != cudaSuccess) {
        cudaGetLastError();
        return set_error(LMMEW_ERR_OOM, "cannot allocate the energy nodes");
    }
    LMMEW_CUDA(cudaMemset(h->d_node_g, 0, 2 * gm * sizeof(float)));
    LMMEW_CUDA(cudaMemcpy(h->d_node_band, bands.data(), bands.size() * sizeof(int2),
                          cudaMemcpyHostToDevice));
    const int total = N.nl * N.nk_pad;
    k_node_matrix<<<(total + 255) / 256, 256>>>(N, kappa, h->d_node_g, h->d_node_g + gm);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    LMMEW_CUDA(cudaDeviceSynchronize());
    h->node_route = 1;
    return node_kernel_attrs();
}

size_t node_angle_bytes(const lm_handle* h) {
    const NodeConst& N = h->nodes;
    return bump_bytes(sizeof(float) * (size_t)h->mc.npc * N.nb_max * N.nl_pad) +
           bump_bytes(sizeof(float) * (size_t)h->mc.B * N.nk_pad) +
           bump_bytes(sizeof(float) * (size_t)h->mc.B * N.W);
}

namespace {

NodeParams node_params(const lm_handle* h, int a0, int a_step, int angles) {
    const ModelConst& m = h->mc;
    const NodeConst& N = h->nodes;
    NodeParams P{};
    P.N = N;
    P.tab = h->d_tab;
    P.a0 = a0;
    P.a_step = a_step;
    P.angles = angles;
    P.B = m.B;
    P.nq = m.nq;
    P.nqt = m.nqt;
    P.npc = m.npc;
    P.nq_pad = m.nqt * kQT;
    P.g = h->d_node_g;
    P.gt = h->d_node_g + (size_t)N.nl_pad * N.nk_pad;
    P.k_of_l = h->d_node_band;
    P.l_of_k = h->d_node_band + N.nl;
    P.chunk_bins = h->d_chunk_bins;
    P.cs = h->d_cs;
    P.crange = h->d_crange;
    P.cv = h->d_cv;
    P.prim = h->d_prim;
    P.status = h->d_status;
    return P;
}

// The slot of the block's first angle in the table buffer and the step
// between slots (streamed tables: the block is built first).
int table_slots(lm_handle* h, int a0, int a_step, int angles, int* slot0, int* step,
                cudaStream_t st) {
    *slot0 = a0;
    *step = a_step;
    if (!h->tab_slots) return LMMEW_OK;
    const int rc = stream_tables(h, a0, a_step, angles, st);
    if (rc != LMMEW_OK) return rc;
    *slot0 = (a0 - h->tab_a0) / h->tab_astep;
    *step = angles > 1 ? a_step / h->tab_astep : 0;
    return LMMEW_OK;
}

}  // namespace

// DB, F and the unscattered sums of angles a0 + i a_step, i < angles.
int node_forward(lm_handle* h, const float* lam_v, int a0, int a_step, int angles, float* dbp,
                 float* F, float* Pr, cudaStream_t st) {
    if (angles <= 0) return LMMEW_OK;
    const ModelConst& m = h->mc;
    const NodeConst& N = h->nodes;
    // angles in blocks of the streamed table buffer (all of them if resident)
    const int per = h->tab_slots ? h->tab_slots : angles;
    for (int i = 0; i < angles; i += per) {
        const int cnt = std::min(per, angles - i);
        NodeParams P = node_params(h, a0 + i * a_step, a_step, cnt);
        int rc = table_slots(h, P.a0, a_step, cnt, &P.slot0, &P.slot_step, st);
        if (rc != LMMEW_OK) return rc;
        P.tab = h->d_tab;
        P.lam = lam_v;
        P.dbp = dbp + (size_t)i * m.npc * N.nb_max * N.nl_pad;
        rc = prof_start(h, st);
        if (rc != LMMEW_OK) return rc;
        k_node_spread<<<(unsigned)(cnt * m.npc * m.W), 32 * N.spread_warps, N.spread_smem, st>>>(P);
        ++h->launches;
        LMMEW_CUDA(cudaGetLastError());
        rc = prof_stop(h, (double)cnt * m.W * m.nq * m.np, st);
        if (rc != LMMEW_OK) return rc;
    }
    NodeParams P = node_params(h, a0, a_step, angles);
    P.lam = lam_v;
    P.dbp = dbp;
    P.F = F;
    P.Pr = Pr;
    const int rows = angles * m.B;
    const int blocks = (rows + kValueRows - 1) / kValueRows + (rows * m.W + 11) / 12;
    k_node_values<<<(unsigned)blocks, 384, sizeof(float) * kValueRows * N.nl, st>>>(P);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    return LMMEW_OK;
}

// Node weights of the cells (angles x bins, from cell0 on) of sorted events.
// F set: from the events' ratios (ll: the cells' log sums); else from weight.
int node_cells(lm_handle* h, int angles, const int* cell_start, int cell0, const float* energy,
               const float* F, const float* Pr, const float* weight, const uint32_t* perm, float* V,
               float* PV, double* ll, cudaStream_t st) {
    const NodeConst& N = h->nodes;
    EventParams P{N, h->lc, F, Pr, h->mc.B};
    const size_t smem = sizeof(float) * (size_t)N.nk_pad * (1 + 4 * kCellWarps);
    k_node_cells<<<(unsigned)(angles * h->mc.B), 32 * kCellWarps, smem, st>>>(
        P, cell_start, cell0, energy, weight, perm, V, PV, ll);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    return LMMEW_OK;
}

// Back projection of the node weights of angles a0 + i a_step: parts of the
// voxel sums per (angle, 32 points, line) and, unscattered, per angle.
int node_back(lm_handle* h, int a0, int a_step, int angles, const float* V, const float* PV,
              float* VG, float* part, float* part_prim, cudaStream_t st) {
    if (angles <= 0) return LMMEW_OK;
    const ModelConst& m = h->mc;
    const NodeConst& N = h->nodes;
    {
        NodeParams P = node_params(h, a0, a_step, angles);
        P.V = V;
        P.PV = PV;
        P.VG = VG;
        P.part_prim = part_prim;
        const int rows = angles * m.B;
        const int blocks = (rows + kValueRows - 1) / kValueRows * ((N.nl + 255) / 256) +
                           angles * ((m.nq + 255) / 256);
        k_node_unvalues<<<(unsigned)blocks, 256, sizeof(float) * kValueRows * N.nk, st>>>(P);
        ++h->launches;
        LMMEW_CUDA(cudaGetLastError());
    }
    const int per = h->tab_slots ? h->tab_slots : angles;
    for (int i = 0; i < angles; i += per) {
        const int cnt = std::min(per, angles - i);
        NodeParams P = node_params(h, a0 + i * a_step, a_step, cnt);
        int rc = table_slots(h, P.a0, a_step, cnt, &P.slot0, &P.slot_step, st);
        if (rc != LMMEW_OK) return rc;
        P.tab = h->d_tab;
        P.VG = VG + (size_t)i * m.B * N.nl_pad;
        P.part = part + (size_t)i * m.npc * m.W * P.nq_pad;
        rc = prof_start(h, st);
        if (rc != LMMEW_OK) return rc;
        k_node_gather<<<(unsigned)(cnt * m.npc * m.W), kGatherThreads, N.gather_smem, st>>>(P);
        ++h->launches;
        LMMEW_CUDA(cudaGetLastError());
        rc = prof_stop(h, (double)cnt * m.W * m.nq * m.np, st);
        if (rc != LMMEW_OK) return rc;
    }
    return LMMEW_OK;
}

// The voxel sums of `angles` angles' parts: with sens the update of lam, else
// into num.
int node_update(lm_handle* h, int angles, const float* part, const float* part_prim,
                const double* sens, float* lam, double* num, cudaStream_t st) {
    const ModelConst& m = h->mc;
    k_node_update<<<(m.nq + 31) / 32, 1024, 0, st>>>(part, (int64_t)angles * m.npc * m.W, part_prim,
                                                     angles, m.nq, m.nqt * kQT, sens, lam, num);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    return LMMEW_OK;
}

int node_loglik(lm_handle* h, const double* ll, int n_ll, const float* lam, const double* sens,
                double* out, cudaStream_t st) {
    k_node_loglik<<<1, 1024, 0, st>>>(ll, n_ll, lam, sens, h->mc.nq, out);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    return LMMEW_OK;
}

int node_events_forward(lm_handle* h, const lm_events* ev, const float* F, const float* Pr, int a0,
                        int angles, float* out_y, cudaStream_t st) {
    const ModelConst& m = h->mc;
    EventParams P{h->nodes, h->lc, F, Pr, m.B};
    NodeWindows win{};
    for (int k = 0; k < m.n_win; ++k) {
        win.lo[k] = (float)m.win_lo[k];
        win.hi[k] = (float)m.win_hi[k];
    }
    k_node_y<<<(unsigned)((ev->n + 255) / 256), 256, 0, st>>>(P, ev->angle, ev->bin, ev->energy_keV,
                                                              ev->n, m.A, m.n_win, win, a0, angles,
                                                              out_y, h->d_status);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    return LMMEW_OK;
}

}  // namespace lmmew
