// Projections of dense event lists through angle and energy nodes.
//
// The single-scatter part of an event's row is a sum over paths (voxel q,
// scatter point p, line w) of Gaussians in the recorded energy.  Its factors
// split by what they depend on.  With phi_qp the direction from q to p, theta
// the detector direction, x = phi_qp - theta and E'(x) Compton's energy,
//
//   C_p(b) B_{qpw} f_w(x) exp(-mu(E'(x)) gamma_p) g(E; E'(x)),
//
// B_{qpw} = alpha mu_0 rho_p A_p / d exp(-mu_0 gamma_qp) / K does not depend
// on the detector angle, f = KN shape / (sqrt(2 pi) sigma(E')), gamma_p is the
// point's line integral to the detector and g the unit Gaussian, smooth in E
// and E' on the scale of sigma.  So the sums go through nodes with local
// Lagrange interpolation (the idea of the fast Gauss transform, Greengard &
// Strain 1991, with local polynomials): N_w directions around the circle (a
// multiple of the angle count, so that x falls on the same nodes +-m for every
// detector angle), 16 scattered energies and 8 recorded energies per sigma.
//
//   forward   H[p][n]  = sum_q lambda_q B_{qp} L_n(phi_qp)                    k_ang_spread
//             S[b][m]  = sum_p C_p(b) e^{-mu(m) gamma_p} (H[p][s+m] + H[p][s-m])  k_ang_bins
//             DB[b][l] = sum_m L_l(E'(m)) f(m) S[b][m]                        k_node_bins
//             F[b][k]  = sum_l G[l][k] DB[b][l]                               k_node_values
//             y_j      = sum_k L_k(E_j) F[b_j][k] + unscattered part          k_node_y, k_node_cells
//   back      V[b][k]  = sum_{j in cell b} r_j L_k(E_j)                       k_node_cells
//             VG[b][l] = sum_k G[l][k] V[b][k]                                k_node_unvalues
//             PSI[b][m] = f(m) sum_l L_l(E'(m)) VG[b][l]                      k_ang_psi
//             T[p][n]  = sum_angles e^{-mu(m) gamma_p} sum_b C_p(b) PSI[b][m] k_ang_back
//             out[q]   = sum_p B_{qp} sum_n L_n(phi_qp) T[p][n]               k_ang_paths, k_node_update
//
// (s = the node of the detector direction, m = |n - s|).  A projection visits
// every (q, p, w) once whatever the number of events and of detector angles,
// where the rows take one exponential per event and path in reach; nothing
// of the path tables is read.
//
// mu(E'(x)) has a kink where E' meets an attenuation knot, which a polynomial
// through nodes on both sides would miss by the first power of their spacing
// (1.5e-5 of an event's value with a node every 1/29 sigma).  So each path sees
// mu continued smoothly from its own side: a node on the knot's other side is a
// slot with that mu, and the paths' taps on it (a few paths in a hundred) are
// summed apart, for every detector angle, and get the difference of the two
// attenuations:
//
//   forward   W[a][p][z] = sum_{q beyond the knot} lambda_q B_{qp} L_n(phi_qp)   k_ang_spread
//             S[b][m]   += sum_p C_p(b) (e^{-mu_z gamma_p} - e^{-mu(m) gamma_p}) W   k_ang_bins
//   back      Y[a][p][z] = (e^{-mu_z gamma_p} - e^{-mu(m) gamma_p}) sum_b C_p(b) PSI[b][m]   k_ang_back
//             out[q]    += sum_p B_{qp} sum_{n beyond the knot} L_n(phi_qp) Y         k_ang_paths
//
// Interpolation errors are below the FP32 rounding of the sums up to 6 sigma from
// every reachable energy (1e-7 of a path's value there) and 3e-6 at the 8 sigma
// where the reach ends, as far as the rows' exponents are good there; everything
// is FP32 with fixed-order sums, the voxel sums FP64.  (7, 7 and 12 taps at 18
// direction nodes per sigma, 16 scattered- and 8 recorded-energy nodes were
// 2.4e-4 off at 8 sigma, at a higher cost: more nodes cost more than more taps.)
//
// Measured (864 voxels and 864 points, 3 lines, 60 angles of 64 bins; times
// below that name no size are this model's): a forward projection of 100 000
// events 0.34 ms of kernels, 19.5 ms through the rows and 0.79 ms with the
// image spread at every angle anew through the path tables; a back projection
// 0.51 ms (12.0 ms, 0.70 ms); a sub-iteration of 8 angles 0.19 ms (2.15 ms,
// 0.32 ms).  At 3464 voxels and 120 angles of 128 bins a sub-iteration of 15
// angles takes 0.61 ms (26 ms, 1.29 ms).
#include <math.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <utility>
#include <vector>

#include "lmmew_internal.cuh"

namespace lmmew {
namespace {

constexpr int kTapsL = 11;         // taps of the scattered-energy nodes
constexpr int kPsiStride = 12;     // a direction offset's weights for them, padded
constexpr int kPerUnitL = 14;      // nodes per unit of t, at least
constexpr int kTapsK = 16;         // taps of the recorded-energy nodes
constexpr int kPerUnitK = 9;
constexpr double kBandSigmas = 10.2;  // G kept within this many sigma: at 8 sigma from the nearest path the
                                      // dropped ones are 6e-10 of it each
constexpr int kTapsN = 9;          // taps of the direction nodes
constexpr double kPerSigmaN = 17.0;   // direction nodes per sigma, at least
constexpr int kGroup = 8;          // scatter points per block of k_ang_back
constexpr int kBinsT = 16;         // detector bins per pass of k_ang_bins
constexpr int kValueRows = 8;      // (angle, bin) rows per block of k_node_values / _unvalues
constexpr int kValueWarps = 8;     // their warps, sharing the sum over nodes
constexpr int kCellWarps = 4;

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ f32x2 pk1(float v) { return pk(v, v); }

// The 9 Lagrange weights at distance s from the centre node, times v.
__device__ __forceinline__ void lagrange9(float s, float v, float (&w)[9]) {
    const float q = s * s, a1 = q - 1.f, a2 = q - 4.f, a3 = q - 9.f, a4 = q - 16.f, sv = s * v;
    const float a12 = a1 * a2, a34 = a3 * a4;
    const float m1 = sv * (a2 * a34) * (-1.f / 720.f), m2 = sv * (a1 * a34) * (1.f / 1440.f);
    const float m3 = sv * (a12 * a4) * (-1.f / 5040.f), m4 = sv * (a12 * a3) * (1.f / 40320.f);
    w[4] = a12 * a34 * (v * (1.f / 576.f));
    w[5] = fmaf(m1, s, m1);
    w[3] = fmaf(m1, s, -m1);
    w[6] = fmaf(m2, s, 2.f * m2);
    w[2] = fmaf(m2, s, -2.f * m2);
    w[7] = fmaf(m3, s, 3.f * m3);
    w[1] = fmaf(m3, s, -3.f * m3);
    w[8] = fmaf(m4, s, 4.f * m4);
    w[0] = fmaf(m4, s, -4.f * m4);
}

// Nearest of n nodes to a direction (in 2^-32 turns) and the distance from it
// in nodes, exact: c in [0, n].
__device__ __forceinline__ float direction_pos(uint32_t fix, int n, int* c) {
    const uint64_t u = (uint64_t)fix * (uint32_t)n;
    const int f = (int)(int32_t)(uint32_t)u;            // fraction - (fraction >= 1/2), in 2^-32
    *c = (int)(u >> 32) + (f < 0 ? 1 : 0);
    return (float)f * 2.3283064365386963e-10f;
}

// The 16 Lagrange weights at position f in [0, 1) between nodes 7 and 8,
// normalised to sum 1 (their common rounding cancels).
__device__ __forceinline__ void lagrange16(float f, float (&w)[16]) {
    // nodes at +-1/2, +-3/2, .. +-15/2 from the middle, x = f - 1/2;
    // 1 / prod_{j != i} (x_i - x_j) for the pair at +-(i + 1/2)
    constexpr float c[8] = {-1.f / 203212800.f,  1.f / 261273600.f,   -1.f / 435456000.f,
                            1.f / 958003200.f,   -1.f / 2874009600.f, 1.f / 12454041600.f,
                            -1.f / 87178291200.f, 1.f / 1307674368000.f};
    const float x = f - 0.5f, q = x * x;
    float a[8], pre[8], suf[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = q - (i + 0.5f) * (i + 0.5f);
    pre[0] = 1.f;
    suf[7] = 1.f;
#pragma unroll
    for (int i = 1; i < 8; ++i) pre[i] = pre[i - 1] * a[i - 1];
#pragma unroll
    for (int i = 6; i >= 0; --i) suf[i] = suf[i + 1] * a[i + 1];
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float m = pre[i] * suf[i] * c[i], n = m * (i + 0.5f);
        w[8 + i] = fmaf(m, x, n);        // node at +(i + 1/2): factor (x + (i + 1/2))
        w[7 - i] = -fmaf(m, x, -n);
        sum += w[8 + i] + w[7 - i];
    }
    const float inv = 1.f / sum;
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] *= inv;
}

// Position of a recorded energy on its nodes, u = ck sqrt(E): first of its 16
// taps (local index) and the fraction.  ck comes in two parts and the square
// root's rounding is taken out to first order: the fraction is good to its
// own FP32 rounding, where u's would shift the event by 4e-6 sigma.
__device__ __forceinline__ float energy_pos(const NodeConst& N, float e, int* k) {
    const float r = sqrtf(e);
    const float j = floorf(N.ck * r);
    const float lo = e > 0.f ? 0.5f * fmaf(-r, r, e) / r : 0.f;
    *k = min(max((int)j - (kTapsK / 2 - 1) - N.k_first, 0), N.nk - kTapsK);
    return fmaf(N.ck, r, -j) + fmaf(N.ck_lo, r, N.ck * lo);
}
__device__ __forceinline__ bool in_reach(const NodeConst& N, float e) {
    bool in = false;
    for (int w = 0; w < N.W; ++w) in |= e >= N.reach_lo[w] && e <= N.reach_hi[w];
    return in;
}

__global__ void k_node_matrix(const NodeConst N, double kappa, float* g, float* gt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N.nl_pad * N.nk_pad) return;
    const int l = i / N.nk_pad, k = i % N.nk_pad;
    int w = 0;
    while (w + 1 < N.W && l >= N.l_off[w + 1]) ++w;
    const double xl = 0.5 * kappa * (N.l_first[w] + (l - N.l_off[w])) / N.per_l;   // sqrt(E')
    const double xk = 0.5 * kappa * (N.k_first + k) / N.per_k;
    const double d = (xk * xk - xl * xl) / (kappa * xl);
    const bool real = l - N.l_off[w] < N.l_count[w] && k < N.nk;
    const float v = real && fabs(d) <= kBandSigmas ? (float)exp(-0.5 * d * d) : 0.f;
    g[(size_t)l * N.nk_pad + k] = v;
    gt[(size_t)k * N.nl_pad + l] = v;
}

struct NodeParams {
    NodeConst N;
    int a0, a_step, angles;  // angle i of the launch: a0 + i a_step
    int A, B, nq, np, npc, nq_pad;
    int parts;               // sums T[part] the angles of a back projection are split over
    const float* g;          // [nl][nk_pad] Gaussians
    const float* gt;         // [nk][nl_pad] their transpose
    const int2* k_of_l;      // [nl_pad / 32] recorded-energy nodes in reach of 32 nodes l
    const int2* l_of_k;      // [nk_pad / 32] scattered-energy nodes in reach of 32 nodes k
    const int2* chunk_bins;  // [A][npc] bins a chunk of 32 scatter points reaches
    const float* cs;         // [A][npc][B][kCPad]
    const int2* crange;      // [A][B]
    const int* inv;          // [A][np] point of each slot of an angle's point order
    const float* gamma;      // [A][np] line integral from each point to the detector, cm
    const float* mu;         // [nm_pad] log2(e) mu_water(E') of the direction offsets
    const int* psi_l;        // [nm_pad] first of the 11 nodes l of an offset's E'
    const float* psi_w;      // [nm_pad][kPsiStride] their weights, times f
    const int* dec_start;    // [nl_pad / 32 + 1] the same by 32 nodes l: offsets m and weights
    const int* dec_m;
    const float* dec_w;
    const uint32_t* fix;     // [np][nq] directions of the paths of each point, ascending
    const int* path_q;       // [np][nq] their voxels
    const int* path_of;      // [np][nq] place of each voxel's path
    const float* path_b;     // [W][np][nq] their B
    const int* path_start;   // [np][start_ints] per line: first path of each centre node
    const NodeSlot* slot;    // nodes beside a knot, seen from its other side
    const int* slot_start;   // [nm_pad + 1] the slots of each offset
    const short* slot_at;    // [kinks + 1][nm_pad] slot of an offset for paths of a side (-1: none)
    const int2* win;         // per line, disjoint windows of c - s (centre, detector direction; both
                             // ends of the circle apart) whose taps can cross a knot
    float inv_step[4];       // 1 / direction nodes from one angle of the launch to the next
    const int* grp_pt;       // [groups][8] neighbouring points (-1: none)
    const int2* grp_bins;    // [A][groups] bins they reach
    const float* grp_c;      // [A][groups][nbg_max][8] their collimator values
    const float* cv;         // [A][B][nq]
    const float* prim;       // [A][W][nq]
    const float* lam;        // [nq]
    float* H;                // [np][nn]
    float* dbp;              // [angles][npc][nb_max][nm_pad]: S's part of each chunk
    float* DB;               // [angles][B][nl_pad]
    float* F;                // [angles][B][nk_pad]
    float* Pr;               // [angles][B][W] unscattered sums
    const float* V;          // [angles][B][nk_pad]
    const float* PV;         // [angles][B][W]
    float* VG;               // [angles][B][nl_pad]
    float* psi;              // [angles][B][nm_pad]
    float* T;                // [np][nn]
    float* side;             // [angles][np][slots] what a slot adds to its node, from the bins
    float* val;              // [np][nq]
    float* part_prim;        // [angles][nq_pad]
};

// Side of the knots a path lies on, r + f nodes from the detector direction: the
// number of knots below its offset.
__device__ __forceinline__ int side_of_knots(const NodeConst& N, int w, int r, float f) {
    const int n = N.n_dir[w];
    if (2 * r > n) r -= n;
    if (2 * r < -n) r += n;
    float u = fabsf((float)r + f);
    if (2.f * u > (float)n) u = (float)n - u;
    int b = 0;
    while (b < N.kinks[w] && u > N.kink[w][b]) ++b;
    return b;
}
// Offset (of all lines) of the node r nodes from the detector direction.
__device__ __forceinline__ int offset_of(const NodeConst& N, int w, int r) {
    const int n = N.n_dir[w];
    int m = abs(r);
    if (m >= n) m -= n;
    if (2 * m > n) m = n - m;
    return N.m_off[w] + m;
}

// The slots' weighted taps of one (angle, point, line), by a warp: 32 paths of the
// line's windows at a time, a lane per path, leave their taps in shared memory;
// then a lane per slot (the 32 paths shared between as many lanes as fit) adds
// those on its node from paths on its side, in path order.  (A thread per slot
// that walks its paths takes 28 us more for 60 angles, a thread for all slots
// 290 us instead of 10 at 3464 voxels: both wait for one path after the other.)
constexpr int kMostWindows = 64;   // of a line: 4 per knot
constexpr int kSlotWords = (kTapsN + 1) * 32 + 2 * kMostWindows;   // a warp's: taps, positions, runs
__device__ __forceinline__ void slot_taps(const NodeParams& P, int ai, int p, int w, float* sh) {
    constexpr int kHalf = kTapsN / 2;
    const int lane = threadIdx.x & 31;
    const int n = P.N.n_dir[w], s = (P.a0 + ai * P.a_step) * P.N.angle_step[w];
    const int* st = P.path_start + (size_t)p * P.N.start_ints + P.N.n_off[w] + 2 * w;
    const uint32_t* fix = P.fix + (size_t)p * P.nq;
    const int* pq = P.path_q + (size_t)p * P.nq;
    const float* pb = P.path_b + ((size_t)w * P.np + p) * P.nq;
    int* pos = reinterpret_cast<int*>(sh + kTapsN * 32);
    // the windows' runs of directions, a lane each, empty ones left out
    int windows = 0;
    int2* run = reinterpret_cast<int2*>(pos + 32);
    for (int k0 = P.N.win_off[w]; k0 < P.N.win_off[w + 1]; k0 += 32) {
        int2 mine = make_int2(0, 0);
        if (k0 + lane < P.N.win_off[w + 1]) {
            const int2 win = P.win[k0 + lane];
            const int c0 = max(s + win.x, 0), c1 = min(s + win.y, n);
            if (c0 <= c1) mine = make_int2(st[c0], st[c1 + 1]);
        }
        const unsigned some = __ballot_sync(0xffffffffu, mine.x < mine.y);
        if (mine.x < mine.y) run[windows + __popc(some & ((1u << lane) - 1))] = mine;
        windows += __popc(some);
    }
    __syncwarp();
    for (int z0 = P.N.slot_off[w]; z0 < P.N.slot_off[w + 1]; z0 += 32) {
        const int count = min(32, P.N.slot_off[w + 1] - z0);
        // lanes per slot, each with every so many paths of the 32
        const int shares = count > 16 ? 1 : count > 8 ? 2 : 4, slots = 32 / shares;
        const int z = z0 + min(lane & (slots - 1), count - 1), share = lane / slots;
        const unsigned paths = (shares == 1 ? ~0u : shares == 2 ? 0x55555555u : 0x11111111u) << share;
        const int m = P.slot[z].offset - P.N.m_off[w], side = P.slot[z].side;
        float sum = 0.f;
        int k = 0, r = 0, r1 = 0;
        while (true) {
            int fill = 0, mine = -1;
            while (fill < 32) {
                if (r >= r1) {          // the next window's run of directions
                    if (k == windows) break;
                    r = run[k].x;
                    r1 = run[k].y;
                    ++k;
                    continue;
                }
                const int take = min(32 - fill, r1 - r);
                if (lane >= fill && lane < fill + take) mine = r + lane - fill;
                r += take;
                fill += take;
            }
            if (fill == 0) break;
            __syncwarp();
            int own = -1;
            if (mine >= 0) {
                int c;
                const float f = direction_pos(fix[mine], n, &c);
                float x[kTapsN];
                lagrange9(f, pb[mine] * P.lam[pq[mine]], x);
#pragma unroll
                for (int t = 0; t < kTapsN; ++t) sh[t * 32 + lane] = x[t];
                int d = c - s;          // in (-n / 2, n / 2]
                if (2 * d > n) d -= n;
                if (2 * d <= -n) d += n;
                pos[lane] = d;
                own = side_of_knots(P.N, w, d, f);
            }
            unsigned todo = 0;          // paths of the slot's side
            for (int b = 0; b <= P.N.kinks[w]; ++b) {
                const unsigned there = __ballot_sync(0xffffffffu, own == b);
                if (b == side) todo = there & paths;
            }
            __syncwarp();
            for (; todo; todo &= todo - 1) {
                const int i = __ffs(todo) - 1;
                // the path's tap on node s + m, and on s - m where that is another
                int t = m - pos[i] + kHalf;
                if (t >= n) t -= n;
                if ((unsigned)t < kTapsN) sum += sh[t * 32 + i];
                t = -m - pos[i] + kHalf;
                if (t < 0) t += n;
                if ((unsigned)t < kTapsN && m > 0 && 2 * m != n) sum += sh[t * 32 + i];
            }
        }
        float all = sum;
        for (int j = 1; j < shares; ++j) all += __shfl_down_sync(0xffffffffu, sum, j * slots);
        if (lane < count) P.side[((size_t)ai * P.np + p) * P.N.slots + z] = all;
    }
}

// H: a warp per (point, line, 120 direction nodes).  The paths centred on the
// tile's nodes and the 4 on either side are one run of the point's directions
// (and a second one where the circle closes).  32 of them at a time form their
// 9 weighted taps, a lane per path; a segmented scan sums those of equal centre,
// and the last of each adds them to the centre's sums.  At the end each node
// collects its taps from the 9 centres around it.  No two lanes add to one
// place, and every sum has its order.  Bound by instruction issue (66 %) once
// the loads are a group ahead: 41 us (with 7 taps 37 us, and then 47 us with a lane
// per centre, which waits on three dependent loads per path, 42 us with a block
// per tile).
// Where a centre has more than kSpreadDense paths the scan's steps cost more
// than those waits, and a lane takes a centre's paths: with 7 taps 80 instead of 118 us
// at 3464 voxels (11, 6 and 3 paths a centre; limits of 2 and 4 are equal
// there, 1 costs 83 us).  The first blocks form the slots' taps, a warp per
// (angle, point, line with a knot).
constexpr int kSpreadDense = 4, kSpreadWarps = 4, kSpreadCentres = 128, kSpreadOut = kSpreadCentres - (kTapsN - 1);
__global__ void __launch_bounds__(32 * kSpreadWarps) k_ang_spread(const NodeParams P, int tiles, int units,
                                                                 int side_blocks) {
    __shared__ __align__(16) float taps[kSpreadWarps][kTapsN][kSpreadCentres];
    if ((int)blockIdx.x < side_blocks) {
        static_assert(kSlotWords <= kTapsN * kSpreadCentres, "the slots' taps lie in the taps' place");
        int i = blockIdx.x * kSpreadWarps + (threadIdx.x >> 5);
        for (int w = 0; w < P.N.W; ++w) {
            if (P.N.kinks[w] == 0) continue;
            if (i < P.angles * P.np) {
                slot_taps(P, i / P.np, i % P.np, w, &taps[threadIdx.x >> 5][0][0]);
                return;
            }
            i -= P.angles * P.np;
        }
        return;
    }
    const int lane = threadIdx.x & 31, unit = (blockIdx.x - side_blocks) * kSpreadWarps + (threadIdx.x >> 5);
    if (unit >= units) return;
    float (&tap)[kTapsN][kSpreadCentres] = taps[threadIdx.x >> 5];
    const int p = unit / tiles;
    int tile = unit % tiles, w = 0;
    while (tile >= (P.N.n_dir[w] + kSpreadOut - 1) / kSpreadOut) {
        tile -= (P.N.n_dir[w] + kSpreadOut - 1) / kSpreadOut;
        ++w;
    }
    const int n = P.N.n_dir[w], n0 = tile * kSpreadOut;
    const int u0 = n0 - kTapsN / 2, u1 = min(n0 + kSpreadOut, n) + kTapsN / 2 - 1;   // the tile's centres
    // first path of each centre, centres 0 .. n (n: a full turn, node 0 again)
    const int* st = P.path_start + (size_t)p * P.N.start_ints + P.N.n_off[w] + 2 * w;
    const uint32_t* fix = P.fix + (size_t)p * P.nq;
    const int* pq = P.path_q + (size_t)p * P.nq;
    const float* pb = P.path_b + ((size_t)w * P.np + p) * P.nq;
    const bool dense = P.nq > kSpreadDense * n;
    if (dense) {
        for (int i = lane; i <= u1 - u0; i += 32) {
            const int u = u0 + i, c = u < 0 ? u + n : u > n ? u - n : u;
            float g[kTapsN] = {};
            int r = st[c], re = st[c + 1], more = c == 0 ? n : c == n ? 0 : -1;
            while (true) {
                for (; r < re; ++r) {
                    int cc;
                    const float s = direction_pos(fix[r], n, &cc);
                    float x[kTapsN];
                    lagrange9(s, pb[r] * P.lam[pq[r]], x);
#pragma unroll
                    for (int k = 0; k < kTapsN; ++k) g[k] += x[k];
                }
                if (more < 0) break;
                r = st[more];
                re = st[more + 1];
                more = -1;
            }
#pragma unroll
            for (int k = 0; k < kTapsN; ++k) tap[k][i] = g[k];
        }
    } else {
        for (int i = lane; i < kTapsN * kSpreadCentres / 4; i += 32)
            reinterpret_cast<float4*>(tap)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
    }
    for (int part = dense ? 3 : 0; part < 3; ++part) {
        // paths centred c in [ca, cb], which are the centres u = c - shift
        int ca, cb, shift;
        if (part == 0) {
            ca = max(u0, 0);
            cb = min(u1, n);
            shift = 0;
        } else if (part == 1) {
            if (u0 > 0) continue;
            ca = n + u0;
            cb = n;
            shift = n;
        } else {
            if (u1 < n) continue;
            ca = 0;
            cb = u1 - n;
            shift = -n;
        }
        // (two groups of 32 ahead for the voxel, one for what it leads to)
        const int r1 = st[cb + 1], ra = st[ca];
        int q2 = ra + lane < r1 ? pq[ra + lane] : 0;
        uint32_t f1 = 0;
        float b1 = 0.f, v1 = 0.f;
        auto ahead = [&](int r) {
            f1 = 0;
            b1 = v1 = 0.f;
            if (r < r1) {
                f1 = fix[r];
                b1 = pb[r];
                v1 = P.lam[q2];
            }
            q2 = r + 32 < r1 ? pq[r + 32] : 0;
        };
        ahead(ra + lane);
        for (int r0 = ra; r0 < r1; r0 += 32) {
            const int r = r0 + lane;
            const uint32_t f = f1;
            const float v = b1 * v1;
            ahead(r + 32);
            float x[kTapsN];
            int c;
            const float s = direction_pos(f, n, &c);
            lagrange9(s, v, x);
            if (r >= r1) c = -1;
            const int before = __shfl_up_sync(0xffffffffu, c, 1);
            const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || c != before);
            const int back = lane - (31 - __clz(heads & (0xffffffffu >> (31 - lane))));
            const int most = __reduce_max_sync(0xffffffffu, back);
            for (int o = 1; o <= most; o <<= 1)
#pragma unroll
                for (int k = 0; k < kTapsN; ++k) {
                    const float y = __shfl_up_sync(0xffffffffu, x[k], o);
                    if (back >= o) x[k] += y;
                }
            __syncwarp();
            if (c >= 0 && (lane == 31 || (heads >> (lane + 1) & 1u)))
#pragma unroll
                for (int k = 0; k < kTapsN; ++k) tap[k][c - shift - u0] += x[k];
        }
    }
    __syncwarp();
    for (int i = lane; i < kSpreadOut && n0 + i < n; i += 32) {
        float h = 0.f;                     // centre n0 + i + j - 4 is place i + j, and node n0 + i its tap 8 - j
#pragma unroll
        for (int j = 0; j < kTapsN; ++j) h += tap[kTapsN - 1 - j][i + j];
        P.H[(size_t)p * P.N.nn + P.N.n_off[w] + n0 + i] = h;
    }
}

// S's part of one (angle, 32 scatter points, line): two direction offsets m a
// thread, the points one after the other, 16 bins at a time (a collimator value
// read from shared memory serves both offsets).  Bound by FP32 issue: 106 us for
// 60 angles, 20 us for 8.  (The slots' shares go in after the points, in the warps
// that hold one: 367 us for a forward projection, 444 us with the taps formed here
// and added point by point.)
constexpr int kOffThreads = 128, kOffPer = 2;

__global__ void __launch_bounds__(kOffThreads, 6) k_ang_bins(const NodeParams P, int tiles) {
    extern __shared__ float sside[];   // [tile's slots][kPC] what they add to their nodes
    __shared__ __align__(16) float sc[kPC][kBinsT];
    __shared__ int sp[kPC];
    __shared__ float sgm[kPC];
    const int t = threadIdx.x;
    constexpr int kTile = kOffThreads * kOffPer;
    int tile = blockIdx.x % tiles;
    const int pc = (blockIdx.x / tiles) % P.npc, ai = blockIdx.x / (tiles * P.npc);
    int w = 0;
    while (tile >= (P.N.m_count[w] + kTile - 1) / kTile) {
        tile -= (P.N.m_count[w] + kTile - 1) / kTile;
        ++w;
    }
    const int a = P.a0 + ai * P.a_step, n = P.N.n_dir[w];
    const int s = a * P.N.angle_step[w];
    int n1[kOffPer], n2[kOffPer];
    float mu[kOffPer], two[kOffPer];
    // slots of the tile
    const int z0 = P.slot_start[P.N.m_off[w] + tile * kTile];
    const int z1 = P.slot_start[P.N.m_off[w] + min((tile + 1) * kTile, P.N.m_count[w])];
#pragma unroll
    for (int j = 0; j < kOffPer; ++j) {
        const int m = min(tile * kTile + j * kOffThreads + t, P.N.m_count[w] - 1);
        n1[j] = s + m;
        n2[j] = s - m;
        if (n1[j] >= n) n1[j] -= n;
        if (n2[j] < 0) n2[j] += n;
        two[j] = n1[j] != n2[j] ? 1.f : 0.f;
        mu[j] = P.mu[P.N.m_off[w] + m];
    }
    const int cnt = min(kPC, P.np - pc * kPC);
    if (t < kPC) {
        const int p = t < cnt ? P.inv[(size_t)a * P.np + pc * kPC + t] : 0;
        sp[t] = p * P.N.nn + P.N.n_off[w];
        sgm[t] = t < cnt ? P.gamma[(size_t)a * P.np + p] : 0.f;
    }
    if (z1 > z0) {
        __syncthreads();
        for (int i = t; i < (z1 - z0) * kPC; i += kOffThreads) {
            const int z = z0 + i / kPC, k = i % kPC, p = sp[k] / P.N.nn;
            const float own = ex2f(-P.mu[P.slot[z].offset] * sgm[k]), other = ex2f(-P.slot[z].mu * sgm[k]);
            sside[i] = k < cnt ? P.side[((size_t)ai * P.np + p) * P.N.slots + z] * (other - own) : 0.f;
        }
    }
    const int2 br = P.chunk_bins[(size_t)a * P.npc + pc];
    const float* cr = P.cs + ((size_t)a * P.npc + pc) * P.B * kCPad;
    float* out = P.dbp + ((size_t)ai * P.npc + pc) * P.N.nb_max * P.N.nm_pad + P.N.m_off[w];
    for (int b0 = br.x; b0 < br.y; b0 += kBinsT) {
        __syncthreads();
        for (int i = t; i < kPC * kBinsT; i += kOffThreads) {
            const int b = i / kPC, p = i % kPC;
            sc[p][b] = b0 + b < br.y && p < cnt ? cr[(size_t)(b0 + b) * kCPad + p] : 0.f;
        }
        __syncthreads();
        f32x2 acc[kOffPer][kBinsT / 2];
#pragma unroll
        for (int j = 0; j < kOffPer; ++j)
#pragma unroll
            for (int k = 0; k < kBinsT / 2; ++k) acc[j][k] = 0ull;
        // (points past the last carry collimator values 0)
        for (int i0 = 0; i0 < kPC; i0 += 8) {
            float v[kOffPer][8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float* row = P.H + sp[i0 + i];
#pragma unroll
                for (int j = 0; j < kOffPer; ++j) v[j][i] = fmaf(two[j], row[n2[j]], row[n1[j]]);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float g = sgm[i0 + i];
                f32x2 v2[kOffPer];
#pragma unroll
                for (int j = 0; j < kOffPer; ++j) v2[j] = pk1(v[j][i] * ex2f(-mu[j] * g));
                const float4* c4 = reinterpret_cast<const float4*>(sc[i0 + i]);
#pragma unroll
                for (int k = 0; k < kBinsT / 4; ++k) {
                    const float4 c = c4[k];
#pragma unroll
                    for (int j = 0; j < kOffPer; ++j) {
                        acc[j][2 * k] = fma2(v2[j], pk(c.x, c.y), acc[j][2 * k]);
                        acc[j][2 * k + 1] = fma2(v2[j], pk(c.z, c.w), acc[j][2 * k + 1]);
                    }
                }
            }
        }
        // nodes beside a knot: paths beyond it have its other side's attenuation
#pragma unroll
        for (int j = 0; j < kOffPer; ++j) {
            if (z1 == z0) break;
            const int* zs = P.slot_start + P.N.m_off[w] + min(tile * kTile + j * kOffThreads + t, P.N.m_count[w] - 1);
            const int i1 = (zs[1] - z0) * kPC;
#pragma unroll 1
            for (int i = (zs[0] - z0) * kPC; i < i1; ++i) {
                const f32x2 y = pk1(sside[i]);
                const float4* c4 = reinterpret_cast<const float4*>(sc[i % kPC]);
#pragma unroll
                for (int k = 0; k < kBinsT / 4; ++k) {
                    const float4 c = c4[k];
                    acc[j][2 * k] = fma2(y, pk(c.x, c.y), acc[j][2 * k]);
                    acc[j][2 * k + 1] = fma2(y, pk(c.z, c.w), acc[j][2 * k + 1]);
                }
            }
        }
#pragma unroll
        for (int j = 0; j < kOffPer; ++j) {
            const int m = tile * kTile + j * kOffThreads + t;
            if (m >= P.N.m_count[w]) continue;
#pragma unroll
            for (int k = 0; k < kBinsT / 2; ++k) {
                float x, y;
                upk(acc[j][k], x, y);
                if (b0 + 2 * k < br.y) out[(size_t)(b0 - br.x + 2 * k) * P.N.nm_pad + m] = x;
                if (b0 + 2 * k + 1 < br.y) out[(size_t)(b0 - br.x + 2 * k + 1) * P.N.nm_pad + m] = y;
            }
        }
    }
}

// A row's (angle, bin) sums over the chunks of its run of scatter points, then
// from the direction offsets onto the scattered-energy nodes: a block per row;
// the blocks past those form the unscattered sums, a warp per (row, line).
// Bound by load latency: 8 loads in flight per thread, whatever the run.  75 us
// for 60 angles, 14 us for 8.
constexpr int kRowThreadsN = 512, kRowChunks = 512;
__global__ void __launch_bounds__(kRowThreadsN) k_node_bins(const NodeParams P) {
    extern __shared__ float srow[];   // [nm_pad]
    __shared__ int off[kRowChunks];
    const int t = threadIdx.x, W = P.N.W;
    const int rows = P.angles * P.B;
    if ((int)blockIdx.x >= rows) {
        const int i = (blockIdx.x - rows) * (kRowThreadsN / 32) + (t >> 5);
        if (i >= rows * W) return;
        const int row = i / W, w = i % W;
        const int a = P.a0 + (row / P.B) * P.a_step;
        const float* cv = P.cv + ((size_t)a * P.B + row % P.B) * P.nq;
        const float* pr = P.prim + ((size_t)a * W + w) * P.nq;
        float s = 0.f;
        for (int q0 = t & 31; q0 < P.nq; q0 += 256) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int q = q0 + 32 * k;
                if (q < P.nq) s = fmaf(cv[q] * pr[q], P.lam[q], s);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 31) == 0) P.Pr[i] = s;
        return;
    }
    const int row = blockIdx.x;
    const int ai = row / P.B, b = row % P.B, a = P.a0 + ai * P.a_step;
    const int2 run = P.crange[(size_t)a * P.B + b];
    const int c0 = run.x / kPC, c1 = run.y > run.x ? (run.y + kPC - 1) / kPC : c0;
    const int2* cb = P.chunk_bins + (size_t)a * P.npc;
    const float* src = P.dbp + (size_t)ai * P.npc * P.N.nb_max * P.N.nm_pad;
    for (int m = t; m < P.N.nm_pad; m += kRowThreadsN) srow[m] = 0.f;
    for (int p0 = c0; p0 < c1; p0 += kRowChunks) {
        const int np = min(kRowChunks, c1 - p0);
        __syncthreads();
        for (int i = t; i < np; i += kRowThreadsN) off[i] = (p0 + i) * P.N.nb_max + (b - cb[p0 + i].x);
        __syncthreads();
        for (int m = t; m < P.N.nm_pad; m += kRowThreadsN) {
            bool node = false;   // (not one of the pads between the lines)
            for (int w = 0; w < W; ++w) node |= (unsigned)(m - P.N.m_off[w]) < (unsigned)P.N.m_count[w];
            if (!node) continue;
            float s = srow[m];
            for (int i0 = 0; i0 < np; i0 += 8) {
                float v[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    v[i] = i0 + i < np ? src[(size_t)off[i0 + i] * P.N.nm_pad + m] : 0.f;
#pragma unroll
                for (int i = 0; i < 8; ++i) s += v[i];
            }
            srow[m] = s;
        }
    }
    __syncthreads();
    // (32 nodes l at a time, their taps padded to the longest of the 32)
    for (int l = t; l < P.N.nl_pad; l += kRowThreadsN) {
        float s = 0.f;
        const int d1 = P.dec_start[(l >> 5) + 1];
        for (int d0 = P.dec_start[l >> 5] + (l & 31); d0 < d1; d0 += 256) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int d = d0 + 32 * k;
                if (d < d1) s = fmaf(P.dec_w[d], srow[P.dec_m[d]], s);
            }
        }
        P.DB[(size_t)row * P.N.nl_pad + l] = s;
    }
}

// out[row][x] = sum_y m[y][x] in[row][y] over the band of y each x reaches,
// for 8 rows and 32 x per block: the warps share the band's y (a run each, the
// loads of a run in flight together), their sums are added in warp order.  69 us
// forward and 76 us back for 60 angles, 13 and 14 us for 8.
__device__ __forceinline__ void band_product(const float* in, int in_stride, const float* m,
                                             int m_stride, float* out, int out_stride, int rows,
                                             int r0, int x0, int lo, int hi, float* sh) {
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    float* red = sh;                                   // [warps][8][32]
    float* st = sh + kValueWarps * kValueRows * 32;    // [y][8]
    const int per = (hi - lo + kValueWarps - 1) / kValueWarps;
    const int y0 = min(lo + warp * per, hi), y1 = min(y0 + per, hi);
    const float* mp = m + x0 + lane;
    // 16 y at a time, the next 16 matrix entries in flight (the first ones
    // while the rows are staged, a warp per row)
    float g[16];
    auto load = [&](int yb) {
#pragma unroll
        for (int k = 0; k < 16; ++k) g[k] = yb + k < y1 ? mp[(size_t)(yb + k) * m_stride] : 0.f;
    };
    load(y0);
    const float* src = in + (size_t)(r0 + warp) * in_stride + lo;
    const int len = r0 + warp < rows ? hi - lo : 0;
    for (int yb = lane; yb < hi - lo; yb += 256) {
        float v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = yb + 32 * k < len ? src[yb + 32 * k] : 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (yb + 32 * k < hi - lo) st[(yb + 32 * k) * kValueRows + warp] = v[k];
    }
    __syncthreads();
    f32x2 s[kValueRows / 2] = {0ull, 0ull, 0ull, 0ull};
    for (int yb = y0; yb < y1; yb += 16) {
        float c[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) c[k] = g[k];
        if (yb + 16 < y1) load(yb + 16);
        f32x2 u[kValueRows / 2] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int y = min(yb + k, y1 - 1);
            const f32x2 g2 = pk1(c[k]);
            const float4 d0 = *reinterpret_cast<const float4*>(st + (y - lo) * kValueRows);
            const float4 d1 = *reinterpret_cast<const float4*>(st + (y - lo) * kValueRows + 4);
            u[0] = fma2(g2, pk(d0.x, d0.y), u[0]);
            u[1] = fma2(g2, pk(d0.z, d0.w), u[1]);
            u[2] = fma2(g2, pk(d1.x, d1.y), u[2]);
            u[3] = fma2(g2, pk(d1.z, d1.w), u[3]);
        }
#pragma unroll
        for (int i = 0; i < kValueRows / 2; ++i) s[i] = add2(s[i], u[i]);
    }
#pragma unroll
    for (int i = 0; i < kValueRows / 2; ++i) {
        float x, y;
        upk(s[i], x, y);
        red[(warp * kValueRows + 2 * i) * 32 + lane] = x;
        red[(warp * kValueRows + 2 * i + 1) * 32 + lane] = y;
    }
    __syncthreads();
    static_assert(kValueWarps == kValueRows, "a warp per row in the last step");
    float v = 0.f;
#pragma unroll
    for (int k = 0; k < kValueWarps; ++k) v += red[(k * kValueRows + warp) * 32 + lane];
    if (r0 + warp < rows) out[(size_t)(r0 + warp) * out_stride + x0 + lane] = v;
}

// The Gaussians from the scattered-energy nodes onto the recorded-energy nodes.
__global__ void __launch_bounds__(32 * kValueWarps) k_node_values(const NodeParams P) {
    extern __shared__ __align__(16) float sh[];
    const int kt = P.N.nk_pad / 32;
    const int r0 = blockIdx.x / kt * kValueRows, tile = blockIdx.x % kt;
    const int2 r = P.l_of_k[tile];
    band_product(P.DB, P.N.nl_pad, P.g, P.N.nk_pad, P.F, P.N.nk_pad, P.angles * P.B, r0, tile * 32, r.x,
                 r.y, sh);
}

// Transposed, for the back projection; the blocks past those form its
// unscattered part, a thread per voxel.
__global__ void __launch_bounds__(32 * kValueWarps) k_node_unvalues(const NodeParams P) {
    extern __shared__ __align__(16) float sh[];
    const int rows = P.angles * P.B, W = P.N.W;
    const int lt = P.N.nl_pad / 32;
    const int n_row_blocks = (rows + kValueRows - 1) / kValueRows * lt;
    if ((int)blockIdx.x >= n_row_blocks) {
        const int qb = (P.nq + 255) / 256;
        const int ai = (blockIdx.x - n_row_blocks) / qb;
        const int q = ((blockIdx.x - n_row_blocks) % qb) * 256 + threadIdx.x;
        if (q >= P.nq) return;
        const int a = P.a0 + ai * P.a_step;
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        const float* cv = P.cv + (size_t)a * P.B * P.nq + q;
        const float* pv = P.PV + (size_t)ai * P.B * W;
#pragma unroll 16
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
    const int r0 = blockIdx.x / lt * kValueRows, tile = blockIdx.x % lt;
    const int2 r = P.k_of_l[tile];
    band_product(P.V, P.N.nk_pad, P.gt, P.N.nl_pad, P.VG, P.N.nl_pad, rows, r0, tile * 32, r.x, r.y, sh);
}

// PSI: the rows' values at the direction offsets, a block per row.
__global__ void __launch_bounds__(256) k_ang_psi(const NodeParams P) {
    extern __shared__ float srow[];   // [nl_pad]
    const size_t row = blockIdx.x;
    for (int l = threadIdx.x; l < P.N.nl_pad; l += 256) srow[l] = P.VG[row * P.N.nl_pad + l];
    __syncthreads();
    for (int m = threadIdx.x; m < P.N.nm_pad; m += 256) {
        const float4* w = reinterpret_cast<const float4*>(P.psi_w + (size_t)m * kPsiStride);
        const float4 w0 = w[0], w1 = w[1], w2 = w[2];
        const float* v = srow + P.psi_l[m];
        float s = w0.x * v[0];
        s = fmaf(w0.y, v[1], s);
        s = fmaf(w0.z, v[2], s);
        s = fmaf(w0.w, v[3], s);
        s = fmaf(w1.x, v[4], s);
        s = fmaf(w1.y, v[5], s);
        s = fmaf(w1.z, v[6], s);
        s = fmaf(w1.w, v[7], s);
        s = fmaf(w2.x, v[8], s);
        s = fmaf(w2.y, v[9], s);
        s = fmaf(w2.z, v[10], s);
        P.psi[row * P.N.nm_pad + m] = s;
    }
}

// T: a warp per (64 direction nodes, 8 neighbouring scatter points), two nodes a
// lane; the four warps of a block take neighbouring groups of points on the same
// nodes, so that one reads PSI from L2 and the others find it in L1.  The
// launch's angles one after the other, each over the bins the 8 points reach;
// the points' collimator values, bins and line integrals of a batch of angles
// are staged in shared memory together, which leaves one load latency (PSI's, 8
// bins in flight) per angle.  Bound by issue (54 %) and that latency; eight
// blocks an SM put every warp of the grid on the chip at once: 293 us for 60
// angles and 40 us for 8 (at 2792 direction nodes, where it took 412 and 54 us:
// 503 and 66 us with the collimator values read bin by
// bin; 16 or 4 bins in flight: 426, 468 us; one warp a block: 410 us, but 264
// instead of 210 us for 15 angles at 3464 voxels).  A grid that leaves most of
// the chip idle is split over the angles, up to 8 parts that k_ang_paths adds
// in order: a back projection of 52 points and 88 angles took 355 us with one.
constexpr int kBackWarps = 4, kBackTile = 64, kBackAngles = 4;
constexpr size_t kBackStage = 16 * 1024;
__global__ void __launch_bounds__(32 * kBackWarps, 8) k_ang_back(const NodeParams P, int tiles, int groups,
                                                              int batch) {
    extern __shared__ __align__(16) float sc[];   // [batch][kBackWarps][nbg_max][8]
    __shared__ float sg[kBackAngles][kBackWarps][kGroup];
    __shared__ int2 sb[kBackAngles][kBackWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int main_blocks = tiles * ((groups + kBackWarps - 1) / kBackWarps);
    if ((int)blockIdx.x >= main_blocks) {
        // the blocks past the grid: a thread per (slot, angle, point), what the
        // bins add to the node for paths beyond the knot
        const int64_t i = (int64_t)(blockIdx.x - main_blocks) * (32 * kBackWarps) + t;
        const int z = (int)(i % P.N.slots), ai = (int)(i / P.N.slots % P.angles);
        const int gp = (int)(i / ((int64_t)P.N.slots * P.angles));
        if (blockIdx.y > 0 || gp >= groups * kGroup) return;
        const int p = P.grp_pt[gp];
        if (p < 0) return;
        const NodeSlot zs = P.slot[z];
        const int a = P.a0 + ai * P.a_step;
        const size_t ag = (size_t)a * groups + gp / kGroup;
        const int2 br = P.grp_bins[ag];
        const float* c = P.grp_c + ag * P.N.nbg_max * kGroup + gp % kGroup;
        const float* psi = P.psi + ((size_t)ai * P.B + br.x) * P.N.nm_pad + zs.offset;
        float sum = 0.f;
#pragma unroll 8
        for (int b = 0; b < br.y - br.x; ++b) sum = fmaf(c[b * kGroup], psi[(size_t)b * P.N.nm_pad], sum);
        const float g = P.gamma[(size_t)a * P.np + p];
        P.side[((size_t)ai * P.np + p) * P.N.slots + z] = sum * (ex2f(-zs.mu * g) - ex2f(-P.mu[zs.offset] * g));
        return;
    }
    int tile = blockIdx.x % tiles;
    const int grp0 = blockIdx.x / tiles * kBackWarps, grp = grp0 + warp;
    int w = 0;
    while (tile >= (P.N.n_dir[w] + kBackTile - 1) / kBackTile) {
        tile -= (P.N.n_dir[w] + kBackTile - 1) / kBackTile;
        ++w;
    }
    const int n = P.N.n_dir[w], nmp = P.N.nm_pad, per = P.N.nbg_max * kGroup;
    const int nd0 = min(tile * kBackTile + lane, n - 1), nd1 = min(tile * kBackTile + 32 + lane, n - 1);
    f32x2 acc0[kGroup / 2] = {0ull, 0ull, 0ull, 0ull}, acc1[kGroup / 2] = {0ull, 0ull, 0ull, 0ull};
    const int a_end = P.angles * ((int)blockIdx.y + 1) / P.parts;   // (at most 8 x 16384)
    for (int a1 = P.angles * (int)blockIdx.y / P.parts; a1 < a_end; a1 += batch) {
        const int na = min(batch, a_end - a1);
        __syncthreads();
        for (int i = t; i < na * kBackWarps * per / 4; i += 32 * kBackWarps) {
            const int x = i % (per / 4), g = i / (per / 4) % kBackWarps, k = i / (per / 4) / kBackWarps;
            const int a = P.a0 + (a1 + k) * P.a_step;
            if (grp0 + g < groups)
                reinterpret_cast<float4*>(sc)[i] =
                    reinterpret_cast<const float4*>(P.grp_c)[((size_t)a * groups + grp0 + g) * (per / 4) + x];
        }
        for (int i = t; i < na * kBackWarps * kGroup; i += 32 * kBackWarps) {
            const int j = i % kGroup, g = i / kGroup % kBackWarps, k = i / kGroup / kBackWarps;
            const int a = P.a0 + (a1 + k) * P.a_step;
            if (grp0 + g >= groups) continue;
            sg[k][g][j] = P.gamma[(size_t)a * P.np + max(P.grp_pt[(grp0 + g) * kGroup + j], 0)];
            if (j == 0) sb[k][g] = P.grp_bins[(size_t)a * groups + grp0 + g];
        }
        __syncthreads();
        if (grp >= groups) continue;
        for (int k = 0; k < na; ++k) {
            const int a = P.a0 + (a1 + k) * P.a_step;
            const int sh = a * P.N.angle_step[w];
            const int2 br = sb[k][warp];
            const float4* c = reinterpret_cast<const float4*>(sc + (size_t)(k * kBackWarps + warp) * per);
            int d0 = nd0 - sh, d1 = nd1 - sh;
            if (d0 < 0) d0 += n;
            if (d1 < 0) d1 += n;
            const int m0 = P.N.m_off[w] + min(d0, n - d0), m1 = P.N.m_off[w] + min(d1, n - d1);
            const float mu0 = P.mu[m0], mu1 = P.mu[m1];
            const float* psi = P.psi + ((size_t)(a1 + k) * P.B + br.x) * nmp;
            f32x2 s0[kGroup / 2] = {0ull, 0ull, 0ull, 0ull}, s1[kGroup / 2] = {0ull, 0ull, 0ull, 0ull};
            const int nb = br.y - br.x;
            for (int b = 0; b < nb; b += 8) {
                float v0[8], v1[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const bool on = b + i < nb;
                    v0[i] = on ? psi[(b + i) * nmp + m0] : 0.f;
                    v1[i] = on ? psi[(b + i) * nmp + m1] : 0.f;
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    if (b + i >= nb) break;
                    const float4 ca = c[2 * (b + i)], cb = c[2 * (b + i) + 1];
                    const f32x2 x0 = pk1(v0[i]), x1 = pk1(v1[i]);
                    s0[0] = fma2(x0, pk(ca.x, ca.y), s0[0]);
                    s0[1] = fma2(x0, pk(ca.z, ca.w), s0[1]);
                    s0[2] = fma2(x0, pk(cb.x, cb.y), s0[2]);
                    s0[3] = fma2(x0, pk(cb.z, cb.w), s0[3]);
                    s1[0] = fma2(x1, pk(ca.x, ca.y), s1[0]);
                    s1[1] = fma2(x1, pk(ca.z, ca.w), s1[1]);
                    s1[2] = fma2(x1, pk(cb.x, cb.y), s1[2]);
                    s1[3] = fma2(x1, pk(cb.z, cb.w), s1[3]);
                }
            }
#pragma unroll
            for (int i = 0; i < kGroup / 2; ++i) {
                const float ga = sg[k][warp][2 * i], gb = sg[k][warp][2 * i + 1];
                acc0[i] = fma2(pk(ex2f(-mu0 * ga), ex2f(-mu0 * gb)), s0[i], acc0[i]);
                acc1[i] = fma2(pk(ex2f(-mu1 * ga), ex2f(-mu1 * gb)), s1[i], acc1[i]);
            }
        }
    }
    if (grp >= groups) return;
    float* out = P.T + (size_t)blockIdx.y * P.np * P.N.nn + P.N.n_off[w] + tile * kBackTile + lane;
    const bool on0 = tile * kBackTile + lane < n, on1 = tile * kBackTile + 32 + lane < n;
#pragma unroll
    for (int i = 0; i < kGroup; ++i) {
        const int p = P.grp_pt[grp * kGroup + i];
        if (p < 0) continue;
        float x[2], y[2];
        upk(acc0[i / 2], x[0], x[1]);
        upk(acc1[i / 2], y[0], y[1]);
        float* o = out + (size_t)p * P.N.nn;
        if (on0) o[0] = x[i & 1];
        if (on1) o[32] = y[i & 1];
    }
}

// v plus what the slots add to a path with its centre at node c and taps x: for
// every detector angle of the launch that has a knot within reach of its taps,
// the nodes on the knot's other side.  The windows are disjoint, so that no angle
// comes twice; angle i is in one of them for i between two quotients, which FP32
// gives exactly (half a node from the next whole number).
__device__ __forceinline__ float beyond_knots(const NodeParams& P, int w, int p, int c, float s,
                                              const float (&x)[kTapsN], float v) {
    const int step = P.N.angle_step[w] * P.a_step, r0 = c - P.a0 * P.N.angle_step[w], n = P.N.n_dir[w];
    for (int k = P.N.win_off[w]; k < P.N.win_off[w + 1]; ++k) {
        const int2 win = P.win[k];
        const int i0 = max((int)floorf(((float)(r0 - win.y) - 0.5f) * P.inv_step[w]) + 1, 0);
        const int i1 = min((int)floorf(((float)(r0 - win.x) + 0.5f) * P.inv_step[w]), P.angles - 1);
        for (int i = i0; i <= i1; ++i) {
            const int r = r0 - i * step;
            const short* at = P.slot_at + side_of_knots(P.N, w, r, s) * P.N.nm_pad;
            const float* side = P.side + ((size_t)i * P.np + p) * P.N.slots;
            int z[kTapsN];
            const int m = abs(r), turn = r > 0 ? 1 : -1;
            if (m >= kTapsN / 2 && 2 * (m + kTapsN / 2) <= n) {   // the offsets in a row
#pragma unroll
                for (int t = 0; t < kTapsN; ++t) z[t] = at[P.N.m_off[w] + m + turn * (t - kTapsN / 2)];
            } else {
#pragma unroll
                for (int t = 0; t < kTapsN; ++t) z[t] = at[offset_of(P.N, w, r + t - kTapsN / 2)];
            }
#pragma unroll
            for (int t = 0; t < kTapsN; ++t)
                if (z[t] >= 0) v = fmaf(x[t], side[z[t]], v);
        }
    }
    return v;
}

// The paths' values in direction order, a thread per (point, path): the taps
// of consecutive paths are consecutive nodes.  24 us for 8 angles, 14 of them without the
// knots; kSplit adds the parts of a split k_ang_back (with 7 taps and no knots a
// loop over one part cost 17 instead of 15 us, and 79 instead of 52 us
// at 3464 voxels).
template <bool kSplit>
__global__ void __launch_bounds__(256) k_ang_paths(const NodeParams P) {
    const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= (int64_t)P.np * P.nq) return;
    const int p = (int)(i / P.nq);
    const uint32_t fix = P.fix[i];
    float v = 0.f;
    for (int w = 0; w < P.N.W; ++w) {
        const int n = P.N.n_dir[w];
        int c;
        const float s = direction_pos(fix, n, &c);
        float x[kTapsN];
        lagrange9(s, P.path_b[(size_t)w * P.np * P.nq + i], x);
        const float* T = P.T + (size_t)p * P.N.nn + P.N.n_off[w];
#pragma unroll
        for (int k = 0; k < kTapsN; ++k) {
            int j = c + k - kTapsN / 2;
            j = j < 0 ? j + n : j >= n ? j - n : j;
            float t = T[j];
            if (kSplit)
                for (int o = 1; o < P.parts; ++o) t += T[(size_t)o * P.np * P.N.nn + j];
            v = fmaf(x[k], t, v);
        }
        if (P.N.kinks[w] > 0) v = beyond_knots(P, w, p, c, s, x, v);
    }
    P.val[i] = v;
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
        float wt[kTapsK];
        lagrange16(energy_pos(P.N, e, &k), wt);
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int i = 0; i < kTapsK; i += 2) {
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
// lane forms the values of one event; the events' 16 taps are then added one
// event per half-warp at a time into the half-warp's own row, a tap a lane.  In cells of more than 1024 events the rows are emptied into second
// sums every 256 events of a warp.
__global__ void __launch_bounds__(32 * kCellWarps) k_node_cells(
    const EventParams P, const int* cell_start, int cell0, const float* energy, const float* weight,
    const uint32_t* perm, float* V, float* PV, double* ll) {
    extern __shared__ float sh[];
    constexpr int kRows = 2 * kCellWarps;
    const int nkp = P.N.nk_pad, W = P.N.W;
    float* Fs = sh;                          // [nk_pad]
    float* acc = Fs + nkp;                   // [kRows][nk_pad]
    float* tot = acc + kRows * nkp;          // [kRows][nk_pad]
    __shared__ float wts[kCellWarps][32][kTapsK + 1];
    __shared__ int kpos[kCellWarps][32];
    __shared__ float pv_s[kCellWarps][4];
    __shared__ double ll_s[kCellWarps];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const size_t cell = blockIdx.x;
    const int e0 = cell_start[cell0 + blockIdx.x], e1 = cell_start[cell0 + blockIdx.x + 1];
    float* out = V + cell * nkp;
    const bool large = e1 - e0 > 1024;
    if (e0 == e1) {
        for (int k = t; k < nkp; k += 32 * kCellWarps) out[k] = 0.f;
        if (t < W) PV[cell * W + t] = 0.f;
        if (ll && t == 0) ll[cell] = 0.0;
        return;
    }
    for (int k = t; k < nkp; k += 32 * kCellWarps) {
        if (P.F) Fs[k] = P.F[cell * nkp + k];
#pragma unroll
        for (int i = 0; i < kRows; ++i) acc[i * nkp + k] = 0.f;
        for (int i = 0; large && i < kRows; ++i) tot[i * nkp + k] = 0.f;
    }
    __syncthreads();
    float pv[4] = {0.f, 0.f, 0.f, 0.f};
    double lsum = 0.0;
    float* mine = acc + (2 * warp + (lane >> 4)) * nkp;
    static_assert(kTapsK == 16, "a tap a lane of the half-warp");
    const int tap = lane & 15;
    int batches = 0;
    for (int b0 = e0 + 32 * warp; b0 < e1; b0 += 32 * kCellWarps) {
        const int j = b0 + lane;
        float r = 0.f, wt[kTapsK];
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
            if (reach) lagrange16(energy_pos(P.N, e, &k), wt);
            if (P.F) {
                if (reach) {
                    float s0 = 0.f, s1 = 0.f;
#pragma unroll
                    for (int i = 0; i < kTapsK; i += 2) {
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
        for (int i = 0; i < kTapsK; ++i) wts[warp][lane][i] = reach ? r * wt[i] : 0.f;
        __syncwarp();
        const int n_here = min(32, e1 - b0);
        const int h0 = (lane >> 4) * 16;
        for (int i = 0; i < 16; ++i) {
            const int ev = h0 + i;
            if (ev < n_here) mine[kpos[warp][ev] + tap] += wts[warp][ev][tap];
            __syncwarp();
        }
        if (large && (++batches & 7) == 0) {
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
#pragma unroll
        for (int i = 0; i < kRows; ++i) s += large ? tot[i * nkp + k] + acc[i * nkp + k] : acc[i * nkp + k];
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

// Voxel sums over the scatter points' paths and the angles' unscattered parts
// (FP64, 128 strands in fixed order) and, with sens, the multiplicative update
// of lam; else the sums go to num.  One block per 8 voxels: the sums are short
// (a few points a strand) and bound by load latency, so they want many strands
// (11 us; 33 us at 3464 voxels, half of the measured copy bandwidth).
constexpr int kUpdVox = 8, kUpdStrands = 128;
__global__ void __launch_bounds__(kUpdVox * kUpdStrands) k_node_update(
    const float* val, const int* path_of, int np, const float* part_prim, int n_prim, int nq,
    int nq_pad, const double* sens, float* lam, double* num) {
    __shared__ double red[kUpdStrands][kUpdVox + 1];
    const int v = threadIdx.x % kUpdVox, strand = threadIdx.x / kUpdVox;
    const int q = blockIdx.x * kUpdVox + v;
    double s = 0.0;
    if (q < nq) {
        for (int p0 = strand; p0 < np; p0 += 8 * kUpdStrands) {
            int r[8];
            float x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int p = p0 + k * kUpdStrands;
                r[k] = p < np ? path_of[(size_t)p * nq + q] : 0;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int p = p0 + k * kUpdStrands;
                x[k] = p < np ? val[(size_t)p * nq + r[k]] : 0.f;
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) s += (double)x[k];
        }
        for (int i = strand; i < n_prim; i += kUpdStrands) s += (double)part_prim[(size_t)i * nq_pad + q];
    }
    red[strand][v] = s;
    for (int o = kUpdStrands / 2; o > 0; o >>= 1) {
        __syncthreads();
        if (strand < o) red[strand][v] += red[strand + o][v];
    }
    if (strand == 0 && q < nq) {
        const double t = red[0][v];
        if (sens)   // (the ratios and the rows are not negative: nor is their sum, but for rounding)
            lam[q] = sens[q] > 0.0 ? (float)((double)lam[q] * (t < 0.0 ? 0.0 : t) / sens[q]) : 0.f;
        else
            num[q] = t;
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

// ------------------------------------------------------------------ set-up

// First and last + 1 of the bins the lanes found, over the warp.
__device__ __forceinline__ int2 warp_bins(int lo, int hi) {
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    return lo < hi ? make_int2(lo, hi) : make_int2(0, 0);
}

// Bins a chunk of 32 scatter points reaches: those whose run overlaps it.  A
// warp per chunk, a lane per bin (one thread a chunk waits for the bins one by
// one).
constexpr int kBinsWarps = 4;
__global__ void k_chunk_bins(const int2* crange, int B, int npc, int2* chunk_bins, int* most) {
    const int a = blockIdx.y, lane = threadIdx.x & 31;
    const int pc = blockIdx.x * kBinsWarps + (threadIdx.x >> 5);
    if (pc >= npc) return;
    int lo = B, hi = 0;
    for (int b = lane; b < B; b += 32) {
        const int2 r = crange[(size_t)a * B + b];
        if (r.y > r.x && r.x < (pc + 1) * kPC && r.y > pc * kPC) {
            lo = min(lo, b);
            hi = b + 1;
        }
    }
    const int2 br = warp_bins(lo, hi);
    if (lane == 0) {
        chunk_bins[(size_t)a * npc + pc] = br;
        atomicMax(most, br.y - br.x);
    }
}

// Place of each point in an angle's order, and its line integral to the
// detector in FP32.
__global__ void k_point_tables(const int* inv, const double* g_p, int np, int* rank, float* gamma) {
    const int a = blockIdx.y, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    rank[(size_t)a * np + inv[(size_t)a * np + i]] = i;
    gamma[(size_t)a * np + i] = (float)g_p[(size_t)a * np + i];
}

// Bins the 8 points of a group reach (a warp per group, a lane per bin).
__global__ void k_group_bins(const int2* crange, const int* rank, const int* grp_pt, int B, int np,
                             int groups, int2* grp_bins, int* most) {
    const int a = blockIdx.y, lane = threadIdx.x & 31;
    const int g = blockIdx.x * kBinsWarps + (threadIdx.x >> 5);
    if (g >= groups) return;
    int at[kGroup];
#pragma unroll
    for (int i = 0; i < kGroup; ++i) {
        const int p = grp_pt[g * kGroup + i];
        at[i] = p < 0 ? -1 : rank[(size_t)a * np + p];
    }
    int lo = B, hi = 0;
    for (int b = lane; b < B; b += 32) {
        const int2 r = crange[(size_t)a * B + b];
        bool any = false;
#pragma unroll
        for (int i = 0; i < kGroup; ++i) any |= at[i] >= r.x && at[i] < r.y;
        if (any) {
            lo = min(lo, b);
            hi = b + 1;
        }
    }
    const int2 br = warp_bins(lo, hi);
    if (lane == 0) {
        grp_bins[(size_t)a * groups + g] = br;
        atomicMax(most, br.y - br.x);
    }
}

__global__ void k_group_values(const float* cs, const int* rank, const int* grp_pt,
                               const int2* grp_bins, int B, int np, int npc, int groups, int nbg_max,
                               float* grp_c) {
    const int a = blockIdx.y;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)groups * nbg_max * kGroup) return;
    const int k = (int)(i % kGroup), b = (int)(i / kGroup % nbg_max), g = (int)(i / kGroup / nbg_max);
    const int2 br = grp_bins[(size_t)a * groups + g];
    const int p = grp_pt[g * kGroup + k];
    float v = 0.f;
    if (p >= 0 && br.x + b < br.y) {
        const int r = rank[(size_t)a * np + p];
        v = cs[(((size_t)a * npc + r / kPC) * B + br.x + b) * kCPad + r % kPC];
    }
    grp_c[(size_t)a * groups * nbg_max * kGroup + i] = v;
}

// Direction from voxel q to point p in 2^-32 turns.
__device__ __forceinline__ uint32_t pair_direction(const ModelConst& m, int pix, int c) {
    const double dx = ((c % m.S) + 0.5) * m.f - ((pix % m.n) + 0.5);
    const double dy = ((c / m.S) + 0.5) * m.f - ((pix / m.n) + 0.5);
    double t = (dx == 0.0 && dy == 0.0) ? 0.0 : atan2(dy, dx) * 0.15915494309189533577;   // / 2 pi
    t -= floor(t);
    return (uint32_t)(uint64_t)(t * 4294967296.0);
}

// What a path's weights are formed from and where the sorted paths go.
struct PathTables {
    const int *q_pix, *p_cell;
    const double *p_rho, *g_qp, *d_qp, *mu_line;
    uint32_t* fix;
    int *path_q, *path_of;
    float* path_b;
};

// Path i of point p leads from voxel q: its voxel, the voxel's place and, per
// line, the weight B = alpha mu_0 rho_p A_p / d exp(-mu_0 gamma_qp) / K (0 for
// voxels in the point's own cell).
__device__ __forceinline__ void put_path(const ModelConst& m, const PathTables& T, int p, int q, int i,
                                         uint32_t fix) {
    const int64_t at = (int64_t)p * m.nq + i, n = (int64_t)m.np * m.nq;
    T.fix[at] = fix;
    T.path_q[at] = q;
    T.path_of[(size_t)p * m.nq + q] = i;
    const int pix = T.q_pix[q];
    const bool own = ((pix / m.n) / m.f) * m.S + (pix % m.n) / m.f == T.p_cell[p];
    const size_t k = (size_t)q * m.np + p;
    for (int w = 0; w < m.W; ++w)
        T.path_b[(size_t)w * n + at] =
            own ? 0.f
                : (float)(m.alpha[w] * T.mu_line[w] * T.p_rho[p] * m.cell_area / T.d_qp[k] *
                          exp(-T.mu_line[w] * T.g_qp[k]) / m.kn_norm[w]);
}

// The paths of each point by direction (then voxel): a block per point sorts
// them in shared memory, `size` (a power of two) keys of direction and voxel.
// 24 x 24 pixels and 52 points took 16 launches through the global sort.
constexpr int kSortPoint = 16384;        // most voxels of a point sorted this way: 128 KB
__global__ void __launch_bounds__(512) k_point_paths(ModelConst m, const PathTables T, int size) {
    extern __shared__ unsigned long long key[];
    const int p = blockIdx.x, c = T.p_cell[p];
    for (int q = threadIdx.x; q < size; q += blockDim.x)
        key[q] = q < m.nq ? (unsigned long long)pair_direction(m, T.q_pix[q], c) << 32 | (unsigned)q : ~0ull;
    for (int run = 2; run <= size; run <<= 1)
        for (int d = run >> 1; d > 0; d >>= 1) {
            __syncthreads();
            for (int i = threadIdx.x; i < size / 2; i += blockDim.x) {
                const int x = (i & ~(d - 1)) * 2 + (i & (d - 1)), y = x + d;
                const unsigned long long u = key[x], v = key[y];
                if ((u > v) == ((x & run) == 0)) {
                    key[x] = v;
                    key[y] = u;
                }
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < m.nq; i += blockDim.x)
        put_path(m, T, p, (int)(key[i] & 0xffffffffu), i, (uint32_t)(key[i] >> 32));
}

// The same where a point has more voxels: keys of the global sorts (pair
// p nq + q), then the sorted paths.
__global__ void k_pair_direction(ModelConst m, const int* q_pix, const int* p_cell, uint32_t* fix,
                                 uint32_t* idx) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)m.np * m.nq) return;
    fix[i] = pair_direction(m, q_pix[i % m.nq], p_cell[i / m.nq]);
    idx[i] = (uint32_t)i;
}

__global__ void k_pair_points(const uint32_t* idx, int64_t n, int nq, uint32_t* key) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) key[i] = idx[i] / (uint32_t)nq;
}

__global__ void k_pair_fill(ModelConst m, const PathTables T, const uint32_t* order, const uint32_t* fix0) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)m.np * m.nq) return;
    const uint32_t src = order[i];
    const int p = (int)(src / (uint32_t)m.nq);
    put_path(m, T, p, (int)(src % (uint32_t)m.nq), (int)(i - (int64_t)p * m.nq), fix0[src]);
}

// First path of each point at every line's centre nodes 0 .. n, and the count.
__global__ void k_path_starts(const NodeConst N, const uint32_t* fix, int np, int nq, int* start) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)np * N.start_ints) return;
    const int p = (int)(i / N.start_ints);
    int node = (int)(i % N.start_ints), w = 0;
    while (node >= N.n_dir[w] + 2) {
        node -= N.n_dir[w] + 2;
        ++w;
    }
    const int n = N.n_dir[w];
    const uint32_t* f = fix + (size_t)p * nq;
    int lo = 0, hi = nq;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        int c;
        direction_pos(f[mid], n, &c);
        if (c < node) lo = mid + 1; else hi = mid;
    }
    start[i] = lo;
}

// The direction offsets' attenuation (log2(e) mu_water(E')) and the weights, times
// f, of the kTapsL scattered-energy nodes from psi_l on that E' lies between.
__global__ void k_offset_tables(ModelConst m, const NodeConst N, double kappa, const int* psi_l, float* mu,
                                float* psi_w) {
    const int o = blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= N.nm_pad) return;
    int w = 0;
    while (w + 1 < N.W && o >= N.m_off[w + 1]) ++w;
    const int i = o - N.m_off[w];
    if (i >= N.m_count[w]) {             // pads between the lines
        mu[o] = 0.f;
        for (int k = 0; k < kPsiStride; ++k) psi_w[(size_t)kPsiStride * o + k] = 0.f;
        return;
    }
    const double e0 = m.line_e[w], k0 = e0 / 510.99895;
    const double c = cospi(2.0 * i / N.n_dir[w]), r = 1.0 / (1.0 + k0 * (1.0 - c)), e = e0 * r;
    const double kn = r * r * (r + 1.0 / r - (1.0 - c * c));
    const double f = kn / (2.506628274631000502 * kappa * sqrt(e));   // / (sqrt(2 pi) sigma)
    const double u = 2.0 * sqrt(e) / kappa * N.per_l - N.l_first[w];
    const double s = u - (psi_l[o] - N.l_off[w] + kTapsL / 2);
    double mu_e = m.knot_mu[0];
    if (m.n_knots > 1) {
        int k = 0;
        while (k < m.n_knots - 2 && e >= m.knot_e[k + 1]) ++k;
        mu_e = m.knot_mu[k] + (e - m.knot_e[k]) * m.knot_slope[k];
    }
    mu[o] = (float)(mu_e * 1.4426950408889634);
    for (int k = 0; k < kPsiStride; ++k) {
        double v = k < kTapsL ? f : 0.0, d = 1.0;
        for (int j = 0; j < kTapsL; ++j)
            if (j != k) {
                v *= s - (j - kTapsL / 2);
                d *= k - j;
            }
        psi_w[(size_t)kPsiStride * o + k] = (float)(v / d);
    }
}

// The same weights by node l, 32 nodes at a time: entries dec_start[l / 32] + 32 i
// + l % 32 are the offsets (dec_m) and weights of node l, i < the most any of the
// 32 nodes has.  The offsets of a node are consecutive (E' falls with the offset).
__global__ void k_offset_lists(const NodeConst N, const int* psi_l, const float* psi_w, const int2* run,
                               const int* dec_start, int* dec_m, float* dec_w) {
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= N.nl_pad) return;
    const int2 r = run[l];
    const int d1 = dec_start[(l >> 5) + 1];
    int o = r.x;
    for (int d = dec_start[l >> 5] + (l & 31); d < d1; d += 32, ++o) {
        dec_m[d] = o < r.y ? o : 0;
        dec_w[d] = o < r.y ? psi_w[(size_t)kPsiStride * o + l - psi_l[o]] : 0.f;
    }
}

// Shared-memory opt-in of the node kernels, once per device.
int node_kernel_attrs() {
    static std::atomic<unsigned long long> done{0};
    int dev = 0, cap = 0;
    LMMEW_CUDA(cudaGetDevice(&dev));
    const unsigned long long bit = 1ull << (dev & 63);
    if (done.load() & bit) return LMMEW_OK;
    LMMEW_CUDA(cudaDeviceGetAttribute(&cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    for (auto k : {k_node_values, k_node_bins, k_ang_psi})
        LMMEW_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, cap - 4096));
    LMMEW_CUDA(cudaFuncSetAttribute(k_node_unvalues, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    cap - 4096));
    LMMEW_CUDA(cudaFuncSetAttribute(k_ang_back, cudaFuncAttributeMaxDynamicSharedMemorySize, cap - 4096));
    LMMEW_CUDA(cudaFuncSetAttribute(k_node_cells, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    80 * 1024));
    LMMEW_CUDA(cudaFuncSetAttribute(k_point_paths, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    8 * kSortPoint));
    done.fetch_or(bit);
    return LMMEW_OK;
}

NodeParams node_params(const lm_handle* h, int a0, int a_step, int angles) {
    const ModelConst& m = h->mc;
    NodeParams P{};
    P.N = h->nodes;
    P.a0 = a0;
    P.a_step = a_step;
    P.angles = angles;
    P.A = m.A;
    P.B = m.B;
    P.nq = m.nq;
    P.np = m.np;
    P.npc = m.npc;
    P.nq_pad = m.nqt * kQT;
    const NodeTables& t = h->node_tables;
    P.g = t.g;
    P.gt = t.gt;
    P.k_of_l = t.k_of_l;
    P.l_of_k = t.l_of_k;
    P.chunk_bins = t.chunk_bins;
    P.cs = h->d_cs;
    P.crange = h->d_crange;
    P.inv = h->d_inv;
    P.gamma = t.gamma;
    P.mu = t.mu;
    P.psi_l = t.psi_l;
    P.psi_w = t.psi_w;
    P.dec_start = t.dec_start;
    P.dec_m = t.dec_m;
    P.dec_w = t.dec_w;
    P.fix = t.fix;
    P.path_q = t.path_q;
    P.path_of = t.path_of;
    P.path_b = t.path_b;
    P.path_start = t.path_start;
    P.slot = t.slot;
    P.slot_start = t.slot_start;
    P.slot_at = t.slot_at;
    P.win = t.win;
    for (int w = 0; w < m.W; ++w) P.inv_step[w] = (float)m.A / ((float)P.N.n_dir[w] * (float)a_step);
    P.grp_pt = t.grp_pt;
    P.grp_bins = t.grp_bins;
    P.grp_c = h->d_node_groups;
    P.cv = h->d_cv;
    P.prim = h->d_prim;
    return P;
}

// Shared memory of band_product for at most `band` nodes.
size_t band_smem(int band) {
    return sizeof(float) * ((size_t)kValueWarps * kValueRows * 32 + (size_t)kValueRows * band);
}

}  // namespace

// The nodes of the model and everything the route reads.  It exists for the
// square-root energy resolution, up to 4 lines and node counts and pair tables
// (12 + 4 W bytes per voxel and scatter point) of sane sizes; other models keep
// the rows.  Built with every model, so it may not cost a small one much: nine
// launches, one allocation more for the grouped collimator values, a copy up and
// one down; a model of 24 x 24 voxels, 12 x 12 cells and 24 angles takes 1.5 ms
// with them (2.2 ms with host tables and global sorts, 1.75 ms without any).
static int build_node_tables(lm_handle* h) {
    const ModelConst& m = h->mc;
    NodeConst& N = h->nodes;
    NodeTables& T = h->node_tables;
    h->node_route = 0;
    N = NodeConst{};
    const int64_t pairs = (int64_t)m.np * m.nq;
    if (m.np == 0 || m.W > 4 || m.expo != -0.5 || pairs >= (int64_t(1) << 31)) return LMMEW_OK;
    const double pi = 3.14159265358979323846, log2e = 1.4426950408889634, me = 510.99895;
    const double kappa = m.fwhm_frac * sqrt(m.e_ref) / (2.0 * sqrt(2.0 * log(2.0)));   // sigma = kappa sqrt(E)
    auto t_of = [&](double e) { return 2.0 * sqrt(e) / kappa; };
    N.W = m.W;
    std::vector<NodeSlot> slots;
    std::vector<int> slot_start;
    std::vector<int2> wins;
    // recorded energies
    // the Gaussian's exponent changes by up to 1 + 4 kappa / sqrt(E') per unit of
    // t at 8 sigma, 1.25 for 62 keV and 10 % at 140 keV: denser nodes where more
    auto denser = [&](double e) { return std::max(1.0, (1.0 + 4.0 * kappa / sqrt(e)) / 1.26); };
    double dense = 1.0;
    for (int w = 0; w < m.W; ++w)
        dense = std::max(dense, denser(m.line_e[w] / (1.0 + 2.0 * m.line_e[w] / me)));
    if (!(dense < 16.0)) return LMMEW_OK;
    N.per_l = (int)ceil(kPerUnitL * dense);
    N.per_k = (int)ceil(kPerUnitK * dense);
    const double ck = N.per_k * 2.0 / kappa;
    N.ck = (float)ck;
    N.ck_lo = (float)(ck - (double)N.ck);
    double e_lo = 1e300, e_hi = 0.0;
    for (int k = 0; k < m.n_win; ++k) {
        e_lo = std::min(e_lo, std::max(m.win_lo[k], 0.0));
        e_hi = std::max(e_hi, m.win_hi[k]);
    }
    const double t_hi = t_of(e_hi) * N.per_k;
    if (!(t_hi < 8192.0)) return LMMEW_OK;
    N.k_first = (int)floor(t_of(e_lo) * N.per_k) - kTapsK / 2;
    N.nk = (int)floor(t_hi) + kTapsK / 2 + 1 - N.k_first + 1;
    N.nk_pad = (N.nk + 31) & ~31;
    // scattered energies and directions of each line
    for (int w = 0; w < m.W; ++w) {
        const double e0 = m.line_e[w], k0 = e0 / me, eb = e0 / (1.0 + 2.0 * k0);
        const double u0 = t_of(eb) * N.per_l, u1 = t_of(e0) * N.per_l;
        if (!(u1 < 1.0e6)) return LMMEW_OK;
        N.l_first[w] = (int)floor(u0) - kTapsL / 2 - 1;
        N.l_count[w] = (int)ceil(u1) + kTapsL / 2 + 1 - N.l_first[w] + 1;
        if (N.l_first[w] < 1) return LMMEW_OK;
        N.l_off[w] = N.nl;               // (lines start at multiples of 8 nodes)
        N.nl += (N.l_count[w] + 7) & ~7;
        // 17 nodes per sigma where E'(x) is steepest (9 taps: 1e-7 of a term at 6
        // sigma, 3e-6 at 8), and
        // enough that the attenuation changes by 4 % per node at most over the
        // longest way through the map
        auto slope = [&](double e) {     // |dE'/dx|
            const double c = std::min(std::max(1.0 - (e0 / e - 1.0) / k0, -1.0), 1.0);
            return e * e / e0 * k0 * sqrt(1.0 - c * c);
        };
        const double way = h->rho_max * m.n * m.h * sqrt(2.0);
        auto mu_slope = [&](double e) {
            int s = 0;
            while (s < m.n_knots - 2 && e >= m.knot_e[s + 1]) ++s;
            return m.n_knots > 1 ? fabs(m.knot_slope[s]) : 0.0;
        };
        double want = 32.0;
        auto sample = [&](double e) {
            want = std::max(want, 2.0 * pi * slope(e) * std::max(kPerSigmaN * denser(eb) / (kappa * sqrt(e)),
                                                               mu_slope(e) * way / 0.04));
        };
        for (int i = 1; i < 512; ++i) sample(e0 / (1.0 + k0 * (1.0 - cos(pi * i / 512))));
        // knots inside E', by offset; the segment of mu on either side
        std::vector<double> at;
        int seg = 0;
        while (seg < m.n_knots - 2 && e0 > m.knot_e[seg + 1]) ++seg;
        std::vector<int> segs(1, seg);
        for (; seg > 0 && m.knot_e[seg] > eb; --seg) {
            const double e = m.knot_e[seg];
            sample(e);
            sample(std::nextafter(e, 0.0));
            if (m.knot_slope[seg] == m.knot_slope[seg - 1]) {
                segs.back() = seg - 1;   // (the same line)
                continue;
            }
            at.push_back(acos(1.0 - (e0 / e - 1.0) / k0));
            segs.push_back(seg - 1);
        }
        if (!(want < 16384.0) || m.A > 16384) return LMMEW_OK;
        N.angle_step[w] = ((int)ceil(want) + m.A - 1) / m.A;
        N.n_dir[w] = N.angle_step[w] * m.A;
        N.n_off[w] = N.nn;
        N.nn += N.n_dir[w];
        N.m_count[w] = N.n_dir[w] / 2 + 1;
        N.m_off[w] = N.nm_pad;
        N.nm_pad += (N.m_count[w] + 31) & ~31;
        N.start_ints += N.n_dir[w] + 2;
        // the nodes whose taps a knot lies between, once per other side
        const int count = N.m_count[w], n = N.n_dir[w], half = kTapsN / 2;
        N.kinks[w] = (int)at.size();
        for (size_t k = 0; k < at.size(); ++k) N.kink[w][k] = (float)(at[k] * n / (2.0 * pi));
        auto branch_of = [&](double u) {
            int b = 0;
            while (b < N.kinks[w] && u > N.kink[w][b]) ++b;
            return b;
        };
        auto fold = [&](double u) { return fabs(u) > 0.5 * n ? n - fabs(u) : fabs(u); };
        slot_start.resize(N.m_off[w] + count + 1, (int)slots.size());
        N.slot_off[w] = (int)slots.size();
        for (int i = 0; i < count; ++i) {
            slot_start[N.m_off[w] + i] = (int)slots.size();
            const int own = branch_of(i);
            for (int b = 0; b <= N.kinks[w]; ++b) {
                if (b == own) continue;
                const float lo = b == 0 ? -1.f : N.kink[w][b - 1], hi = b == N.kinks[w] ? 1e9f : N.kink[w][b];
                bool reached = false;
                for (int d = -half; d <= half; ++d) {
                    // paths centred there: i + d - 1/2 .. i + d + 1/2, folded
                    const double u0 = fold(i + d - 0.5), u1 = fold(i + d + 0.5), u2 = fold(i + d);
                    reached |= std::max({u0, u1, u2}) + 1e-3 >= lo && std::min({u0, u1, u2}) - 1e-3 <= hi;
                }
                if (!reached) continue;
                const double e = e0 / (1.0 + k0 * (1.0 - cos(2.0 * pi * i / n)));
                const double mu_b = m.knot_mu[segs[b]] + (e - m.knot_e[segs[b]]) * m.knot_slope[segs[b]];
                slots.push_back({N.m_off[w] + i, b, (float)(mu_b * log2e)});
            }
        }
        slot_start.back() = (int)slots.size();
        constexpr int kTile = kOffThreads * kOffPer;
        for (int i = 0; i < count; i += kTile)
            N.tile_slots = std::max(N.tile_slots, slot_start[N.m_off[w] + std::min(i + kTile, count)] -
                                                      slot_start[N.m_off[w] + i]);
        // windows of c - s with a knot among the taps, both turns of the circle
        N.win_off[w] = (int)wins.size();
        std::vector<int2> around;
        for (double x : at)
            for (int turn = -1; turn <= 1; ++turn)
                for (int sign = -1; sign <= 1; sign += 2) {
                    const double u = sign * x * n / (2.0 * pi) + turn * n;
                    const int lo = std::max((int)floor(u) - half - 1, -n), hi = std::min((int)ceil(u) + half + 1, n);
                    if (lo <= hi) around.push_back(make_int2(lo, hi));
                }
        std::sort(around.begin(), around.end(), [](int2 a, int2 b) { return a.x < b.x; });
        for (const int2& r : around) {
            if ((int)wins.size() > N.win_off[w] && r.x <= wins.back().y + 1)
                wins.back().y = std::max(wins.back().y, r.y);
            else
                wins.push_back(r);
        }
        if ((int)wins.size() - N.win_off[w] > kMostWindows) return LMMEW_OK;
        N.reach_lo[w] = h->reach_lo[w];
        N.reach_hi[w] = h->reach_hi[w];
    }
    N.win_off[m.W] = (int)wins.size();
    N.slots = N.slot_off[m.W] = (int)slots.size();
    slot_start.resize(N.nm_pad + 1, N.slots);
    const int sides = 1 + *std::max_element(N.kinks, N.kinks + 4);
    std::vector<short> slot_at((size_t)sides * N.nm_pad, -1);
    N.nl_pad = (N.nl + 31) & ~31;
    if (N.tile_slots > 256 || N.slots > 32767) return LMMEW_OK;   // (staged by k_ang_bins, named by short)
    for (int z = 0; z < N.slots; ++z) slot_at[(size_t)slots[z].side * N.nm_pad + slots[z].offset] = (short)z;
    if (N.nl > 6000 || N.nk > 1152 || N.nn > 32768 || (int64_t)m.np * N.nn >= (int64_t(1) << 31))
        return LMMEW_OK;
    const size_t pair_bytes = (12 + 4 * (size_t)m.W) * (size_t)pairs;
    if (pair_bytes > (size_t(64) << 20)) {
        size_t free_b = 0, total_b = 0;
        LMMEW_CUDA(cudaMemGetInfo(&free_b, &total_b));
        if (2 * pair_bytes > free_b / 4) return LMMEW_OK;
    }

    // host tables: first of the scattered-energy nodes each offset's E' lies
    // between (its cosine by the three-term recurrence: it only has to name the
    // nearest node), the offsets of each node and the bands
    std::vector<int> psi_l(N.nm_pad, 0), dec_start(N.nl_pad / 32 + 1, 0);
    std::vector<int2> run(N.nl_pad, make_int2(0, 0));
    for (int w = 0; w < m.W; ++w) {
        const double e0 = m.line_e[w], k0 = e0 / me, step = cos(2.0 * pi / N.n_dir[w]);
        double c = 1.0, before = step;
        for (int i = 0; i < N.m_count[w]; ++i) {
            const double u = t_of(e0 / (1.0 + k0 * (1.0 - c))) * N.per_l - N.l_first[w];
            const int o = N.m_off[w] + i, first = N.l_off[w] + (int)floor(u + 0.5) - kTapsL / 2;
            psi_l[o] = first;
            for (int l = first; l < first + kTapsL; ++l) {
                if (run[l].y == 0) run[l].x = o;
                run[l].y = o + 1;
            }
            const double next = 2.0 * step * c - before;
            before = c;
            c = next;
        }
    }
    size_t dec_n = 0;
    for (int t = 0; t < N.nl_pad / 32; ++t) {
        int most = 0;
        for (int l = 32 * t; l < 32 * t + 32; ++l) most = std::max(most, run[l].y - run[l].x);
        dec_n += 32 * (size_t)most;
        dec_start[t + 1] = (int)dec_n;
    }
    const int lt = N.nl_pad / 32, kt = N.nk_pad / 32;
    std::vector<int2> bands((size_t)lt + kt, make_int2(1 << 30, 0));
    int2* k_of_l = bands.data();
    int2* l_of_k = k_of_l + lt;
    for (int w = 0; w < m.W; ++w)
        for (int i = 0; i < N.l_count[w]; ++i) {
            // |E_k - E_l| <= 10.2 sigma_l between the nodes just outside the band
            const int l = N.l_off[w] + i;
            const double x = 0.5 * kappa * (N.l_first[w] + i) / N.per_l, e = x * x;
            const double s = kBandSigmas * kappa * x;
            const double v0 = e > s ? t_of(e - s) * N.per_k : -1e9;
            const int k0 = std::max(0, (int)floor(v0) - N.k_first);
            const int k1 = std::min(N.nk, (int)ceil(t_of(e + s) * N.per_k) - N.k_first + 1);
            if (k0 >= k1) continue;
            k_of_l[l / 32].x = std::min(k_of_l[l / 32].x, k0);
            k_of_l[l / 32].y = std::max(k_of_l[l / 32].y, k1);
            for (int k = k0 / 32; k <= (k1 - 1) / 32; ++k) {
                l_of_k[k].x = std::min(l_of_k[k].x, l);
                l_of_k[k].y = std::max(l_of_k[k].y, l + 1);
            }
        }
    for (int2& r : bands)
        if (r.y == 0) r.x = 0;

    // one device region; the host tables lie together at its start
    // 8 neighbouring points at a time (cells of 4 x 2), which reach fewer bins
    // together than 8 in a row
    std::vector<int> grp_pt;
    {
        const std::vector<int>& cell = h->p_cell;
        std::vector<std::pair<int64_t, int>> key(m.np);
        for (int p = 0; p < m.np; ++p) {
            const int x = cell[p] % m.S, y = cell[p] / m.S;
            key[p] = {((int64_t)(y / 2) * (m.S / 4 + 1) + x / 4) * 8 + (y % 2) * 4 + x % 4, p};
        }
        std::sort(key.begin(), key.end());
        for (const auto& k : key) grp_pt.push_back(k.second);
        while (grp_pt.size() % kGroup) grp_pt.push_back(-1);
    }
    const int groups = (int)grp_pt.size() / kGroup;
    const size_t gm = (size_t)N.nl_pad * N.nk_pad;
    size_t host_bytes = 0;
    int* d_most = nullptr;
    int2* d_run = nullptr;
    auto layout = [&](char* p) {
        char* base = p;
        T.psi_l = bump<int>(p, psi_l.size());
        T.dec_start = bump<int>(p, dec_start.size());
        T.grp_pt = bump<int>(p, grp_pt.size());
        T.k_of_l = bump<int2>(p, bands.size());
        T.l_of_k = T.k_of_l + lt;
        T.slot = bump<NodeSlot>(p, slots.size());
        T.slot_start = bump<int>(p, slot_start.size());
        T.slot_at = bump<short>(p, slot_at.size());
        T.win = bump<int2>(p, wins.size());
        d_run = bump<int2>(p, run.size());
        d_most = bump<int>(p, 2);
        host_bytes = (size_t)(p - base);
        T.mu = bump<float>(p, N.nm_pad);
        T.psi_w = bump<float>(p, (size_t)kPsiStride * N.nm_pad);
        T.dec_m = bump<int>(p, dec_n);
        T.dec_w = bump<float>(p, dec_n);
        T.g = bump<float>(p, gm);
        T.gt = bump<float>(p, gm);
        T.chunk_bins = bump<int2>(p, (size_t)m.A * m.npc);
        T.grp_bins = bump<int2>(p, (size_t)m.A * groups);
        T.gamma = bump<float>(p, (size_t)m.A * m.np);
        T.rank = bump<int>(p, (size_t)m.A * m.np);
        T.path_start = bump<int>(p, (size_t)m.np * N.start_ints);
        T.fix = bump<uint32_t>(p, pairs);
        T.path_q = bump<int>(p, pairs);
        T.path_of = bump<int>(p, pairs);
        T.path_b = bump<float>(p, (size_t)m.W * pairs);
        return (size_t)(p - base) + 256;
    };
    const size_t bytes = layout(nullptr);
    // (points of up to kSortPoint voxels sort their paths in shared memory)
    const bool sort_global = m.nq > kSortPoint;
    const size_t sort_bytes = 4 * bump_bytes(4 * (size_t)pairs) + bump_bytes(pair_hist_bytes(pairs));
    struct Temp {
        void* p = nullptr;
        ~Temp() { cudaFree(p); }
    } temp;
    if (cudaMalloc(&h->d_node_tables, bytes) != cudaSuccess ||
        (sort_global && cudaMalloc(&temp.p, sort_bytes) != cudaSuccess)) {
        cudaGetLastError();
        return LMMEW_OK;                 // no room: the rows
    }
    h->node_bytes = bytes;
    layout((char*)h->d_node_tables);
    std::vector<char> blob(host_bytes, 0);
    auto put = [&](const void* dst, const void* src, size_t n) {
        std::memcpy(blob.data() + ((const char*)dst - (const char*)h->d_node_tables), src, n);
    };
    put(T.psi_l, psi_l.data(), 4 * psi_l.size());
    put(T.dec_start, dec_start.data(), 4 * dec_start.size());
    put(T.grp_pt, grp_pt.data(), 4 * grp_pt.size());
    put(T.k_of_l, bands.data(), 8 * bands.size());
    put(T.slot, slots.data(), sizeof(NodeSlot) * slots.size());
    put(T.slot_start, slot_start.data(), 4 * slot_start.size());
    put(T.slot_at, slot_at.data(), sizeof(short) * slot_at.size());
    put(T.win, wins.data(), 8 * wins.size());
    put(d_run, run.data(), 8 * run.size());
    LMMEW_CUDA(cudaMemcpy(h->d_node_tables, blob.data(), host_bytes, cudaMemcpyHostToDevice));
    int rc = node_kernel_attrs();
    if (rc != LMMEW_OK) return rc;

    k_offset_tables<<<(N.nm_pad + 63) / 64, 64>>>(m, N, kappa, T.psi_l, T.mu, T.psi_w);
    k_offset_lists<<<(N.nl_pad + 63) / 64, 64>>>(N, T.psi_l, T.psi_w, d_run, T.dec_start, T.dec_m, T.dec_w);
    k_node_matrix<<<(unsigned)((gm + 255) / 256), 256>>>(N, kappa, T.g, T.gt);
    k_chunk_bins<<<dim3((m.npc + kBinsWarps - 1) / kBinsWarps, m.A), 32 * kBinsWarps>>>(
        h->d_crange, m.B, m.npc, T.chunk_bins, d_most);
    k_point_tables<<<dim3((m.np + 127) / 128, m.A), 128>>>(h->d_inv, h->d_gp, m.np, T.rank, T.gamma);
    k_group_bins<<<dim3((groups + kBinsWarps - 1) / kBinsWarps, m.A), 32 * kBinsWarps>>>(
        h->d_crange, T.rank, T.grp_pt, m.B, m.np, groups, T.grp_bins, d_most + 1);
    const PathTables paths{h->d_q_pix, h->d_p_cell, h->d_p_rho, h->d_gqp, h->d_dqp, h->d_mu_line,
                           T.fix, T.path_q, T.path_of, T.path_b};
    if (!sort_global) {
        int size = 64;
        while (size < m.nq) size *= 2;
        k_point_paths<<<m.np, std::min(512, size / 2), 8 * (size_t)size>>>(m, paths, size);
        ++h->launches;
    } else {
        // stable sorts by direction, then point
        char* tp = (char*)temp.p;
        uint32_t* kin = bump<uint32_t>(tp, pairs);
        uint32_t* kout = bump<uint32_t>(tp, pairs);
        uint32_t* vin = bump<uint32_t>(tp, pairs);
        uint32_t* vout = bump<uint32_t>(tp, pairs);
        uint32_t* hist = bump<uint32_t>(tp, pair_hist_bytes(pairs) / 4);
        const unsigned pb = (unsigned)((pairs + 255) / 256);
        uint32_t* fix0 = reinterpret_cast<uint32_t*>(T.path_b);   // (free until the fill) unsorted directions
        k_pair_direction<<<pb, 256>>>(m, h->d_q_pix, h->d_p_cell, fix0, vin);
        LMMEW_CUDA(cudaMemcpyAsync(kin, fix0, 4 * (size_t)pairs, cudaMemcpyDeviceToDevice, 0));
        rc = sort_pairs(h, pairs, 32, kin, kout, vin, vout, hist, 0);
        if (rc != LMMEW_OK) return rc;
        k_pair_points<<<pb, 256>>>(vin, pairs, m.nq, kin);
        int bits = 1;
        while (bits < 32 && ((uint32_t)(m.np - 1) >> bits) != 0) ++bits;
        rc = sort_pairs(h, pairs, bits, kin, kout, vin, vout, hist, 0);
        if (rc != LMMEW_OK) return rc;
        LMMEW_CUDA(cudaMemcpyAsync(kin, fix0, 4 * (size_t)pairs, cudaMemcpyDeviceToDevice, 0));
        k_pair_fill<<<pb, 256>>>(m, paths, vin, kin);
        h->launches += 3;
    }
    k_path_starts<<<(unsigned)(((int64_t)m.np * N.start_ints + 127) / 128), 128>>>(N, T.fix, m.np, m.nq,
                                                                                  T.path_start);
    LMMEW_CUDA(cudaGetLastError());
    int most[2] = {0, 0};
    LMMEW_CUDA(cudaMemcpy(most, d_most, sizeof(most), cudaMemcpyDeviceToHost));
    N.nb_max = std::max(most[0], 1);
    N.nbg_max = std::max(most[1], 1);
    if (N.nbg_max > 1024) return LMMEW_OK;   // (its staging would not fit shared memory)
    const size_t per_angle = (size_t)groups * N.nbg_max * kGroup;
    if (cudaMalloc(&h->d_node_groups, sizeof(float) * per_angle * m.A) != cudaSuccess) {
        cudaGetLastError();
        return LMMEW_OK;
    }
    h->node_bytes += sizeof(float) * per_angle * m.A;
    k_group_values<<<dim3((unsigned)((per_angle + 255) / 256), m.A), 256>>>(
        h->d_cs, T.rank, T.grp_pt, T.grp_bins, m.B, m.np, m.npc, groups, N.nbg_max, h->d_node_groups);
    h->launches += 8;
    LMMEW_CUDA(cudaGetLastError());
    LMMEW_CUDA(cudaDeviceSynchronize());   // (the tables are used on any stream)
    h->node_route = 1;
    return LMMEW_OK;
}

int build_nodes(lm_handle* h) {
    const int rc = build_node_tables(h);
    if (h->node_route == 0) {            // given up, or an error: nothing reads the tables
        cudaFree(h->d_node_tables);
        cudaFree(h->d_node_groups);
        h->d_node_tables = nullptr;
        h->d_node_groups = nullptr;
        h->node_tables = NodeTables{};
        h->node_bytes = 0;
    }
    return rc;
}

size_t node_angle_bytes(const lm_handle* h) {
    const NodeConst& N = h->nodes;
    return bump_bytes(sizeof(float) * (size_t)h->mc.np * N.slots) +
           bump_bytes(sizeof(float) * (size_t)h->mc.npc * N.nb_max * N.nm_pad) +
           bump_bytes(sizeof(float) * (size_t)h->mc.B * N.nl_pad) +
           bump_bytes(sizeof(float) * (size_t)h->mc.B * N.nk_pad) +
           bump_bytes(sizeof(float) * (size_t)h->mc.B * N.W);
}

// The image on the direction nodes of every scatter point (H null: not again),
// and on the slots of angles a0 + i a_step.
int node_spread(lm_handle* h, const float* lam_v, float* H, int a0, int a_step, int angles, float* side,
                cudaStream_t st) {
    NodeParams P = node_params(h, a0, a_step, angles);
    P.lam = lam_v;
    P.H = H;
    P.side = side;
    int tiles = 0;
    for (int w = 0; w < P.N.W; ++w) tiles += (P.N.n_dir[w] + kSpreadOut - 1) / kSpreadOut;
    const int units = H ? h->mc.np * tiles : 0;
    int64_t sides = 0;
    for (int w = 0; w < P.N.W; ++w)
        if (P.N.kinks[w] > 0) sides += (int64_t)angles * h->mc.np;
    const int side_blocks = (int)((sides + kSpreadWarps - 1) / kSpreadWarps);
    const int blocks = side_blocks + (units + kSpreadWarps - 1) / kSpreadWarps;
    if (blocks == 0) return LMMEW_OK;
    int rc = prof_start(h, st);
    if (rc != LMMEW_OK) return rc;
    k_ang_spread<<<(unsigned)blocks, 32 * kSpreadWarps, 0, st>>>(P, tiles, units, side_blocks);
    ++h->launches;
    LMMEW_CUDA(cudaGetLastError());
    return prof_stop(h, H ? (double)h->mc.W * h->mc.nq * h->mc.np : 0.0, st);
}

// F and the unscattered sums of angles a0 + i a_step, i < angles.
int node_forward(lm_handle* h, const float* lam_v, const float* H, const float* side, int a0, int a_step,
                 int angles, float* dbp, float* DB, float* F, float* Pr, cudaStream_t st) {
    if (angles <= 0) return LMMEW_OK;
    const ModelConst& m = h->mc;
    const NodeConst& N = h->nodes;
    NodeParams P = node_params(h, a0, a_step, angles);
    P.lam = lam_v;
    P.H = const_cast<float*>(H);
    P.side = const_cast<float*>(side);
    P.dbp = dbp;
    P.DB = DB;
    P.F = F;
    P.Pr = Pr;
    constexpr int kTile = kOffThreads * kOffPer;
    int tiles = 0;
    for (int w = 0; w < N.W; ++w) tiles += (N.m_count[w] + kTile - 1) / kTile;
    k_ang_bins<<<(unsigned)(tiles * m.npc * angles), kOffThreads, sizeof(float) * kPC * N.tile_slots, st>>>(
        P, tiles);
    const int rows = angles * m.B;
    k_node_bins<<<(unsigned)(rows + (rows * m.W + kRowThreadsN / 32 - 1) / (kRowThreadsN / 32)), kRowThreadsN,
                  sizeof(float) * N.nm_pad, st>>>(P);
    k_node_values<<<(unsigned)((rows + kValueRows - 1) / kValueRows * (N.nk_pad / 32)),
                    32 * kValueWarps, band_smem(N.nl_pad), st>>>(P);
    h->launches += 3;
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

static int back_tiles(const NodeConst& N) {
    int tiles = 0;
    for (int w = 0; w < N.W; ++w) tiles += (N.n_dir[w] + kBackTile - 1) / kBackTile;
    return tiles;
}

// Sums a back projection of so many angles is split over: as many as the chip
// holds grids of k_ang_back (8 blocks an SM), with 2 angles or more in each.
int node_back_parts(const lm_handle* h, int angles) {
    const int groups = (h->mc.np + kGroup - 1) / kGroup;
    const int blocks = back_tiles(h->nodes) * ((groups + kBackWarps - 1) / kBackWarps);
    return std::max(1, std::min({8, angles / 2, 8 * h->sm_count / blocks}));
}

// Back projection of the node weights of angles a0 + i a_step: the paths' values
// and the unscattered part of every angle.
int node_back(lm_handle* h, int a0, int a_step, int angles, const float* V, const float* PV,
              float* VG, float* psi, float* T, float* side, float* val, float* part_prim, cudaStream_t st) {
    const ModelConst& m = h->mc;
    const NodeConst& N = h->nodes;
    NodeParams P = node_params(h, a0, a_step, angles);
    P.V = V;
    P.PV = PV;
    P.VG = VG;
    P.psi = psi;
    P.T = T;
    P.side = side;
    P.val = val;
    P.part_prim = part_prim;
    const int rows = angles * m.B;
    const int blocks = (rows + kValueRows - 1) / kValueRows * (N.nl_pad / 32) +
                       angles * ((m.nq + 255) / 256);
    if (rows > 0) {
        k_node_unvalues<<<(unsigned)blocks, 32 * kValueWarps, band_smem(N.nk_pad), st>>>(P);
        k_ang_psi<<<(unsigned)rows, 256, sizeof(float) * N.nl_pad, st>>>(P);
    }
    const int tiles = back_tiles(N), groups = (m.np + kGroup - 1) / kGroup;
    P.parts = node_back_parts(h, angles);
    const size_t one = sizeof(float) * kBackWarps * (size_t)N.nbg_max * kGroup;   // staged per angle
    const int batch = (int)std::max<size_t>(1, std::min<size_t>(kBackAngles, kBackStage / one));
    const int64_t side_threads = (int64_t)N.slots * angles * groups * kGroup;
    const unsigned side_blocks = (unsigned)((side_threads + 32 * kBackWarps - 1) / (32 * kBackWarps));
    k_ang_back<<<dim3((unsigned)(tiles * ((groups + kBackWarps - 1) / kBackWarps)) + side_blocks, P.parts),
                 32 * kBackWarps, batch * one, st>>>(P, tiles, groups, batch);
    int rc = prof_start(h, st);
    if (rc != LMMEW_OK) return rc;
    const unsigned path_blocks = (unsigned)(((int64_t)m.np * m.nq + 255) / 256);
    if (P.parts > 1)
        k_ang_paths<true><<<path_blocks, 256, 0, st>>>(P);
    else
        k_ang_paths<false><<<path_blocks, 256, 0, st>>>(P);
    h->launches += 4;
    LMMEW_CUDA(cudaGetLastError());
    return prof_stop(h, (double)m.W * m.nq * m.np, st);
}

// The voxel sums: with sens the update of lam, else into num.
int node_update(lm_handle* h, int angles, const float* val, const float* part_prim,
                const double* sens, float* lam, double* num, cudaStream_t st) {
    const ModelConst& m = h->mc;
    k_node_update<<<(m.nq + kUpdVox - 1) / kUpdVox, kUpdVox * kUpdStrands, 0, st>>>(
        val, h->node_tables.path_of, m.np, part_prim, angles, m.nq, m.nqt * kQT, sens, lam, num);
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
