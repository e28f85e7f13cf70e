// Treecode far field of the real-charge and Kelvin-image pair sums of one large cavity (FP32
// path).  The paper evaluates the pair sum of eq. phirffinall with the FMM for N up to 1e6
// (Sec. 4.2, Algorithm 1 step 5); here a GPU treecode over the records' Morton order replaces the
// direct real and Kelvin pair sums, and the surface images keep their direct sum (3M sources per
// target).
//
// Octree.  Node (l, c) is Morton cell c of the 2^l-per-axis grid over [-a, a]^3; its records are
// a contiguous run of sorted positions (k_order_keys / k_order_sort sort by a key of key_lv >= L
// levels).  The real tree's node holds the charges of the run, the Kelvin tree's node the images
// of the same charges, except images farther than kFarImageRel a from the centre ("far images"),
// which form one expansion about the centre instead.
//   k_tree_marks  record range of every node of levels kTreeTop..L (first and last position of
//                 each key prefix)
//   k_tree_leaf   level L: bounding box, centre, radius and the multipole moments (a warp per node
//                 and tree, lane-strided records, fixed-order warp sums)
//   k_tree_up     levels L-1..kTreeTop: box and radius from the children, moments by shifting
//                 the children's moments to the parent's centre (a block per node and tree, a warp
//                 per child, or per two children at order 16)
//   k_tree_far    the far images' expansion about the centre (fixed-order block sums, the last
//                 block adds the blocks in order)
//   k_tree_eval   persistent warps over items (32 consecutive targets, one tree, an eighth of
//                 its root cells): depth-first traversal of the item's subtrees from the
//                 level-kTreeTop cells; a node far from every target of the group (radius <=
//                 theta (distance of the target from the centre)) with at
//                 least cmin records is evaluated from its moments at each target, a near leaf (or a
//                 far node too small for its moments to pay) by the direct pair sum, with FP32
//                 coordinates relative to the node's centre or, next to it, hi/lo differences
//                 (p2p); then the far-image expansion at each target.  Writes the
//                 real and the Kelvin sums as the (hi, lo) partials of chunks 0..kTreeRootSplit-1
//                 and kTreeRootSplit..2 kTreeRootSplit-1, which the reduction adds as it adds every
//                 chunk.
// Every sum runs in a fixed order (no atomics on values), so results do not depend on scheduling.
//
// Solid harmonics (unnormalised associated Legendre functions P_n^m without the Condon-Shortley
// phase), for 0 <= m <= n:
//   R_n^m(x) = |x|^n P_n^m(cos t) e^{i m f} / (n + m)!,   I_n^m(x) = (n - m)! P_n^m(cos t) e^{i m f} / |x|^(n+1),
// so that, by the addition theorem of the Legendre polynomials, for |y| < |x|
//   1/|x - y| = sum_n [ R_n^0(y) I_n^0(x) + 2 Re sum_{m >= 1} conj(R_n^m(y)) I_n^m(x) ].
// Both satisfy three-term recurrences in Cartesian coordinates (r^2 = |x|^2):
//   R_m^m = R_{m-1}^{m-1} (x + i y) / (2m),     R_n^m = [(2n-1) z R_{n-1}^m - r^2 R_{n-2}^m] / (n^2 - m^2),
//   I_m^m = I_{m-1}^{m-1} (2m-1)(x + i y) / r^2, I_n^m = [(2n-1) z I_{n-1}^m - ((n-1)^2 - m^2) I_{n-2}^m] / r^2,
// with R_0^0 = 1, I_0^0 = 1/r.  A node of centre c and radius rho stores the moments
// M_n^m = sum_j Q_j conj(R_n^m((y_j - c)/s)) in units of s, the power of two above rho (so that 1/s is
// exact and costs an integer operation), and gives phi(x) = (1/s) sum w_m Re(M_n^m I_n^m((x - c)/s))
// (w_0 = 1, w_m = 2).  The far images give L_n^m = sum_j Q_j conj(I_n^m(y_j/a)) and
// phi(x) = (1/a) sum w_m Re(L_n^m R_n^m(x/a)) inside the cavity.
// Shift of a child's moments (centre c', unit s') to the parent (c, s0): with b = (c' - c)/s0,
// s = s'/s0, and the solid harmonics continued to m < 0 in the Condon-Shortley convention
// (X_n^{-m} = conj(X_n^m), X_n^m -> (-1)^m X_n^m for m > 0), the addition theorem
// R_n^m(u + v) = sum_{j,k} R_j^k(u) R_{n-j}^{m-k}(v) of the regular harmonics gives
//   M_n^m = (-1)^m sum_{j <= n} s^j sum_k A_j^k conj(B_{n-j}^{m-k}),
//   A_j^k = (-1)^k M'_j^k (k >= 0), conj(M'_j^{-k}) (k < 0);  B_l^t = (-1)^t R_l^t(b) (t >= 0), conj(R_l^{-t}(b)) (t < 0).
// Moments are stored by column pair: (n, 2k) and (n, 2k + 1) side by side as (Re, Re, Im, Im), k
// outermost, rows n = 2k..P (the odd column's entry at n = 2k is zero), which is how the evaluation
// reads them; the far-image expansion by column, (n, m) at m (P + 1) - m (m - 1)/2 + (n - m).
#include <algorithm>
#include <cmath>

#include "df64.cuh"
#include "fp32_pair.cuh"
#include "tree.h"

namespace hsma {

__host__ __device__ constexpr int tree_col(int P, int m) { return m * (P + 1) - m * (m - 1) / 2; }
// entry (row n of pair k) of a node's moments
__host__ __device__ constexpr int tree_pair(int P, int k, int n) { return k * (P + 2 - k) + n - 2 * k; }

__device__ __forceinline__ void put_moment(float4* M, int P, int n, int m, float re, float im)
{
  float* e = reinterpret_cast<float*>(M + tree_pair(P, m >> 1, n)) + (m & 1);
  e[0] = re;
  e[2] = im;
  if ((m & 1) == 0 && n == m) e[1] = e[3] = 0.f;  // the odd column starts a row later
}
__device__ __forceinline__ float2 get_moment(const float4* M, int P, int n, int m)
{
  const float* e = reinterpret_cast<const float*>(M + tree_pair(P, m >> 1, n)) + (m & 1);
  return make_float2(e[0], e[2]);
}

// Whether a Kelvin record lies beyond kFarImageRel a (its high part, rounded without contraction,
// so that every kernel classifies a record the same way).
__device__ __forceinline__ bool far_image(float4 h, float rfar2)
{
  return __fadd_rn(__fadd_rn(__fmul_rn(h.x, h.x), __fmul_rn(h.y, h.y)), __fmul_rn(h.z, h.z)) > rfar2;
}

__device__ __forceinline__ float warp_min(float v)
{
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// Sums of 32 values over the warp's lanes, transposed: lane l returns the sum of value l, added
// pairwise in the order of a butterfly (lanes 16 apart first, then 8, 4, 2, 1).  31 shuffles, where a
// butterfly for each value takes 160.
__device__ __forceinline__ float warp_sums(float (&v)[32], int lane)
{
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int k = 0; k < o; ++k) {
      const float keep = up ? v[o + k] : v[k], give = up ? v[k] : v[o + k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return v[0];
}

// ---------------------------------------------------------------------------------------
// Record ranges: sorted position i starts node (l, c) if the previous record's key prefix
// differs, and ends it if the next one's does.  node[] is zeroed before (empty nodes keep 0, 0).
__global__ __launch_bounds__(256) void k_tree_marks(TreeView t)
{
  const SysDev& S = t.sys[0];
  const int n = S.n;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const long long c0 = S.chg;
  const int k = t.key[c0 + t.perm[c0 + i]];
  const int kp = i > 0 ? t.key[c0 + t.perm[c0 + i - 1]] : -1;
  const int kn = i + 1 < n ? t.key[c0 + t.perm[c0 + i + 1]] : -1;
  for (int l = kTreeTop; l <= t.L; ++l) {
    const int sh = 3 * (t.key_lv - l);
    const int id = k >> sh;
    const long long g = tree_node_index(l, id);
    if (i == 0 || (kp >> sh) != id) t.node[g].x = i;
    if (i == n - 1 || (kn >> sh) != id) t.node[g].y = i + 1;
  }
}

// ---------------------------------------------------------------------------------------
// Leaves: geometry and moments, a warp per (level-L node, tree).  Columns m and P - m together have
// P + 2 coefficients whatever m, 2 (P + 2) sums of one transposed reduction (two of them for order
// 16), and the records are read once per pair of columns: 36 and 216 us at N = 1e5 and 1e6, 98 and
// 555 with both trees in one warp and a butterfly per sum.
constexpr int kLeafWarps = 4;
template <int P>
__global__ __launch_bounds__(32 * kLeafWarps) void k_tree_leaf(TreeView t)
{
  constexpr int NQ = tree_nq(P);
  const int lane = threadIdx.x & 31;
  const long long c = (long long)blockIdx.x * kLeafWarps + (threadIdx.x >> 5);
  if (c >= (1LL << (3 * t.L))) return;  // whole warps
  const SysDev& S = t.sys[0];
  const int n = S.n;
  const long long nodes = tree_node_count(t.L);
  const long long g = tree_node_index(t.L, c);
  const int2 be = t.node[g];
  const float a = 1.f / t.inv_a;
  const int tr = blockIdx.y;
  const float4* __restrict__ H = t.hi + S.src + (long long)tr * n;
  const float4* __restrict__ Lo = t.lo + S.src + (long long)tr * n;
  float mn0 = 3.0e38f, mn1 = 3.0e38f, mn2 = 3.0e38f, mx0 = -3.0e38f, mx1 = -3.0e38f, mx2 = -3.0e38f;
  for (int j = be.x + lane; j < be.y; j += 32) {
    const float4 h = H[j];
    if (tr == 1 && far_image(h, t.rfar2)) continue;
    mn0 = fminf(mn0, h.x);
    mn1 = fminf(mn1, h.y);
    mn2 = fminf(mn2, h.z);
    mx0 = fmaxf(mx0, h.x);
    mx1 = fmaxf(mx1, h.y);
    mx2 = fmaxf(mx2, h.z);
  }
  mn0 = warp_min(mn0);
  mn1 = warp_min(mn1);
  mn2 = warp_min(mn2);
  mx0 = warp_max(mx0);
  mx1 = warp_max(mx1);
  mx2 = warp_max(mx2);
  float4* geo = t.geo + (long long)tr * nodes + g;
  float4* bx = t.box + 2 * ((long long)tr * nodes + g);
  float4* M = t.mom + ((long long)tr * nodes + g) * NQ;
  if (!(mn0 <= mx0)) {
    if (lane == 0) {
      *geo = make_float4(0.f, 0.f, 0.f, -1.f);
      bx[0] = make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.f);
      bx[1] = make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.f);
    }
    for (int k = lane; k < NQ; k += 32) M[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const float cx = 0.5f * (mn0 + mx0), cy = 0.5f * (mn1 + mx1), cz = 0.5f * (mn2 + mx2);
  float r2max = 0.f;
  for (int j = be.x + lane; j < be.y; j += 32) {
    const float4 h = H[j];
    if (tr == 1 && far_image(h, t.rfar2)) continue;
    const float dx = h.x - cx, dy = h.y - cy, dz = h.z - cz;
    r2max = fmaxf(r2max, dx * dx + dy * dy + dz * dz);
  }
  // (a margin for the rounding of the hi coordinates and of the distance)
  const float rho = sqrtf(warp_max(r2max)) * 1.000001f + 2e-7f * a + 1e-6f * a;
  if (lane == 0) {
    *geo = make_float4(cx, cy, cz, rho);
    bx[0] = make_float4(mn0, mn1, mn2, 0.f);
    bx[1] = make_float4(mx0, mx1, mx2, 0.f);
  }
  const float ir = inv_unit(rho);
#pragma unroll
  for (int m0 = 0; 2 * m0 <= P; ++m0) {
    constexpr int NC = P + 2;
    float cr[NC], ci[NC];  // column m0 (n = m0..P), then column P - m0
#pragma unroll
    for (int k = 0; k < NC; ++k) cr[k] = ci[k] = 0.f;
    for (int j = be.x + lane; j < be.y; j += 32) {
      const float4 h = H[j];
      if (tr == 1 && far_image(h, t.rfar2)) continue;
      const float4 l = Lo[j];
      const float vx = ((h.x - cx) + l.x) * ir, vy = ((h.y - cy) + l.y) * ir, vz = ((h.z - cz) + l.z) * ir;
      const float r2 = vx * vx + vy * vy + vz * vz;
      float dr = h.w, di = 0.f;  // Q R_m^m
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int m = half ? P - m0 : m0;
        if (half && 2 * m0 == P) break;
#pragma unroll
        for (int k = half ? m0 + 1 : 1; k <= m; ++k) {
          const float s = 0.5f / (float)k;
          const float nr = (dr * vx - di * vy) * s;
          di = (dr * vy + di * vx) * s;
          dr = nr;
        }
        const int at = half ? P - m0 + 1 : 0;
        float p0r = 0.f, p0i = 0.f, p1r = dr, p1i = di;
        cr[at] += p1r;
        ci[at] -= p1i;
#pragma unroll
        for (int nn = m + 1; nn <= P; ++nn) {
          const float A = (float)(2 * nn - 1) * vz;
          const float inv = 1.f / (float)(nn * nn - m * m);
          const float qr = (A * p1r - r2 * p0r) * inv, qi = (A * p1i - r2 * p0i) * inv;
          cr[at + nn - m] += qr;
          ci[at + nn - m] -= qi;
          p0r = p1r;
          p0i = p1i;
          p1r = qr;
          p1i = qi;
        }
      }
    }
    // lane k: the real parts of coefficient k, lane 16 + k (order 16: another reduction) the imaginary
    float sr, si;
    if constexpr (NC <= 16) {
      float v[32];
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        v[k] = k < NC ? cr[k] : 0.f;
        v[16 + k] = k < NC ? ci[k] : 0.f;
      }
      sr = warp_sums(v, lane);
      si = __shfl_xor_sync(0xffffffffu, sr, 16);
    } else {
      float v[32], u[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        v[k] = k < NC ? cr[k] : 0.f;
        u[k] = k < NC ? ci[k] : 0.f;
      }
      sr = warp_sums(v, lane);
      si = warp_sums(u, lane);
    }
    const int nc0 = P - m0 + 1;
    if (lane < (2 * m0 == P ? nc0 : NC)) {
      const int m = lane < nc0 ? m0 : P - m0, n_ = lane < nc0 ? m0 + lane : P - m0 + lane - nc0;
      put_moment(M, P, n_, m, sr, si);
    }
  }
}

// ---------------------------------------------------------------------------------------
// Upward pass, level l < L: a block per node and tree, a warp per child (order 16: per two
// children, for the shared memory), the children's shifted moments summed in child order.  Bound by
// the latency of a child's chain (stage, 91 sums of up to 91 products): a warp that walked the
// eight children took 250 us at each of the levels of 64 and 512 nodes (N = 1e5: the build and the
// rest of the step 1041 us, 576 us so).
template <int P>
constexpr int up_warps() { return P > 12 ? 4 : 8; }
template <int P>
__device__ __forceinline__ void decode_nm(int idx, int& n, int& m)
{
  m = 0;
  while (m < P && idx >= tree_col(P, m + 1)) ++m;
  n = m + (idx - tree_col(P, m));
}

template <int P>
__global__ __launch_bounds__(32 * (P > 12 ? 4 : 8)) void k_tree_up(TreeView t, int l)
{
  constexpr int NM = tree_nm(P), NQ = tree_nq(P);
  constexpr int W = P > 12 ? 4 : 8;
  constexpr int OUT = (NM + 31) / 32;
  constexpr int KW = 2 * P + 1;  // k = -P..P
  // per warp, for the child being shifted: A[j][k] = s^j A_j^k and B[l][t] = conj(B_l^t), dense
  // over -P <= k, t <= P (entries with |k| > j or |t| > l are never read)
  __shared__ float2 sAd[W][(P + 1) * KW], sBd[W][(P + 1) * KW];
  __shared__ float sPow[W][P + 1];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long c = blockIdx.x;
  const int tr = blockIdx.y;
  const long long nodes = tree_node_count(t.L);
  const long long g = tree_node_index(l, c);
  const long long g0 = tree_node_index(l + 1, 8 * c);
  const long long base = (long long)tr * nodes;
  float4 cg = make_float4(0.f, 0.f, 0.f, -1.f);
  float4 bmn = make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.f), bmx = make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.f);
  if (lane < 8) {
    cg = t.geo[base + g0 + lane];
    if (cg.w >= 0.f) {
      bmn = t.box[2 * (base + g0 + lane)];
      bmx = t.box[2 * (base + g0 + lane) + 1];
    }
  }
  const bool ne = lane < 8 && cg.w >= 0.f;
  const unsigned any = __ballot_sync(0xffffffffu, ne);
  float4* geo = t.geo + base + g;
  float4* bx = t.box + 2 * (base + g);
  float4* M = t.mom + (base + g) * NQ;
  if (!any) {  // (the same in every warp)
    if (threadIdx.x == 0) {
      *geo = make_float4(0.f, 0.f, 0.f, -1.f);
      bx[0] = make_float4(3.0e38f, 3.0e38f, 3.0e38f, 0.f);
      bx[1] = make_float4(-3.0e38f, -3.0e38f, -3.0e38f, 0.f);
    }
    for (int k = threadIdx.x; k < NQ; k += blockDim.x) M[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  const float mn0 = warp_min(bmn.x), mn1 = warp_min(bmn.y), mn2 = warp_min(bmn.z);
  const float mx0 = warp_max(bmx.x), mx1 = warp_max(bmx.y), mx2 = warp_max(bmx.z);
  const float cx = 0.5f * (mn0 + mx0), cy = 0.5f * (mn1 + mx1), cz = 0.5f * (mn2 + mx2);
  float rr = 0.f;
  if (ne) {
    const float dx = cg.x - cx, dy = cg.y - cy, dz = cg.z - cz;
    rr = sqrtf(dx * dx + dy * dy + dz * dz) + cg.w;
  }
  const float rho = warp_max(rr) * 1.000001f;
  if (threadIdx.x == 0) {
    *geo = make_float4(cx, cy, cz, rho);
    bx[0] = make_float4(mn0, mn1, mn2, 0.f);
    bx[1] = make_float4(mx0, mx1, mx2, 0.f);
  }
  const float irp = inv_unit(rho);
  int on[OUT], om[OUT];
#pragma unroll
  for (int q = 0; q < OUT; ++q) {
    const int idx = lane + 32 * q;
    if (idx < NM) {
      decode_nm<P>(idx, on[q], om[q]);
    } else {
      on[q] = -1;
      om[q] = 0;
    }
  }
  float2 acc[8 / W][OUT];
#pragma unroll
  for (int kk = 0; kk < 8 / W; ++kk) {
    const int k = w * (8 / W) + kk;
#pragma unroll
    for (int q = 0; q < OUT; ++q) acc[kk][q] = make_float2(0.f, 0.f);
    if (!((any >> k) & 1u)) continue;  // whole warps
    const float kx = __shfl_sync(0xffffffffu, cg.x, k), ky = __shfl_sync(0xffffffffu, cg.y, k);
    const float kz = __shfl_sync(0xffffffffu, cg.z, k), kr = __shfl_sync(0xffffffffu, cg.w, k);
    const float s = irp / inv_unit(kr);
    const float bxv = (kx - cx) * irp, byv = (ky - cy) * irp, bzv = (kz - cz) * irp;
    const float4* Mc = t.mom + (base + g0 + k) * NQ;
    if (lane <= P) {
      // column m = lane of R(b) into B (both signs of t), and s^lane
      const int m = lane;
      const float r2 = bxv * bxv + byv * byv + bzv * bzv;
      float dr = 1.f, di = 0.f;
      for (int j = 1; j <= m; ++j) {
        const float f = 0.5f / (float)j;
        const float nr = (dr * bxv - di * byv) * f;
        di = (dr * byv + di * bxv) * f;
        dr = nr;
      }
      const float sgn = (m & 1) ? -1.f : 1.f;
      float p0r = 0.f, p0i = 0.f, p1r = dr, p1i = di;
      for (int nn = m; nn <= P; ++nn) {
        if (nn > m) {
          const float A = (float)(2 * nn - 1) * bzv;
          const float inv = 1.f / (float)(nn * nn - m * m);
          const float qr = (A * p1r - r2 * p0r) * inv, qi = (A * p1i - r2 * p0i) * inv;
          p0r = p1r;
          p0i = p1i;
          p1r = qr;
          p1i = qi;
        }
        // conj(B_nn^m) = (-1)^m conj(R_nn^m); conj(B_nn^-m) = R_nn^m
        sBd[w][nn * KW + P + m] = make_float2(sgn * p1r, -sgn * p1i);
        if (m > 0) sBd[w][nn * KW + P - m] = make_float2(p1r, p1i);
      }
      float sp = 1.f;
      for (int j = 0; j < m; ++j) sp *= s;
      sPow[w][m] = sp;
    }
    __syncwarp();
    for (int e = lane; e < (P + 1) * KW; e += 32) {
      const int j = e / KW, kq = e - j * KW - P;
      if (kq > j || -kq > j) continue;
      const int ka = kq >= 0 ? kq : -kq;
      float2 A = get_moment(Mc, P, j, ka);
      if (kq >= 0) {
        if (kq & 1) A = make_float2(-A.x, -A.y);
      } else {
        A.y = -A.y;
      }
      const float sj = sPow[w][j];
      sAd[w][e] = make_float2(sj * A.x, sj * A.y);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < OUT; ++q) {
      const int n = on[q], m = om[q];
      if (n < 0) continue;
      float ar = 0.f, ai = 0.f;
      for (int j = 0; j <= n; ++j) {
        const int l2 = n - j;
        const int k0 = max(-j, m - l2), k1 = min(j, m + l2);
        const float2* Aj = &sAd[w][j * KW + P];
        const float2* Bl = &sBd[w][l2 * KW + P + m];  // Bl[-kq] = conj(B_{l2}^{m-kq})
        for (int kq = k0; kq <= k1; ++kq) {
          const float2 A = Aj[kq], B = Bl[-kq];
          ar = fmaf(A.x, B.x, ar);
          ar = fmaf(-A.y, B.y, ar);
          ai = fmaf(A.x, B.y, ai);
          ai = fmaf(A.y, B.x, ai);
        }
      }
      acc[kk][q] = make_float2(ar, ai);
    }
    __syncwarp();
  }
  // the children in order, through the warps' own (spent) tables
  __syncthreads();
  float2* sum = &sAd[0][0];  // [8][NM]
  static_assert(8 * tree_nm(P) <= W * (P + 1) * KW, "the children's moments fit the tables");
#pragma unroll
  for (int kk = 0; kk < 8 / W; ++kk)
#pragma unroll
    for (int q = 0; q < OUT; ++q)
      if (on[q] >= 0) sum[(w * (8 / W) + kk) * NM + lane + 32 * q] = acc[kk][q];
  __syncthreads();
  for (int i = threadIdx.x; i < NM; i += blockDim.x) {
    float2 v = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      v.x += sum[k * NM + i].x;
      v.y += sum[k * NM + i].y;
    }
    int n, m;
    decode_nm<P>(i, n, m);
    const float sg = (m & 1) ? -1.f : 1.f;
    put_moment(M, P, n, m, sg * v.x, sg * v.y);
  }
}

// ---------------------------------------------------------------------------------------
// Far images: L_n^m = sum Q conj(I_n^m(y/a)) over Kelvin records beyond kFarImageRel a.  A block takes
// batches of 32 records dealt out over the grid (far images are runs of the order: a block with its
// own run of records had all of the work or none), its warps the columns m = w, w + 8, ... of a batch
// (the latency of all 325 sums in one warp was the kernel: 87 and 373 us at N = 1e5 and 1e6; 62 and 213 so).
constexpr int kFarWarps = 8;
constexpr int kFarNM = tree_nm(kFarOrder);
__global__ __launch_bounds__(32 * kFarWarps) void k_tree_far(TreeView t)
{
  __shared__ float2 sum[kFarNM];  // the block's sums (a column belongs to one warp)
  __shared__ float2 acc[kFarWarps][kFarNM];
  __shared__ bool last;
  const SysDev& S = t.sys[0];
  const int n = S.n;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kFarNM; i += blockDim.x) sum[i] = make_float2(0.f, 0.f);
  __syncthreads();
  for (int j0 = 32 * blockIdx.x; j0 < n; j0 += 32 * gridDim.x) {
    const int j = j0 + lane;
    float4 h = make_float4(0.f, 0.f, 0.f, 0.f), lo = h;
    bool far = false;
    if (j < n) {
      h = t.hi[S.src + n + j];
      far = far_image(h, t.rfar2);
      if (far) lo = t.lo[S.src + n + j];
    }
    if (!__any_sync(0xffffffffu, far)) continue;
    // other lanes evaluate a dummy point 4a out on the x axis with zero strength
    const float Q = far ? h.w : 0.f;
    const float ux = far ? (h.x + lo.x) * t.inv_a : 4.f, uy = far ? (h.y + lo.y) * t.inv_a : 0.f;
    const float uz = far ? (h.z + lo.z) * t.inv_a : 0.f;
    const float r2 = ux * ux + uy * uy + uz * uz;
    const float i2 = __frcp_rn(r2);
    float dr = Q * rsqrt_mufu(r2), di = 0.f;  // Q I_0^0
#pragma unroll
    for (int m = 0; m <= kFarOrder; ++m) {
      if (m > 0) {
        const float f = (float)(2 * m - 1) * i2;
        const float nr = (dr * ux - di * uy) * f;
        di = (dr * uy + di * ux) * f;
        dr = nr;
      }
      if (m % kFarWarps != w) continue;  // whole warps
      float cr[kFarOrder + 1], ci[kFarOrder + 1];
      float p0r = 0.f, p0i = 0.f, p1r = dr, p1i = di;
      cr[0] = p1r;
      ci[0] = -p1i;
#pragma unroll
      for (int nn = m + 1; nn <= kFarOrder; ++nn) {
        const float A = (float)(2 * nn - 1) * uz, B = (float)((nn - 1) * (nn - 1) - m * m);
        const float qr = (A * p1r - B * p0r) * i2, qi = (A * p1i - B * p0i) * i2;
        cr[nn - m] = qr;
        ci[nn - m] = -qi;
        p0r = p1r;
        p0i = p1i;
        p1r = qr;
        p1i = qi;
      }
      float v[32], u[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) {
        v[k] = k <= kFarOrder - m ? cr[k] : 0.f;
        u[k] = k <= kFarOrder - m ? ci[k] : 0.f;
      }
      const float sr = warp_sums(v, lane), si = warp_sums(u, lane);
      if (lane <= kFarOrder - m) {
        float2& a = sum[tree_col(kFarOrder, m) + lane];
        a.x += sr;
        a.y += si;
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kFarNM; i += blockDim.x) t.farp[(long long)blockIdx.x * kFarNM + i] = sum[i];
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(t.ctr, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // warp w adds blocks w, w + kFarWarps, ..., then the warps' sums in order
  for (int i = lane; i < kFarNM; i += 32) {
    float2 s = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int b = w; b < (int)gridDim.x; b += kFarWarps) {
      const float2 v = __ldcg(t.farp + (long long)b * kFarNM + i);
      s.x += v.x;
      s.y += v.y;
    }
    acc[w][i] = s;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kFarNM; i += blockDim.x) {
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kFarWarps; ++q) {
      s.x += acc[q][i].x;
      s.y += acc[q][i].y;
    }
    t.farL[i] = s;
  }
  if (threadIdx.x == 0) *t.ctr = 0u;
}

// ---------------------------------------------------------------------------------------
// Evaluation.
// phi at target (th, tl) of a node's moments M (shared memory, stored to order P; centre and radius
// gc), the series truncated at order q <= P.
//
// I_n^m = Q_n^m z^m with z = (x + i y)/r^2 and a real recurrence in n: Q_m^m = (2m-1)!!/r,
// Q_n^m = (2n-1) w Q_{n-1}^m - ((n-1)^2 - m^2) Q_{n-2}^m / r^2, w = z/r^2.  So the column sums
// C_m = sum_n M_n^m Q_n^m take, per coefficient, the recurrence once (not for a real and an imaginary
// part) and two multiply-adds, and z enters in one Horner sum of 2 Re sum_m C_m z^m.  Packed FP32 over
// the columns 2k, 2k + 1 (FFMA2 / FMUL2): per two coefficients one 16-byte shared load, the two
// factors of Q_{n-2}, three operations of the recurrence and two of the sums -- 3.5 instructions a
// coefficient where the recurrence on (Re, Im) took 5.  The columns run in two groups so that the state
// (two rows and the sums) fits the registers of 24 warps per SM (one group spills: N = 1e6 22.4 ms at 16
// warps; three groups at 28 warps 20.1).  The evaluation is issue-bound
// (76 % of the slots): with this series, the direct sums relative to the node's centre and one
// reduction for the three tests of a node it takes 1.75 ms at N = 1e5 and 19.9 ms at N = 1e6 (theta =
// 0.5, order 12; 2.47 and 24.2 ms before), at the same error (7.6e-8 at N = 1e5).
template <int P, int K0, int K1>
__device__ __forceinline__ void series_group(const float4* M, float wz, float i2, float ri, int q,
                                             float2 (&CR)[K1 - K0], float2 (&CI)[K1 - K0])
{
  constexpr int NK = K1 - K0;
  float2 a[NK], b[NK];
#pragma unroll
  for (int k = 0; k < NK; ++k) a[k] = b[k] = CR[k] = CI[k] = make_float2(0.f, 0.f);
#pragma unroll
  for (int n = 2 * K0; n <= P; ++n) {
    if (n > q) break;
    const float A = (float)(2 * n - 1) * wz;
    const float2 A2 = make_float2(A, A);
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const int m = 2 * (K0 + k);
      if (n < m) continue;
      float2 v;
      if (n == m) {
        float f = ri;  // (2m - 1)!! / r
#pragma unroll
        for (int j = 1; j < 2 * m; j += 2) f *= (float)j;
        v = make_float2(f, 0.f);
      } else {
        const float2 B2 = make_float2((float)(m * m - (n - 1) * (n - 1)) * i2,
                                      (float)((m + 1) * (m + 1) - (n - 1) * (n - 1)) * i2);
        v = __ffma2_rn(B2, b[k], __fmul2_rn(A2, a[k]));
        if (n == m + 1) {
          float f = ri;
#pragma unroll
          for (int j = 1; j < 2 * (m + 1); j += 2) f *= (float)j;
          v.y = f;
        }
      }
      b[k] = a[k];
      a[k] = v;
      const float4 mm = M[tree_pair(P, K0 + k, n)];
      CR[k] = __ffma2_rn(make_float2(mm.x, mm.y), v, CR[k]);
      CI[k] = __ffma2_rn(make_float2(mm.z, mm.w), v, CI[k]);
    }
  }
}

// S <- S z + C
__device__ __forceinline__ void horner(float& sr, float& si, float zx, float zy, float cr, float ci)
{
  const float nr = fmaf(sr, zx, fmaf(-si, zy, cr));
  si = fmaf(sr, zy, fmaf(si, zx, ci));
  sr = nr;
}

// Column pairs K0..K1 - 1 of the series, added to the Horner sum (s <- s z^(2 (K1 - K0)) + ...); the
// real column m = 0 (K0 = 0) is returned and left out.
template <int P, int K0, int K1>
__device__ __forceinline__ float series_add(const float4* M, float wz, float i2, float ri, int q, float px, float py,
                                            float& sr, float& si)
{
  if (K0 > 0 && q < 2 * K0) return 0.f;
  float2 CR[K1 - K0], CI[K1 - K0];
  series_group<P, K0, K1>(M, wz, i2, ri, q, CR, CI);
#pragma unroll
  for (int k = K1 - K0 - 1; k >= 0; --k) {
    horner(sr, si, px, py, CR[k].y, CI[k].y);
    if (K0 + k > 0) horner(sr, si, px, py, CR[k].x, CI[k].x);
  }
  return CR[0].x;
}

template <int P>
__device__ __forceinline__ float m2p(const float4* M, float4 gc, float4 th, float4 tl, int q)
{
  constexpr int KP = P / 2 + 1;  // column pairs
  const float ir = inv_unit(gc.w);
  const float ux = ((th.x - gc.x) + tl.x) * ir, uy = ((th.y - gc.y) + tl.y) * ir, uz = ((th.z - gc.z) + tl.z) * ir;
  const float r2 = ux * ux + uy * uy + uz * uz;
  float i2 = __fdividef(1.f, r2);
  i2 = fmaf(i2, fmaf(-r2, i2, 1.f), i2);  // (a Newton step: 1/r2 to its rounding, as a division)
  const float ri = rsqrt_mufu(r2);
  const float px = ux * i2, py = uy * i2, wz = uz * i2;
  float sr = 0.f, si = 0.f;
  // groups of column pairs, the highest first
  series_add<P, P / 4, KP>(M, wz, i2, ri, q, px, py, sr, si);
  const float c0 = series_add<P, 0, P / 4>(M, wz, i2, ri, q, px, py, sr, si);
  return fmaf(2.f, fmaf(sr, px, -si * py), c0) * ir;
}

// phi at the target of the far images' expansion (|x| < a)
__device__ __forceinline__ float l2p_far(const float2* __restrict__ L, float4 th, float4 tl, float inv_a)
{
  const float ux = (th.x + tl.x) * inv_a, uy = (th.y + tl.y) * inv_a, uz = (th.z + tl.z) * inv_a;
  const float r2 = ux * ux + uy * uy + uz * uz;
  float dr = 1.f, di = 0.f;  // R_0^0
  float acc = 0.f;
  // (once per Kelvin item: rolled loops keep the registers for the traversal)
#pragma unroll 1
  for (int m = 0; m <= kFarOrder; ++m) {
    if (m > 0) {
      const float f = 0.5f / (float)m;
      const float nr = (dr * ux - di * uy) * f;
      di = (dr * uy + di * ux) * f;
      dr = nr;
    }
    const float2* Lc = L + tree_col(kFarOrder, m);
    float2 ll = __ldg(Lc);
    float col = ll.x * dr - ll.y * di;
    float p0r = 0.f, p0i = 0.f, p1r = dr, p1i = di;
#pragma unroll 1
    for (int nn = m + 1; nn <= kFarOrder; ++nn) {
      const float A = (float)(2 * nn - 1) * uz;
      const float inv = 1.f / (float)(nn * nn - m * m);
      const float qr = (A * p1r - r2 * p0r) * inv, qi = (A * p1i - r2 * p0i) * inv;
      ll = __ldg(Lc + (nn - m));
      col = fmaf(ll.x, qr, col);
      col = fmaf(-ll.y, qi, col);
      p0r = p1r;
      p0i = p1i;
      p1r = qr;
      p1i = qi;
    }
    acc += m == 0 ? col : 2.f * col;
  }
  return acc * inv_a;
}

// Direct sum of the records [be.x, be.y) of a node at the lane's target, staged 32 at a time through
// the warp's shared buffer; two sources per step as packed FP32, side by side in the buffer (a
// source past the range is far away and has no charge).
//  EXACT: with the (hi, lo) coordinate difference of inv_hilo (accurate to FP32 rounding at any
//    distance, e.g. a charge next to its own Kelvin image); checked: the node holds some of the
//    group's own targets, and the source at sorted position `self` is skipped.
//  Otherwise, for a node whose radius is at most kRelRadius times its distance from every target:
//    the difference of the FP32 coordinates relative to the node's centre c.  Two roundings form a
//    coordinate (its hi part less the centre's, which is mostly exact, and the lo part), one the
//    difference; with d >= |t - c| - rho the distance d is off by at most u (1 + 2 (1 + r)/(1 - r)) = 9 u
//    = 5.4e-7 of it (u = 2^-24, r = kRelRadius), of either sign.  9 operations for two pairs instead of
//    15, half the shared loads and half the staging; nine tenths of the direct pairs at N = 1e5 (step
//    2.27 ms, 2.66 with hi/lo differences throughout; 23.4 and 24.5 at N = 1e6).  Over 40 drawn cavities
//    (N = 20000 to 200000, theta 0.4 to 0.6, orders 8, 12 and 16) the potentials' errors against the FP64
//    path are 1.0008 times those with hi/lo differences throughout, and 0.866 times those before the
//    series by column pairs.
// kelvin: records beyond rfar2 count as zero.  Each batch's FP32 sum is added to the compensated
// total (a leaf of a dense cluster holds thousands of sources of similar size and mixed sign).
constexpr float kRelRadius = 0.6f;
struct P2PShared {
  float x[32], y[32], z[32], q[32], lx[32], ly[32], lz[32];
};
template <bool EXACT>
__device__ __forceinline__ void p2p(const float4* __restrict__ H, const float4* __restrict__ Lo, int2 be, float4 gc,
                                    float4 th, float4 tl, int self, bool checked, bool kelvin, float rfar2,
                                    P2PShared& sh, df& total)
{
  const int lane = threadIdx.x & 31;
  // EXACT: the target's hi parts, else its coordinates relative to the centre
  const float tx = EXACT ? th.x : (th.x - gc.x) + tl.x, ty = EXACT ? th.y : (th.y - gc.y) + tl.y,
              tz = EXACT ? th.z : (th.z - gc.z) + tl.z;
  const float2 X = make_float2(tx, tx), Y = make_float2(ty, ty), Z = make_float2(tz, tz);
  for (int j0 = be.x; j0 < be.y; j0 += 32) {
    const int j = j0 + lane;
    float4 h = make_float4(1.0e18f, 0.f, 0.f, 0.f), l = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j < be.y) {
      h = H[j];
      l = Lo[j];
      if (kelvin && far_image(h, rfar2)) h.w = 0.f;
    }
    __syncwarp();  // the previous batch has been read
    // (negated: the differences are sums)
    sh.x[lane] = EXACT ? -h.x : -((h.x - gc.x) + l.x);
    sh.y[lane] = EXACT ? -h.y : -((h.y - gc.y) + l.y);
    sh.z[lane] = EXACT ? -h.z : -((h.z - gc.z) + l.z);
    sh.q[lane] = h.w;
    if (EXACT) {
      sh.lx[lane] = -l.x;
      sh.ly[lane] = -l.y;
      sh.lz[lane] = -l.z;
    }
    __syncwarp();
    const int m = min(32, be.y - j0);
    float2 acc = make_float2(0.f, 0.f);  // one batch of 32 sources
#pragma unroll 2
    for (int k = 0; k < m; k += 4) {
      float4 f[7];
      f[0] = *reinterpret_cast<const float4*>(&sh.x[k]);
      f[1] = *reinterpret_cast<const float4*>(&sh.y[k]);
      f[2] = *reinterpret_cast<const float4*>(&sh.z[k]);
      f[3] = *reinterpret_cast<const float4*>(&sh.q[k]);
      if (EXACT) {
        f[4] = *reinterpret_cast<const float4*>(&sh.lx[k]);
        f[5] = *reinterpret_cast<const float4*>(&sh.ly[k]);
        f[6] = *reinterpret_cast<const float4*>(&sh.lz[k]);
      }
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        auto two = [&](int i) { return p ? make_float2(f[i].z, f[i].w) : make_float2(f[i].x, f[i].y); };
        float2 ex = __fadd2_rn(X, two(0)), ey = __fadd2_rn(Y, two(1)), ez = __fadd2_rn(Z, two(2));
        if (EXACT) {
          ex = __fadd2_rn(__fadd2_rn(make_float2(tl.x, tl.x), two(4)), ex);
          ey = __fadd2_rn(__fadd2_rn(make_float2(tl.y, tl.y), two(5)), ey);
          ez = __fadd2_rn(__fadd2_rn(make_float2(tl.z, tl.z), two(6)), ez);
        }
        const float2 r2 = __ffma2_rn(ez, ez, __ffma2_rn(ey, ey, __fmul2_rn(ex, ex)));
        float2 inv = make_float2(rsqrt_mufu(r2.x), rsqrt_mufu(r2.y));
        if (EXACT && checked) {  // the target itself
          if (j0 + k + 2 * p == self) inv.x = 0.f;
          if (j0 + k + 2 * p + 1 == self) inv.y = 0.f;
        }
        acc = __ffma2_rn(two(3), inv, acc);
      }
    }
    total = total + two_sum(acc.x, acc.y);
  }
}

// One work item: a group of 32 consecutive targets (sorted positions 32 grp ..) against the
// subtrees of one tree below root cells [rs R/kTreeRootSplit, (rs + 1) R/kTreeRootSplit) (tr = 0:
// real charges, 1: Kelvin images, the far-image expansion with rs = 0); traversal and evaluation,
// written to the item's own partial row (chunk tr kTreeRootSplit + rs).
template <int P>
__device__ __forceinline__ void eval_group(const TreeView& t, float2* __restrict__ part, int grp, int tr, int rs,
                                           int* stk, int2* sbe, float4* sgc, P2PShared& sp2, float4* smom)
{
  constexpr int NQ = tree_nq(P);
  const int lane = threadIdx.x & 31;
  const SysDev& S = t.sys[0];
  const int n = S.n;
  const int i = grp * 32 + lane;
  const bool on = i < n;
  const int ic = on ? i : n - 1;
  const float4 th = t.hi[S.src + ic], tl = t.lo[S.src + ic];
  const float theta2 = t.theta * t.theta, margin = 4e-7f / t.inv_a;
  const long long nodes = tree_node_count(t.L);
  df acc = df_make(0.f, 0.f);
  constexpr int R = 1 << (3 * kTreeTop);
  {
    const float4* __restrict__ H = t.hi + S.src + (long long)tr * n;
    const float4* __restrict__ Lo = t.lo + S.src + (long long)tr * n;
    const float4* __restrict__ G = t.geo + (long long)tr * nodes;
    const float4* __restrict__ MM = t.mom + (long long)tr * nodes * NQ;
    const int self = tr == 0 ? i : -1;
    __syncwarp();
    constexpr int RS = R / kTreeRootSplit;
    static_assert(RS <= 32, "a lane per root of an item");
    // depth first: an opened node leaves at most 8 - 1 more entries, once per level below the roots
    static_assert(RS + 7 * (kTreeMaxLevel - kTreeTop) <= kTreeStack, "traversal stack depth");
    int sp = 0;
    {
      // the item's roots with sources, the lowest cell on top; a stack entry carries the node's
      // record range and geometry, read when it is pushed (eight or fewer loads side by side)
      const long long gr = tree_node_index(kTreeTop, rs * RS + lane);
      int2 rb = make_int2(0, 0);
      float4 rgc = make_float4(0.f, 0.f, 0.f, -1.f);
      if (lane < RS) {
        rb = t.node[gr];
        if (rb.y > rb.x) rgc = G[gr];
      }
      const unsigned ok = __ballot_sync(0xffffffffu, lane < RS && rb.y > rb.x && rgc.w >= 0.f);
      if (lane < RS && ((ok >> lane) & 1u)) {
        const int at = __popc(ok >> (lane + 1));
        stk[at] = (kTreeTop << 26) | (rs * RS + lane);
        sbe[at] = rb;
        sgc[at] = rgc;
      }
      sp = __popc(ok);
      __syncwarp();
    }
    while (sp > 0) {
      --sp;
      const int e = stk[sp];
      const int2 be = sbe[sp];
      const float4 gc = sgc[sp];
      __syncwarp();  // every lane has read the entry before a push overwrites it
      const int l = e >> 26, c = e & ((1 << 26) - 1);
      const int g = (int)tree_node_index(l, 0) + c;  // (levels to 7: below 2^22)
      // the node is far when its series converges with ratio rho / |t - c| <= theta at every
      // target of the group (each lane tests its own target; a margin covers the lo parts)
      const float dx = th.x - gc.x, dy = th.y - gc.y, dz = th.z - gc.z;
      const float rm = gc.w + margin;
      // (the nearest target decides: one reduction serves the three tests of the node)
      const float d2 = __uint_as_float(
          __reduce_min_sync(0xffffffffu, __float_as_uint(fmaf(dz, dz, fmaf(dy, dy, dx * dx)))));
      const bool far = rm * rm <= theta2 * d2;
      if (far && be.y - be.x >= t.cmin) {
        // the order whose truncation at the group's largest ratio rho/|t - c| stays within a tenth
        // of the order-P bound at theta: (q + 1) log(ratio) <= log(0.1 theta^(P+1)) (the divisions'
        // last bits move an order only next to a whole number); order 16 keeps every node at its order
        int q = P;
        if constexpr (P <= 12) {
          q = min(P, max(2, (int)ceilf(__fdividef(t.log_eps, 0.5f * __logf(__fdividef(rm * rm, d2)))) - 1));
        }
        // the node's moments staged in shared memory by coalesced warp loads
        const float4* src = MM + (size_t)g * NQ;
        for (int i = lane; i < NQ; i += 32) smom[i] = __ldg(src + i);
        __syncwarp();
        acc = acc + two_sum(m2p<P>(smom, gc, th, tl, q), 0.f);
        __syncwarp();
      } else if (far || l == t.L) {
        if (rm * rm <= kRelRadius * kRelRadius * d2) {
          p2p<false>(H, Lo, be, gc, th, tl, -1, false, tr == 1, t.rfar2, sp2, acc);
        } else {
          const bool checked = tr == 0 && be.x < grp * 32 + 32 && be.y > grp * 32;
          p2p<true>(H, Lo, be, gc, th, tl, self, checked, tr == 1, t.rfar2, sp2, acc);
        }
      } else {
        // open: the children with sources, the lowest cell on top
        const int gch = 8 * g + 1;  // the first child: 8 ((8^l - 1)/7 + c) + 1
        int2 cb = make_int2(0, 0);
        float4 cg = make_float4(0.f, 0.f, 0.f, -1.f);
        if (lane < 8) {
          cb = t.node[gch + lane];
          if (cb.y > cb.x) cg = G[gch + lane];
        }
        const unsigned ne = __ballot_sync(0xffffffffu, lane < 8 && cb.y > cb.x && cg.w >= 0.f);
        if (lane < 8 && ((ne >> lane) & 1u)) {
          const int at = sp + __popc(ne >> (lane + 1));
          stk[at] = ((l + 1) << 26) | (8 * c + lane);
          sbe[at] = cb;
          sgc[at] = cg;
        }
        sp += __popc(ne);
        __syncwarp();
      }
    }
  }
  if (tr == 1 && rs == 0) acc = acc + two_sum(l2p_far(t.farL, th, tl, t.inv_a), 0.f);
  if (on) part[S.part + (long long)(tr * kTreeRootSplit + rs) * n + i] = make_float2(acc.hi, acc.lo);
}

template <int P>
__global__ __launch_bounds__(32 * kTreeEvalWarps, kTreeEvalMinBlocks) void k_tree_eval(TreeView t,
                                                                                       float2* __restrict__ part)
{
  constexpr int NQ = tree_nq(P);
  __shared__ int s_stack[kTreeEvalWarps][kTreeStack];
  __shared__ int2 s_sbe[kTreeEvalWarps][kTreeStack];
  __shared__ float4 s_sgc[kTreeEvalWarps][kTreeStack];
  __shared__ float4 s_mom[kTreeEvalWarps][NQ];
  __shared__ __align__(16) P2PShared s_p2p[kTreeEvalWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const SysDev& S = t.sys[0];
  const int n = S.n;
  constexpr int IPG = 2 * kTreeRootSplit;  // items per group
  const int items = IPG * ((n + 31) / 32), workers = gridDim.x * kTreeEvalWarps;
  // persistent warps: the first item by the warp's index, then items from the work counter (the
  // cost of an item varies with its distance from the interface and from the centre)
  for (int it = blockIdx.x * kTreeEvalWarps + w; it < items;) {
    const int r = it % IPG;
    eval_group<P>(t, part, it / IPG, r & 1, r >> 1, s_stack[w], s_sbe[w], s_sgc[w], s_p2p[w], s_mom[w]);
    int nx = 0;
    if (lane == 0) nx = workers + (int)atomicAdd(t.ctr + 1, 1u);
    it = __shfl_sync(0xffffffffu, nx, 0);
  }
}

// ---------------------------------------------------------------------------------------
int tree_levels(long long n)
{
  // leaves of ~25-50 charges for charges spread through the ball (52 % of the cube)
  const double v = std::log(std::max<double>((double)n, 1.0) / 25.0) / std::log(8.0);
  return std::min(kTreeMaxLevel, std::max(3, (int)std::lround(v)));
}

bool tree_order_supported(int P) { return P == 8 || P == 12 || P == 16; }

template <int P>
static void build_p(const TreeView& t, int n, cudaStream_t st)
{
  const long long leaves = 1LL << (3 * t.L);
  k_tree_leaf<P><<<dim3((unsigned)((leaves + kLeafWarps - 1) / kLeafWarps), 2), 32 * kLeafWarps, 0, st>>>(t);
  for (int l = t.L - 1; l >= kTreeTop; --l) {
    const long long cells = 1LL << (3 * l);
    k_tree_up<P><<<dim3((unsigned)cells, 2), 32 * up_warps<P>(), 0, st>>>(t, l);
  }
}

void launch_tree_build(const TreeView& t, int n, cudaStream_t st)
{
  cudaMemsetAsync(t.node, 0, sizeof(int2) * (size_t)tree_node_count(t.L), st);
  cudaMemsetAsync(t.ctr, 0, 2 * sizeof(unsigned int), st);  // k_tree_far's and k_tree_eval's counters
  if (n <= 0) return;
  k_tree_marks<<<(n + 255) / 256, 256, 0, st>>>(t);
  if (t.P == 8) build_p<8>(t, n, st);
  else if (t.P == 12) build_p<12>(t, n, st);
  else build_p<16>(t, n, st);
  k_tree_far<<<kFarBlocks, 32 * kFarWarps, 0, st>>>(t);
}

void launch_tree_eval(const TreeView& t, int n, float2* part, cudaStream_t st)
{
  if (n <= 0) return;
  static int sms = 0;
  if (!sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 1;
  }
  const int items = 2 * kTreeRootSplit * ((n + 31) / 32);
  const unsigned blocks = (unsigned)std::min<long long>((items + kTreeEvalWarps - 1) / kTreeEvalWarps,
                                                        (long long)sms * kTreeEvalMinBlocks);
  if (t.P == 8) k_tree_eval<8><<<blocks, 32 * kTreeEvalWarps, 0, st>>>(t, part);
  else if (t.P == 12) k_tree_eval<12><<<blocks, 32 * kTreeEvalWarps, 0, st>>>(t, part);
  else k_tree_eval<16><<<blocks, 32 * kTreeEvalWarps, 0, st>>>(t, part);
}

}  // namespace hsma
