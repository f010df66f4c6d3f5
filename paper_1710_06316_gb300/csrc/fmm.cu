// fmm.cu -- far-field sums of the node-patch operator: adaptive FMM + point-to-point.
//
// For x = [f; h] every source node t carries a charge c_t = a_t h_t and a dipole
// strength g_t = -a_t f_t along its normal n_t (Eq. 6 with the far rule: integrand
// constant on the patch).  With G = 1/(4 pi r), u = exp(-kappa r)/(4 pi r) and the
// dipole entering as d . grad_y, the four far sums of the solution flow (Sec. 2,
// step 3b: single- and double-layer Laplace and Yukawa) are
//     PhiL(p) = sum_t c_t G + (g_t / eps_bar) n_t . grad_y G
//     PhiY(p) = sum_t c_t u + g_t n_t . grad_y u
// and their target normal derivatives n_p . grad_x.  They are evaluated together in one
// tree pass (the "ViewSet" idea of Sec. 3.1): every box carries one Laplace and one
// Yukawa expansion.
//
// Expansions: tensor-product Chebyshev interpolation of the kernel on each box
// (n = order points per dimension, n^3 weights per box and kernel).  The same
// weights serve the single and the double layer (Sec. 3.2 notes the two share their
// expansion form): the dipole enters P2M through the gradient of the interpolating
// polynomial, and the normal derivative leaves L2P the same way.  M2L is a dense
// n^3 x n^3 kernel matrix per (level, offset); the paper's FMM97 plane-wave M2L is
// replaced by these dense translations, which are contractions suited to the GPU.
//
// Lists: 1 and 3 by P2P (Sec. 3.2 modified method), 2 by M2L, 4 by P2L (S_to_L).
#include <cmath>
#include <mutex>

#include "internal.cuh"

namespace afmpb {

// Per-order tables (index = order n), written once per device before the first handle
// uses them, so that handles of different orders can run side by side.
__constant__ float c_cheb[kMaxOrder + 1][kMaxOrder * kMaxOrder];     // Cm[m][k] = w_k T_k(x_m)
__constant__ float c_m2m[kMaxOrder + 1][2 * kMaxOrder * kMaxOrder];  // S2[c][m][m']
__constant__ float c_nodes[kMaxOrder + 1][kMaxOrder];                // Chebyshev points on [-1, 1]

// s_m(x) and s_m'(x) for the n interpolation polynomials.
template <int N>
__device__ __forceinline__ void cheb_basis(float x, float s[N], float ds[N]) {
  float T[N], dT[N];
  T[0] = 1.0f;
  dT[0] = 0.0f;
  if (N > 1) {
    T[1] = x;
    dT[1] = 1.0f;
  }
#pragma unroll
  for (int k = 2; k < N; ++k) {
    T[k] = 2.0f * x * T[k - 1] - T[k - 2];
    dT[k] = 2.0f * T[k - 1] + 2.0f * x * dT[k - 1] - dT[k - 2];
  }
#pragma unroll
  for (int m = 0; m < N; ++m) {
    float a = 0.0f, b = 0.0f;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      a = fmaf(c_cheb[N][m * kMaxOrder + k], T[k], a);
      b = fmaf(c_cheb[N][m * kMaxOrder + k], dT[k], b);
    }
    s[m] = a;
    ds[m] = b;
  }
}

// 1 / w of a box of `level` (w = w0 2^-level; the power of two is exact).
__device__ __forceinline__ float inv_width(float inv_w0, int level) { return ldexpf(inv_w0, level); }

__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// ------------------------------------------------------------------------------------
// P2M: leaf sources -> Laplace and Yukawa multipole weights.
//   A[ijk] += c Sx[i] (Sy[j] Sz[k]),  B[ijk] += dSx[i] (g_x Sy Sz) + Sx[i] (g_y dSy Sz + g_z Sy dSz)
// Lane (part, k) holds the weights (., j, k) of both sums for JL of the j, so that a node's
// factors are read once per N JL weights, and the x direction runs on packed FP32 pairs.
// Each weight adds its leaf's nodes in order.  Two shapes, with the same sums:
//   * many leaves (kWide false): half of the j to a lane, 2 N lanes to a leaf, so N = 6 puts
//     two leaves in a warp, N = 8 two, N = 4 four.  Instruction issue bounds it: a thread per
//     (j, k) with N weights took 3.3 times the instructions and left 28 of 64 lanes idle at
//     N = 6 (35.8 us on the 163,842-node sphere, alone).
//   * few leaves at odd orders (kWide), where the other shape stages 6, 10 or 16 nodes of a leaf
//     at a time and has lanes without a last j: a warp to a leaf, all lanes staging its nodes,
//     and one or two j to a lane.  The chain of a leaf's nodes bounds it: order 3 on 10,242
//     nodes 42 us in the other shape, 20 so, 163,842 nodes 57 / 29; order 5 on 642 nodes 24 / 14.
// ------------------------------------------------------------------------------------
constexpr int kP2MWarps = 4;        // warps per CTA
// kWide at odd orders, up to this many warps of the other shape per SM (at even orders it gains
// a few us of P2M and nothing in a product).
constexpr int kP2MWideWarps = 12;
template <int N>
constexpr bool kP2MHasWide = N % 2 == 1;

template <int N, bool kWide>
struct P2MShape {
  static constexpr int H = (N + 1) / 2;               // packed pairs along x
  static constexpr int JL = !kWide ? H : N * N <= 32 ? 1 : 2;   // j of a lane
  static constexpr int G = (N + JL - 1) / JL * N;     // lanes of a leaf
  static constexpr int Leaves = kWide ? 1 : 32 / G;   // leaves of a warp
  static constexpr int CH = 32 / Leaves;              // nodes of a leaf staged at a time
  static_assert(G <= 32, "a leaf's lanes are of one warp");
  // a node's row: Sx (2 H), dSx (2 H), (Sy, Sy, dSy, dSy) per j, (Sz, dSz) per k, (c, gx, gy, gz)
  static constexpr int oY = 4 * H, oZ = oY + 4 * N, oW = (oZ + 2 * N + 3) & ~3, Row = oW + 4;
};

template <int N, bool kWide>
__global__ void __launch_bounds__(32 * kP2MWarps) k_p2m(int nleaf, const int4 *__restrict__ leaf_rec,
                                                        float inv_w0, const float4 *__restrict__ pos,
                                                        const float4 *__restrict__ nrm, const float2 *__restrict__ xs,
                                                        float inv_ebar, float *__restrict__ M) {
  using P = P2MShape<N, kWide>;
  constexpr int N3 = N * N * N, H = P::H, JL = P::JL, CH = P::CH;
  __shared__ __align__(16) float sm[kP2MWarps][32 * P::Row];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l0 = (blockIdx.x * kP2MWarps + warp) * P::Leaves;
  if (l0 >= nleaf) return;                              // whole warps
  after_previous();
  float *buf = sm[warp];
  const int sub = lane / P::G, part = lane % P::G / N, k = lane % N;   // this lane's weights
  const int ssub = lane / CH, snode = lane % CH;                       // the node that it stages
  const int4 none = make_int4(0, 0, 0, 0);
  const int4 rec = sub < P::Leaves && l0 + sub < nleaf ? leaf_rec[l0 + sub] : none;
  const int4 srec = ssub < P::Leaves && l0 + ssub < nleaf ? leaf_rec[l0 + ssub] : none;
  const int nodes = rec.z - rec.y, snodes = srec.z - srec.y;
  const int most = __reduce_max_sync(0xffffffffu, nodes);
  const float invw = inv_width(inv_w0, srec.w);
  float2 A[JL][H], B[JL][H];
#pragma unroll
  for (int j = 0; j < JL; ++j)
#pragma unroll
    for (int i = 0; i < H; ++i) A[j][i] = B[j][i] = make_float2(0.f, 0.f);
  float4 pn = make_float4(0.f, 0.f, 0.f, 0.f), qn = pn;  // the next chunk's node, read ahead
  float2 fn = make_float2(0.f, 0.f);
  auto fetch = [&](int c0) {
    if (c0 + snode >= snodes) return;
    const int t = srec.y + c0 + snode;
    pn = pos[t];
    qn = nrm[t];
    fn = xs[t];
  };
  fetch(0);
  for (int c0 = 0; c0 < most; c0 += CH) {
    const float4 p = pn, q = qn;
    const float2 fh = fn;
    fetch(c0 + CH);
    if (c0 + snode < snodes) {
      float *row = buf + (ssub * CH + snode) * P::Row;
      float s[N], ds[N];
      cheb_basis<N>(p.x * invw, s, ds);
#pragma unroll
      for (int i = 0; i < H; ++i) {
        const bool two = 2 * i + 1 < N;
        *reinterpret_cast<float2 *>(row + 2 * i) = make_float2(s[2 * i], two ? s[(2 * i + 1) % N] : 0.f);
        *reinterpret_cast<float2 *>(row + 2 * H + 2 * i) = make_float2(ds[2 * i], two ? ds[(2 * i + 1) % N] : 0.f);
      }
      cheb_basis<N>(p.y * invw, s, ds);
#pragma unroll
      for (int j = 0; j < N; ++j)
        *reinterpret_cast<float4 *>(row + P::oY + 4 * j) = make_float4(s[j], s[j], ds[j], ds[j]);
      cheb_basis<N>(p.z * invw, s, ds);
#pragma unroll
      for (int m = 0; m < N; ++m) *reinterpret_cast<float2 *>(row + P::oZ + 2 * m) = make_float2(s[m], ds[m]);
      const float g = -p.w * fh.x * invw;
      *reinterpret_cast<float4 *>(row + P::oW) = make_float4(p.w * fh.y, g * q.x, g * q.y, g * q.z);
    }
    __syncwarp();
    const int cnt = min(CH, nodes - c0);
#pragma unroll 2
    for (int t = 0; t < cnt; ++t) {
      const float *row = buf + (sub * CH + t) * P::Row;
      const float4 w = *reinterpret_cast<const float4 *>(row + P::oW);
      const float2 z = *reinterpret_cast<const float2 *>(row + P::oZ + 2 * k);
      float2 x[H], dx[H];
#pragma unroll
      for (int i = 0; i < H; ++i) {
        x[i] = *reinterpret_cast<const float2 *>(row + 2 * i);
        dx[i] = *reinterpret_cast<const float2 *>(row + 2 * H + 2 * i);
      }
      const float2 sz = dup2(z.x), dsz = dup2(z.y);
      const float2 wc = dup2(w.x), wx = dup2(w.y), wy = dup2(w.z), wz = dup2(w.w);
#pragma unroll
      for (int jj = 0; jj < JL; ++jj) {
        const int j = part * JL + jj;                   // the last part of an odd N has one j less
        if (N % JL && j >= N) continue;
        const float4 y = *reinterpret_cast<const float4 *>(row + P::oY + 4 * j);
        const float2 sy = make_float2(y.x, y.y), dsy = make_float2(y.z, y.w);
        const float2 yz = __fmul2_rn(sy, sz);
        const float2 pa = __fmul2_rn(wc, yz), pb = __fmul2_rn(wx, yz);
        const float2 pq = __ffma2_rn(wy, __fmul2_rn(dsy, sz), __fmul2_rn(wz, __fmul2_rn(sy, dsz)));
#pragma unroll
        for (int i = 0; i < H; ++i) {
          A[jj][i] = __ffma2_rn(pa, x[i], A[jj][i]);
          B[jj][i] = __ffma2_rn(pb, dx[i], __ffma2_rn(pq, x[i], B[jj][i]));
        }
      }
    }
    __syncwarp();
  }
  if (sub >= P::Leaves || l0 + sub >= nleaf) return;
  float *out = M + (size_t)rec.x * 2 * N3 + k;
#pragma unroll
  for (int jj = 0; jj < JL; ++jj) {
    const int j = part * JL + jj;
    if (N % JL && j >= N) continue;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const float a = (i & 1) ? A[jj][i / 2].y : A[jj][i / 2].x, v = (i & 1) ? B[jj][i / 2].y : B[jj][i / 2].x;
      out[(i * N + j) * N] = fmaf(v, inv_ebar, a);
      out[N3 + (i * N + j) * N] = a + v;
    }
  }
}

// ------------------------------------------------------------------------------------
// M2M and L2L: one CTA per (parent, kernel), all of its children together, one tensor axis
// at a time behind three barriers (six per child when a CTA took one child after the
// other).  L2L does once what the children of a parent share: two and four applications of
// the 1-D operators S2[c] along x and y instead of eight.  M2M keeps the children's sums
// apart until the end and adds them in child order (sharing their sums the same way is
// faster, 28 against 36 us on the 163,842-node sphere, but its rounding reaches the
// solution through the BF16 pairs that the weights become).  Latency bounds both on small
// levels (M2M took 11 us a level, alone), shared-memory reads on large ones.  A thread's
// rows of S2 along an axis stay in registers (from constant memory, reads that differ
// across a warp are serialised).
// ------------------------------------------------------------------------------------
// Rows of S2[0] and S2[1] (columns with kTranspose) at point `row`, from shared memory.
template <int N, bool kTranspose>
__device__ __forceinline__ void axis_rows(const float *sS, int row, float (&S)[2][N]) {
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int q = 0; q < N; ++q) S[c][q] = sS[c * N * N + (kTranspose ? q * N + row : row * N + q)];
}

template <int N>
__device__ __forceinline__ void stage_m2m_ops(float *sS) {
  for (int e = threadIdx.x; e < 2 * N * N; e += blockDim.x) {
    const int c = e / (N * N), r = (e / N) % N, q = e % N;
    sS[e] = c_m2m[N][c * kMaxOrder * kMaxOrder + r * kMaxOrder + q];
  }
}

// The children of this CTA's parent by octant.
__device__ __forceinline__ void load_children(const int32_t *__restrict__ par_child, int (&child)[8]) {
  const int4 *p = reinterpret_cast<const int4 *>(par_child) + 2 * (size_t)blockIdx.x;
  const int4 a = p[0], b = p[1];
  child[0] = a.x; child[1] = a.y; child[2] = a.z; child[3] = a.w;
  child[4] = b.x; child[5] = b.y; child[6] = b.z; child[7] = b.w;
}

template <int N>
constexpr int kAxisThreads = (N * N * N + 31) / 32 * 32;     // a thread to a weight

// Every parent of one level sums its children's translated multipoles.
template <int N>
__global__ void __launch_bounds__(kAxisThreads<N>) k_m2m(const int32_t *__restrict__ par,
                                                         const int32_t *__restrict__ par_child, float *__restrict__ M) {
  constexpr int N3 = N * N * N;
  __shared__ float s8[8][N3], t8[8][N3], sS[2 * N * N];
  const int b = par[blockIdx.x], kt = blockIdx.y;
  int child[8];
  load_children(par_child, child);
  stage_m2m_ops<N>(sS);
  after_previous();
  const int m = threadIdx.x;
  const bool act = m < N3;
  const int i = m / (N * N), j = (m / N) % N, k = m % N;
  if (act) {
    float v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = child[c] >= 0 ? M[((size_t)child[c] * 2 + kt) * N3 + m] : 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) s8[c][m] = v[c];
  }
  __syncthreads();
  float S[2][N];
  if (act) {
    axis_rows<N, false>(sS, k, S);
#pragma unroll
    for (int c = 0; c < 8; ++c) {                       // octants 4 cx + 2 cy + cz
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < N; ++q) t = fmaf(S[c & 1][q], s8[c][m - k + q], t);
      t8[c][m] = t;
    }
  }
  __syncthreads();
  if (act) {
    axis_rows<N, false>(sS, j, S);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < N; ++q) t = fmaf(S[(c >> 1) & 1][q], t8[c][m + (q - j) * N], t);
      s8[c][m] = t;
    }
  }
  __syncthreads();
  if (act) {
    axis_rows<N, false>(sS, i, S);
    float sum = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < N; ++q) t = fmaf(S[c >> 2][q], s8[c][m + (q - i) * N * N], t);
      sum += t;
    }
    M[((size_t)b * 2 + kt) * N3 + m] = sum;
  }
}

// Every box of the level below `ls` adds its parent's local expansion, re-interpolated.
template <int N>
__global__ void __launch_bounds__(kAxisThreads<N>) k_l2l(const int32_t *__restrict__ par,
                                                         const int32_t *__restrict__ par_child, float *__restrict__ L) {
  constexpr int N3 = N * N * N;
  __shared__ float s1[N3], s2[2][N3], s4[4][N3], sS[2 * N * N];
  const int b = par[blockIdx.x], kt = blockIdx.y;
  int child[8];
  load_children(par_child, child);
  stage_m2m_ops<N>(sS);
  after_previous();
  const int m = threadIdx.x;
  const bool act = m < N3;
  const int i = m / (N * N), j = (m / N) % N, k = m % N;
  float v[8];                                           // the children's own expansions
  if (act) {
    s1[m] = L[((size_t)b * 2 + kt) * N3 + m];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = child[c] >= 0 ? L[((size_t)child[c] * 2 + kt) * N3 + m] : 0.f;
  }
  __syncthreads();
  float S[2][N];
  if (act) {
    axis_rows<N, true>(sS, i, S);
#pragma unroll
    for (int c = 0; c < 2; ++c) {                       // cx
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < N; ++q) t = fmaf(S[c][q], s1[m + (q - i) * N * N], t);
      s2[c][m] = t;
    }
  }
  __syncthreads();
  if (act) {
    axis_rows<N, true>(sS, j, S);
#pragma unroll
    for (int c = 0; c < 4; ++c) {                       // (cx, cy)
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < N; ++q) t = fmaf(S[c & 1][q], s2[c >> 1][m + (q - j) * N], t);
      s4[c][m] = t;
    }
  }
  __syncthreads();
  if (act) {
    axis_rows<N, true>(sS, k, S);
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      if (child[c] < 0) continue;
      float t = 0.f;
#pragma unroll
      for (int q = 0; q < N; ++q) t = fmaf(S[c & 1][q], s4[c >> 1][m - k + q], t);
      L[((size_t)child[c] * 2 + kt) * N3 + m] = v[c] + t;
    }
  }
}

// ------------------------------------------------------------------------------------
// M2L (FP32, CUDA cores).  One CTA per (row tile of 64 target weights, (level, offset)
// group, kernel); the 64 x n^3 slice of the translation matrix stays in shared memory
// while the group's pairs stream through in chunks of 32.  Results are added with
// atomics (several offsets feed the same target box).
// ------------------------------------------------------------------------------------
template <int N>
__global__ void __launch_bounds__(256) k_m2l(const M2LGroup *__restrict__ groups, const int2 *__restrict__ pairs,
                                             const float *__restrict__ Klap, const float *__restrict__ Kyuk,
                                             const dbl4 *__restrict__ center, int yuk_min_level,
                                             const float *__restrict__ M, float *__restrict__ L) {
  constexpr int N3 = N * N * N;
  constexpr int RT = 64, PC = 32, LD = N3 + 1;
  extern __shared__ float smem[];
  float *Ks = smem;                 // [RT][LD]
  float *Ms = smem + RT * LD;       // [N3][PC]
  const M2LGroup g = groups[blockIdx.y];
  const int kt = blockIdx.z;
  if (kt == 1 && g.level < yuk_min_level) return;
  const int r0 = blockIdx.x * RT;
  const int rows = min(RT, N3 - r0);
  const size_t N6 = (size_t)N3 * N3;
  const float *K = kt == 0 ? Klap + (size_t)g.offset * N6 : Kyuk + ((size_t)g.level * kNumOffsets + g.offset) * N6;
  for (int e = threadIdx.x; e < RT * N3; e += blockDim.x) {
    int r = e / N3, c = e % N3;
    Ks[r * LD + c] = r < rows ? K[(size_t)(r0 + r) * N3 + c] : 0.0f;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int pc = 0; pc < g.count; pc += PC) {
    const int cnt = min(PC, g.count - pc);
    __syncthreads();
    for (int e = threadIdx.x; e < N3 * PC; e += blockDim.x) {
      int p = e / N3, k = e % N3;
      float v = 0.0f;
      if (p < cnt) v = M[((size_t)pairs[g.start + pc + p].y * 2 + kt) * N3 + k];
      Ms[k * PC + p] = v;
    }
    __syncthreads();
    float acc[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
    const float *k0 = Ks + lane * LD, *k1 = Ks + (lane + 32) * LD;
#pragma unroll 4
    for (int k = 0; k < N3; ++k) {
      const float a0 = k0[k], a1 = k1[k];
      const float4 mv = *reinterpret_cast<const float4 *>(Ms + k * PC + warp * 4);
      acc[0][0] = fmaf(a0, mv.x, acc[0][0]); acc[0][1] = fmaf(a0, mv.y, acc[0][1]);
      acc[0][2] = fmaf(a0, mv.z, acc[0][2]); acc[0][3] = fmaf(a0, mv.w, acc[0][3]);
      acc[1][0] = fmaf(a1, mv.x, acc[1][0]); acc[1][1] = fmaf(a1, mv.y, acc[1][1]);
      acc[1][2] = fmaf(a1, mv.z, acc[1][2]); acc[1][3] = fmaf(a1, mv.w, acc[1][3]);
    }
    const float scale = kt == 0 ? (float)(1.0 / center[pairs[g.start].x].w) : 1.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int p = warp * 4 + q;
      if (p >= cnt) continue;
      const int tb = pairs[g.start + pc + p].x;
      float *dst = L + ((size_t)tb * 2 + kt) * N3 + r0;
      if (lane < rows) atomicAdd(dst + lane, acc[0][q] * scale);
      if (lane + 32 < rows) atomicAdd(dst + lane + 32, acc[1][q] * scale);
    }
  }
}

// M2L matrices: Laplace for a unit box (scaled by 1/w when used), Yukawa per level.
__global__ void k_m2l_table(int N, int nslots, const int3 *__restrict__ offs, double kw, double invw,
                            float *__restrict__ out) {
  const int N3 = N * N * N;
  const int64_t tot = (int64_t)nslots * N3 * N3;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    int slot = (int)(e / ((int64_t)N3 * N3));
    int rem = (int)(e % ((int64_t)N3 * N3));
    int mt = rem / N3, ms = rem % N3;
    int3 o = offs[slot];
    const float *nd = c_nodes[N];
    double tx = nd[mt / (N * N)], ty = nd[(mt / N) % N], tz = nd[mt % N];
    double sx = 2.0 * o.x + nd[ms / (N * N)], sy = 2.0 * o.y + nd[(ms / N) % N], sz = 2.0 * o.z + nd[ms % N];
    double r = sqrt((tx - sx) * (tx - sx) + (ty - sy) * (ty - sy) + (tz - sz) * (tz - sz));
    double v = kInv4Pi / r;
    if (kw >= 0.0) v = exp(-kw * r) * v * invw;
    out[e] = (float)v;
  }
}

// ------------------------------------------------------------------------------------
// P2L: list-4 sources straight into a box's local weights.
// ------------------------------------------------------------------------------------
template <int N>
__global__ void __launch_bounds__(256) k_p2l(const int32_t *__restrict__ xbox, const int64_t *__restrict__ xptr,
                                             const int32_t *__restrict__ xidx, const int32_t *__restrict__ bbeg,
                                             const int32_t *__restrict__ bend, const dbl4 *__restrict__ center,
                                             const float4 *__restrict__ pos, const float4 *__restrict__ nrm,
                                             const float2 *__restrict__ xs, float inv_ebar, float kappa,
                                             float *__restrict__ L) {
  constexpr int N3 = N * N * N;
  constexpr int CH = 128;
  __shared__ float4 sp[CH], sn[CH];
  const int b = xbox[blockIdx.x];
  const dbl4 cb = center[b];
  const float w = (float)cb.w;
  float accL[(N3 + 255) / 256], accY[(N3 + 255) / 256];
  float px[(N3 + 255) / 256], py[(N3 + 255) / 256], pz[(N3 + 255) / 256];
#pragma unroll
  for (int r = 0; r < (N3 + 255) / 256; ++r) {
    accL[r] = accY[r] = 0.0f;
    int m = threadIdx.x + 256 * r;
    if (m < N3) {
      px[r] = w * c_nodes[N][m / (N * N)];
      py[r] = w * c_nodes[N][(m / N) % N];
      pz[r] = w * c_nodes[N][m % N];
    }
  }
  for (int64_t j = xptr[b]; j < xptr[b + 1]; ++j) {
    const int c = xidx[j];
    const dbl4 cc = center[c];
    const float ox = (float)(cc.x - cb.x), oy = (float)(cc.y - cb.y), oz = (float)(cc.z - cb.z);
    for (int s0 = bbeg[c]; s0 < bend[c]; s0 += CH) {
      const int cnt = min(CH, bend[c] - s0);
      __syncthreads();
      for (int t = threadIdx.x; t < cnt; t += blockDim.x) {
        float4 p = pos[s0 + t], q = nrm[s0 + t];
        float2 fh = xs[s0 + t];
        sp[t] = make_float4(p.x + ox, p.y + oy, p.z + oz, p.w * fh.y);
        sn[t] = make_float4(q.x, q.y, q.z, -p.w * fh.x);
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < (N3 + 255) / 256; ++r) {
        if (threadIdx.x + 256 * r >= N3) continue;
        float aL = accL[r], aY = accY[r];
        for (int t = 0; t < cnt; ++t) {
          const float4 y = sp[t], q = sn[t];
          const float dx = px[r] - y.x, dy = py[r] - y.y, dz = pz[r] - y.z;
          const float r2 = dx * dx + dy * dy + dz * dz;
          const float ri = rsqrtf(r2);
          const float rr = r2 * ri;
          const float G = ri, G3 = ri * ri * ri;
          const float ndt = q.x * dx + q.y * dy + q.z * dz;
          const float e = __expf(-kappa * rr);
          const float g1 = e * (1.0f + kappa * rr) * G3;
          aL += y.w * G + q.w * inv_ebar * ndt * G3;
          aY += y.w * e * G + q.w * ndt * g1;
        }
        accL[r] = aL;
        accY[r] = aY;
      }
    }
  }
  const float s = (float)kInv4Pi;
#pragma unroll
  for (int r = 0; r < (N3 + 255) / 256; ++r) {
    int m = threadIdx.x + 256 * r;
    if (m < N3) {
      L[(size_t)b * 2 * N3 + m] += s * accL[r];
      L[(size_t)b * 2 * N3 + N3 + m] += s * accY[r];
    }
  }
}

// ------------------------------------------------------------------------------------
// L2P: evaluate both local expansions and their normal derivatives at leaf targets.
// One thread per node in Morton order, whatever leaf it is in: every lane has a node (a CTA
// per leaf left 28 of 64 lanes idle on leaves of 36).  A CTA's nodes span a few leaves,
// whose weights are staged in shared memory; where they span more than kL2PLeaves leaves, a
// thread reads its leaf's weights from L2 instead.  (Staged round after round, for a few nodes
// each time, L2P took 53 us on 642 nodes in leaves of three and 45 us on 163,842 in leaves of
// ten; 12 and 27 us so.)  Each sum runs in
// ascending order of its points: the gradient of a nearly constant field is a small
// difference, and a sum in another order moves it by more than the rest of the product's
// rounding (which rules out packed pairs along z; pairs along y or of value and derivative
// need the weights twice or transposed, and shared memory bounds them: 0.65 ms on 5.03M
// nodes).  Instruction issue and the weights' reads bound it on large meshes and the
// chain of loads (block record, leaf records, weights) on small ones.
//
// With kOut the product is assembled here (Eq. 5), where the far sums are in registers:
//   y1 = alpha f - PhiL + PhiY,   y2 = alpha h - dn PhiL + dn PhiY / eps_bar
// over far and P2P sums, the near correction being in the P2P sums; y goes to y[perm[t]]
// (kOut == 2: caller order) or y[t] (kOut == 1).  That takes the combine and the scatter
// (two launches and their passes over memory) off the end of the product.
// ------------------------------------------------------------------------------------
constexpr int kL2PLeaves = 6;       // leaves staged
constexpr int kL2PResident = 4;     // blocks per SM: registers for many of a thread's loads in flight

// (phi, grad phi) of a local expansion at a node, the gradient in box half widths.
template <int N>
__device__ __forceinline__ float4 l2p_eval(const float *Lk, const float (&sx)[N], const float (&dsx)[N],
                                           const float (&sy)[N], const float (&dsy)[N], const float (&sz)[N],
                                           const float (&dsz)[N]) {
  float phi0 = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float a = 0.f, bj = 0.f, cj = 0.f;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const float *row = Lk + (i * N + j) * N;
      float u = 0.f, du = 0.f;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        float l;
        if (N % 2 == 0) {                        // two weights to an 8-byte load
          const float2 v = reinterpret_cast<const float2 *>(row)[k / 2];
          l = (k & 1) ? v.y : v.x;
        } else {
          l = row[k];
        }
        u = fmaf(l, sz[k], u);
        du = fmaf(l, dsz[k], du);
      }
      a = fmaf(u, sy[j], a);
      bj = fmaf(u, dsy[j], bj);
      cj = fmaf(du, sy[j], cj);
    }
    phi0 = fmaf(a, sx[i], phi0);
    gx = fmaf(a, dsx[i], gx);
    gy = fmaf(bj, sx[i], gy);
    gz = fmaf(cj, sx[i], gz);
  }
  return make_float4(phi0, gx, gy, gz);
}

template <int N, int kOut>
__global__ void __launch_bounds__(kL2PNodes, kL2PResident) k_l2p(int64_t n, const int2 *__restrict__ blk,
                                                   const int4 *__restrict__ leaf_rec, float inv_w0,
                                                   const float4 *__restrict__ pos, const float4 *__restrict__ nrm,
                                                   const float *__restrict__ L, float4 *__restrict__ phi,
                                                   const float2 *__restrict__ xs, const float4 *__restrict__ pnear,
                                                   const int32_t *__restrict__ perm, float alpha, float inv_ebar,
                                                   int64_t ldy, float *__restrict__ y) {
  constexpr int N3 = N * N * N;
  __shared__ __align__(16) float sL[kL2PLeaves][2 * N3];
  __shared__ int4 srec[kL2PLeaves];
  const int64_t t = blockIdx.x * (int64_t)kL2PNodes + threadIdx.x;
  const int2 lr = blk[blockIdx.x];
  const bool node = t < n;
  float4 p = make_float4(0.f, 0.f, 0.f, 0.f), q = p, pn = p;
  float2 x = make_float2(0.f, 0.f);
  int64_t o = t;
  if (node) {
    p = pos[t];
    q = nrm[t];
    if (kOut) {
      x = xs[t];
      pn = pnear[t];
      if (kOut == 2) o = perm[t];
    }
  }
  auto eval = [&](const float *w, int level) {          // this thread's node, from its leaf's weights
    const float invw = inv_width(inv_w0, level);
    float sx[N], dsx[N], sy[N], dsy[N];
    float sz[N], dsz[N];
    cheb_basis<N>(p.z * invw, sz, dsz);
    cheb_basis<N>(p.x * invw, sx, dsx);
    cheb_basis<N>(p.y * invw, sy, dsy);
    float2 out[2];
#pragma unroll 1
    for (int kt = 0; kt < 2; ++kt) {
      const float4 v = l2p_eval<N>(w + kt * N3, sx, dsx, sy, dsy, sz, dsz);
      const float2 u = make_float2(v.x, (q.x * v.y + q.y * v.z + q.z * v.w) * invw);
      if (kt == 0) out[0] = u;
      else out[1] = u;
    }
    if (kOut) {
      y[o] = alpha * x.x + (-(out[0].x + pn.x) + (out[1].x + pn.z));
      y[ldy + o] = alpha * x.y + (-(out[0].y + pn.y) + (out[1].y + pn.w) * inv_ebar);
    } else {
      phi[t] = make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
    }
  };
  if (lr.y - lr.x >= kL2PLeaves) {                      // small leaves
    if (!node) return;
    int lo = lr.x, hi = lr.y;                           // the leaf whose nodes end after t
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (leaf_rec[mid].z > t) hi = mid;
      else lo = mid + 1;
    }
    const int4 rec = leaf_rec[lo];
    eval(L + (size_t)rec.x * 2 * N3, rec.w);
    return;
  }
  const int nl = lr.y + 1 - lr.x;
  if (threadIdx.x < nl) srec[threadIdx.x] = leaf_rec[lr.x + threadIdx.x];
  __syncthreads();
#pragma unroll 4
  for (int e = threadIdx.x; e < nl * N3; e += kL2PNodes) {       // two weights at a time
    const int l = e / N3;
    reinterpret_cast<float2 *>(&sL[0][0])[e] =
        reinterpret_cast<const float2 *>(L + (size_t)srec[l].x * 2 * N3)[e - l * N3];
  }
  __syncthreads();
  if (!node) return;
  int l = 0;
  while (l + 1 < nl && t >= srec[l].z) ++l;
  eval(&sL[l][0], srec[l].w);
}

// ------------------------------------------------------------------------------------
// P2P (lists 1 and 3): point (far-rule) sums over t != p, both kernels, both outputs.
// ------------------------------------------------------------------------------------
constexpr int kP2PChunk = 768;      // sources staged in shared memory at a time (24 KB)
constexpr int kP2PPairs = kP2PChunk / 2;
constexpr int kP2PRegBlocks = kP2PResident;

// Far-rule sums of one source at one target, without the 1/(4 pi):
//   PhiL += c/r + (g/eps_bar) (n.d)/r^3
//   dn PhiL += -c (n0.d)/r^3 + (g/eps_bar) [(n0.n)/r^3 - 3 (n.d)(n0.d)/r^5]
//   PhiY += c e/r + g (n.d) e1/r^3,           e = exp(-kr), e1 = e (1 + kr)
//   dn PhiY += e1 [g (n0.n) - c (n0.d)]/r^3 - 3 g e2 (n.d)(n0.d)/r^5,  e2 = e (1 + kr + (kr)^2/3)
// with d = x_target - y_source.  g enters only through the vector g n.  With
//   P = g n.d,  Q = n0.d,  S = g n0.n,  p2 = P/r^2,  k1 = 1 + kr,  m = S - (3 p2 + c) Q
// (3 e2 = 3 e1 + e (kr)^2, and (kr)^2 p2 = k^2 P) the four sums are
//   PhiL += (p2/eps_bar + c)/r,              dn PhiL += (1/eps_bar) [m + (1 - eps_bar) c Q]/r^3,
//   PhiY += e (k1 p2 + c)/r,                 dn PhiY += e (k1 m - k^2 P Q)/r^3.
// For eps_bar < 1 the bracket of dn PhiL would cancel down to eps_bar c Q under a factor
// 1/eps_bar (eps_in 80, eps_out 2: 15 times the rounding of its terms), so there
//   u = S - (3 p2 + eps_bar c) Q,  dn PhiL += (1/eps_bar) u/r^3,  m = u + (eps_bar - 1) c Q,
// where both parts of m have one sign as the bracket's have for eps_bar >= 1: one operation
// more, in loops of their own (kLow; products of 163,842 nodes 394 us above, 393 below).
// The FP32 pipe bounds the kernel, so the count of its operations per pair is what this
// form is for: 35 (43 in the order the formulas are printed in), 38 where the pair's
// distance has to be tested, 25 and 27 without salt (k = 0: e = k1 = 1 and no exp2).
// Measured, P2P alone, at the same deal of work: 0.255 -> 0.235 ms (163,842-node sphere,
// leaves of 80), 0.582 -> 0.519 ms (leaves of 192).
//
// The sums run on packed FP32 pairs (sm_100 FFMA2 / FADD2 / FMUL2): each thread takes
// its target against two sources per instruction, lane 0 an even and lane 1 an odd
// source of the staged chunk.  The target's coordinates, normal and skip radius sit in
// both lanes for the whole loop; the staging stores every source component already
// paired with its neighbour's, so no instruction of the loop packs or broadcasts.
// Every packed operation rounds each lane as its scalar counterpart does, so the
// distance and skip test below are the scalar p2p_r2 / p2p_evaluates, bit for bit.
// 2^x on the special-function unit (PTX ex2.approx); e^-kr = 2^(-kr log2 e).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1/sqrt(x) on the special-function unit, flushing subnormal inputs (PTX rsqrt.approx.ftz):
// P2P evaluates it only for r^2 above the squared skip radius (~1e-2 A^2), far from the
// subnormal range, so the flush changes nothing there and saves the subnormal handling
// that rsqrtf carries.
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct P2PTarget {
  float2 x, y, z;        // position in the target leaf's frame, both lanes
  float2 nx, ny, nz;     // unit normal n0
  float2 rs;             // scaled skip radius
};

// Factors of the pair sums that all pairs of a problem share, in both lanes.
struct P2PConst {
  float2 inv_e;          // 1 / eps_bar
  float2 kappa;          // k
  float2 nkl2e;          // -k log2(e)
  float2 kappa2;         // k^2
  float2 wc;             // 1 - eps_bar (kLow: eps_bar - 1)
};

struct P2PSums {
  float2 sL, nD, sY, dY; // a target's four sums (see p2p_pair2)
};

// sources: a = (-x0, -x1, -y0, -y1), b = (-z0, -z1, c0, c1), c = (gnx0, gnx1, gny0, gny1),
// d = (gnz0, gnz1, w0, w1); positions in the target leaf's frame.  kTest: w = skip radius,
// and pairs inside it contribute nothing here (the near CSR carries their whole near-rule
// value; t == p is among them).  Otherwise no pair can be inside it and w = wc c.
// Sums: sL, sY as above; nD = eps_bar dn PhiL; dY.  Without salt the two kernels differ in
// eps_bar alone and the product takes their difference: the parts with and without it are
// summed apart, sL = sum p2/r, sY = sum c/r, nD = sum (S - 3 p2 Q)/r^3, dY = sum c Q/r^3.
template <bool kTest, bool kSalt, bool kLow>
__device__ __forceinline__ void p2p_pair2(const P2PTarget &t, const float4 &a, const float4 &b, const float4 &c,
                                          const float4 &d, const P2PConst &k, P2PSums &s) {
  const float2 dx = __fadd2_rn(t.x, make_float2(a.x, a.y));
  const float2 dy = __fadd2_rn(t.y, make_float2(a.z, a.w));
  const float2 dz = __fadd2_rn(t.z, make_float2(b.x, b.y));
  const float2 cc = make_float2(b.z, b.w);
  const float2 gx = make_float2(c.x, c.y), gy = make_float2(c.z, c.w), gz = make_float2(d.x, d.y);
  const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));   // p2p_r2
  float2 ri;
  if (kTest) {
    const float2 R = __fadd2_rn(t.rs, make_float2(d.z, d.w));                      // p2p_evaluates
    const float2 RR = __fmul2_rn(R, R);
    ri = make_float2(r2.x > RR.x ? rsqrt_approx(r2.x) : 0.0f, r2.y > RR.y ? rsqrt_approx(r2.y) : 0.0f);
  } else {
    ri = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
  }
  const float2 ri2 = __fmul2_rn(ri, ri);
  const float2 P = __ffma2_rn(gx, dx, __ffma2_rn(gy, dy, __fmul2_rn(gz, dz)));
  const float2 Q = __ffma2_rn(t.nx, dx, __ffma2_rn(t.ny, dy, __fmul2_rn(t.nz, dz)));
  const float2 S = __ffma2_rn(t.nx, gx, __ffma2_rn(t.ny, gy, __fmul2_rn(t.nz, gz)));
  const float2 p2 = __fmul2_rn(P, ri2);
  const float2 G3 = __fmul2_rn(ri, ri2);
  if (!kSalt) {
    s.sL = __ffma2_rn(ri, p2, s.sL);
    s.sY = __ffma2_rn(ri, cc, s.sY);
    s.nD = __ffma2_rn(G3, __ffma2_rn(__fmul2_rn(p2, Q), dup2(-3.0f), S), s.nD);
    s.dY = __ffma2_rn(G3, __fmul2_rn(cc, Q), s.dY);
    return;
  }
  const float2 h = __ffma2_rn(p2, dup2(3.0f), kLow ? __fmul2_rn(cc, dup2(1.0f / k.inv_e.x)) : cc);
  const float2 u = __ffma2_rn(make_float2(-h.x, -h.y), Q, S);
  const float2 dc = kTest ? __fmul2_rn(cc, k.wc) : make_float2(d.z, d.w);
  const float2 v = __ffma2_rn(dc, Q, u);
  const float2 m = kLow ? v : u;
  s.nD = __ffma2_rn(G3, kLow ? u : v, s.nD);
  s.sL = __ffma2_rn(ri, __ffma2_rn(k.inv_e, p2, cc), s.sL);
  const float2 rr = __fmul2_rn(r2, ri);
  const float2 arg = __fmul2_rn(rr, k.nkl2e);
  const float2 ex = make_float2(ex2_approx(arg.x), ex2_approx(arg.y));
  const float2 k1 = __ffma2_rn(rr, k.kappa, dup2(1.0f));
  const float2 ei = __fmul2_rn(ex, ri);
  s.sY = __ffma2_rn(ei, __ffma2_rn(k1, p2, cc), s.sY);
  const float2 V = __fmul2_rn(__fmul2_rn(P, Q), k.kappa2);
  s.dY = __ffma2_rn(__fmul2_rn(ei, ri2), __ffma2_rn(k1, m, make_float2(-V.x, -V.y)), s.dY);
}

// The sums of one target, (PhiL, dn PhiL, PhiY, dn PhiY) without the 1/(4 pi), from its
// accumulators.
__device__ __forceinline__ float4 p2p_sums(bool salt, float inv_e, const P2PSums &s) {
  const float a = s.sL.x + s.sL.y, b = s.nD.x + s.nD.y, c = s.sY.x + s.sY.y, d = s.dY.x + s.dY.y;
  if (salt) return make_float4(a, inv_e * b, c, d);
  return make_float4(fmaf(inv_e, a, c), fmaf(inv_e, b, -d), a + c, b - d);
}

// A thread's share of a staged chunk: pairs e, e + slices, ... of its tested part (below
// ntest), then of the others, for both of its targets.
template <bool kSalt, bool kLow>
__device__ __forceinline__ void p2p_chunk(int e, int slices, int ntest, int npairs, const float4 *sa, const float4 *sb,
                                          const float4 *sc, const float4 *sd, const P2PTarget &tg, const P2PTarget &tg2,
                                          const P2PConst &kc, P2PSums &acc, P2PSums &acc2) {
  for (; e < ntest; e += slices) {
    const float4 qa = sa[e], qb = sb[e], qc = sc[e], qd = sd[e];
    p2p_pair2<true, kSalt, kLow>(tg, qa, qb, qc, qd, kc, acc);
    p2p_pair2<true, kSalt, kLow>(tg2, qa, qb, qc, qd, kc, acc2);
  }
  for (; e < npairs; e += slices) {
    const float4 qa = sa[e], qb = sb[e], qc = sc[e], qd = sd[e];
    p2p_pair2<false, kSalt, kLow>(tg, qa, qb, qc, qd, kc, acc);
    p2p_pair2<false, kSalt, kLow>(tg2, qa, qb, qc, qd, kc, acc2);
  }
}

// A unit that covers its leaf's whole source list stores; a part of a split leaf adds.
__device__ __forceinline__ void store_or_add(float4 *p, float4 v, bool whole) {
  if (whole) *p = v;
  else asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}

// A P2P argument: the kernel's own, or (batched) the unit's problem's, read from shared
// memory where it is used so that no pointer stays live across the loops.
#define P2P_ARG(name) (kBatch ? s_req.name : name##_1)

// The body of the P2P kernels: with kBatch the work units of several problems share one
// launch, unit.req naming the problem whose arrays (reqs[unit.req], copied to shared memory
// per unit) it reads, and units of a problem whose *active flag is 0 are skipped.
template <bool kBatch>
__device__ __forceinline__ void p2p_body(const P2PUnit *__restrict__ units,
                                         const int4 *__restrict__ leaf_rec_1, const float4 *__restrict__ src_1,
                                         const int2 *__restrict__ slot_1, const float4 *__restrict__ pos_1,
                                         const float4 *__restrict__ nrm_1, const float2 *__restrict__ xs_1,
                                         float inv_ebar_1, float kappa_1, float skip_scale_1, float4 *__restrict__ phi_1,
                                         const P2PReq *__restrict__ reqs) {
  __shared__ float4 sa[kP2PPairs], sb[kP2PPairs], sc[kP2PPairs], sd[kP2PPairs];
  __shared__ float4 red[2 * kP2PThreads];
  __shared__ __align__(8) P2PReq s_req;
  // One block per work unit, the costliest first: the block scheduler deals them out as
  // blocks finish (a static deal to resident blocks left the slowest 15% behind: 0.234
  // against 0.201 ms on the 163,842-node sphere).  A unit is one leaf's targets against a
  // range of its source boxes; leaves with more pairs than the unit budget are split, and
  // their units add into the (zeroed) output.  All that a block has to know of its unit
  // before it can fetch sources is laid out at setup (unit, leaf record, source records and
  // slots: two dependent loads, no scan of the boxes).
  const int4 unit = reinterpret_cast<const int4 *>(units + blockIdx.x)[0];
  const int4 share = reinterpret_cast<const int4 *>(units + blockIdx.x)[1];    // tested, total, whole, -
  if constexpr (kBatch) {
    static_assert(sizeof(P2PReq) % 8 == 0, "copied as 8-byte words");
    if (threadIdx.x < sizeof(P2PReq) / 8)
      reinterpret_cast<uint64_t *>(&s_req)[threadIdx.x] = reinterpret_cast<const uint64_t *>(reqs + unit.w)[threadIdx.x];
    __syncthreads();
    if (s_req.active && *s_req.active == 0) return;    // uniform: the problem has stopped
  }
  P2PConst kc;
  {
    const float inv_e = P2P_ARG(inv_ebar), kap = P2P_ARG(kappa);
    kc.inv_e = dup2(inv_e);
    kc.kappa = dup2(kap);
    kc.nkl2e = dup2(-1.4426950408889634f * kap);
    kc.kappa2 = dup2(kap * kap);
    kc.wc = dup2(inv_e > 1.0f ? 1.0f / inv_e - 1.0f : 1.0f - 1.0f / inv_e);
  }
  const bool salt = kc.kappa.x > 0.0f, low = kc.inv_e.x > 1.0f;
  const int4 rec = P2P_ARG(leaf_rec)[unit.x];
  const int tb = rec.y, te = rec.z;
  // each thread takes two targets, t and t + tile, against the same sources
  const int tile = min((te - tb + 1) / 2, kP2PThreads);
  const int slices = kP2PThreads / tile;
  const int ti = threadIdx.x % tile, si = threadIdx.x / tile;
  const int nf = share.x, nfe = (nf + 1) & ~1, total = share.y;
  for (int t0 = tb; t0 < te; t0 += 2 * tile) {
    const int t = t0 + ti, t2 = t + tile;
    const bool act = si < slices && t < te;
    const bool act2 = act && t2 < te;
    P2PTarget tg, tg2;
    {
      const float4 xp = act ? P2P_ARG(pos)[t] : make_float4(0, 0, 0, 0);
      const float4 np = act ? P2P_ARG(nrm)[t] : make_float4(0, 0, 0, 0);
      tg.x = dup2(xp.x); tg.y = dup2(xp.y); tg.z = dup2(xp.z);
      tg.nx = dup2(np.x); tg.ny = dup2(np.y); tg.nz = dup2(np.z);
      tg.rs = dup2(p2p_skip_radius(P2P_ARG(skip_scale), np.w));
      // a missing second target repeats the first (its sums are not stored)
      const float4 xq = act2 ? P2P_ARG(pos)[t2] : xp;
      const float4 nq = act2 ? P2P_ARG(nrm)[t2] : np;
      tg2.x = dup2(xq.x); tg2.y = dup2(xq.y); tg2.z = dup2(xq.z);
      tg2.nx = dup2(nq.x); tg2.ny = dup2(nq.y); tg2.nz = dup2(nq.z);
      tg2.rs = dup2(p2p_skip_radius(P2P_ARG(skip_scale), nq.w));
    }
    P2PSums acc{}, acc2{};
    for (int c0 = 0; c0 < total; c0 += kP2PChunk) {
      const int cnt = min(kP2PChunk, total - c0);
      const int npairs = (cnt + 1) >> 1;
      const int ntest = min(max(nfe - c0, 0), cnt) >> 1;       // pairs of the tested part
      int first = unit.y;
      if (c0 > 0) {
        for (int last = unit.z - 1; first < last;) {           // the first entry that reaches beyond c0
          const int mid = (first + last) >> 1;
          const int2 sl = P2P_ARG(slot)[mid];
          if (sl.x + sl.y > c0) last = mid;
          else first = mid + 1;
        }
        __syncthreads();                                       // the last chunk has been read
      }
      // sixteen threads to a source box
      for (int en = first + (threadIdx.x >> 4); en < unit.z; en += kP2PThreads / 16) {
        const int2 sl = P2P_ARG(slot)[en];                     // first slot, nodes
        if (sl.x >= c0 + kP2PChunk) break;
        const float4 box = P2P_ARG(src)[en];                   // centre difference, first node
        const int hi = min(sl.x + sl.y, c0 + kP2PChunk);
        const bool tested = sl.x < nf;
        const int beg = __float_as_int(box.w) - sl.x;
        for (int j = max(sl.x, c0) + (threadIdx.x & 15); j < hi; j += 16) {
          const float4 p = P2P_ARG(pos)[beg + j], q = P2P_ARG(nrm)[beg + j];
          const float2 fh = P2P_ARG(xs)[beg + j];
          const float px = __fadd_rn(p.x, box.x), py = __fadd_rn(p.y, box.y), pz = __fadd_rn(p.z, box.z);
          const float cw = p.w * fh.y, g = -p.w * fh.x;
          const int e = j - c0, pr = e >> 1, ln = e & 1;
          float *fa = reinterpret_cast<float *>(sa + pr), *fb = reinterpret_cast<float *>(sb + pr);
          float *fc = reinterpret_cast<float *>(sc + pr), *fd = reinterpret_cast<float *>(sd + pr);
          fa[ln] = -px; fa[2 + ln] = -py;
          fb[ln] = -pz; fb[2 + ln] = cw;
          fc[ln] = g * q.x; fc[2 + ln] = g * q.y;
          fd[ln] = g * q.z;
          fd[2 + ln] = tested ? p2p_skip_radius(P2P_ARG(skip_scale), q.w) : cw * kc.wc.x;
          // the odd slot after the last source of either part: its neighbour's place, no
          // weight, and in the tested part a radius that leaves it out
          if (ln == 0 && (j + 1 == nf || j + 1 == total)) {
            fa[1] = -px; fa[3] = -py;
            fb[1] = -pz; fb[3] = 0.f;
            fc[1] = 0.f; fc[3] = 0.f;
            fd[1] = 0.f;
            fd[3] = tested ? 3.0e18f : 0.f;
          }
        }
      }
      __syncthreads();
      if (act) {
        if (!salt) p2p_chunk<false, false>(si, slices, ntest, npairs, sa, sb, sc, sd, tg, tg2, kc, acc, acc2);
        else if (!low) p2p_chunk<true, false>(si, slices, ntest, npairs, sa, sb, sc, sd, tg, tg2, kc, acc, acc2);
        else p2p_chunk<true, true>(si, slices, ntest, npairs, sa, sb, sc, sd, tg, tg2, kc, acc, acc2);
      }
    }
    red[threadIdx.x] = p2p_sums(salt, kc.inv_e.x, acc);
    red[kP2PThreads + threadIdx.x] = p2p_sums(salt, kc.inv_e.x, acc2);
    __syncthreads();                                           // the sums are there, the last chunk is free
    if (si == 0 && t < te) {
      const float s = (float)kInv4Pi;
      float4 a = red[ti];
      for (int k = 1; k < slices; ++k) {
        const float4 v = red[k * tile + ti];
        a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
      }
      store_or_add(P2P_ARG(phi) + t, make_float4(s * a.x, s * a.y, s * a.z, s * a.w), share.z != 0);
      if (t2 < te) {
        float4 c = red[kP2PThreads + ti];
        for (int k = 1; k < slices; ++k) {
          const float4 v = red[kP2PThreads + k * tile + ti];
          c.x += v.x; c.y += v.y; c.z += v.z; c.w += v.w;
        }
        store_or_add(P2P_ARG(phi) + t2, make_float4(s * c.x, s * c.y, s * c.z, s * c.w), share.z != 0);
      }
    }
    if (total == 0) __syncthreads();                           // no staging barrier before the sums' next use
  }
}

__global__ void __launch_bounds__(kP2PThreads, kP2PRegBlocks) k_p2p(const P2PUnit *__restrict__ units,
                                                                    const int4 *__restrict__ leaf_rec,
                                                                    const float4 *__restrict__ src,
                                                                    const int2 *__restrict__ slot,
                                                                    const float4 *__restrict__ pos,
                                                                    const float4 *__restrict__ nrm,
                                                                    const float2 *__restrict__ xs, float inv_ebar,
                                                                    float kappa, float skip_scale,
                                                                    float4 *__restrict__ phi) {
  p2p_body<false>(units, leaf_rec, src, slot, pos, nrm, xs, inv_ebar, kappa, skip_scale, phi, nullptr);
}

// P2P of several problems in one launch: the units of all of them, cost-ordered together.
__global__ void __launch_bounds__(kP2PThreads, kP2PRegBlocks) k_p2p_batch(const P2PUnit *__restrict__ units,
                                                                          const P2PReq *__restrict__ reqs) {
  p2p_body<true>(units, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, 0.f, 0.f, 0.f, nullptr, reqs);
}

// ------------------------------------------------------------------------------------
// Combine (Eq. 5): y1 = alpha f - PhiL + PhiY + sum_near (dB f - dA h)
//                  y2 = alpha h - dn PhiL + dn PhiY / eps_bar + sum_near (dD f - dC h)
// Eight lanes per row walk the near-field CSR.
// ------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_combine(int64_t n, int parts, float alpha, float inv_ebar,
                                                 const float2 *__restrict__ xs, const float4 *__restrict__ pfar,
                                                 const float4 *__restrict__ pnear, const int64_t *__restrict__ nptr,
                                                 const int32_t *__restrict__ ncol, const float4 *__restrict__ ncoef,
                                                 float *__restrict__ ys) {
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t p = gid >> 3;
  const int sub = threadIdx.x & 7;
  const bool row = p < n;           // every lane stays for the shuffles below
  float a1 = 0.f, a2 = 0.f;
  if (row && (parts & AFMPB_PART_NEAR)) {
    for (int64_t j = nptr[p] + sub; j < nptr[p + 1]; j += 8) {
      const float4 c = ncoef[j];
      const float2 x = xs[ncol[j]];
      a1 = fmaf(c.y, x.x, fmaf(-c.x, x.y, a1));
      a2 = fmaf(c.w, x.x, fmaf(-c.z, x.y, a2));
    }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    a1 += __shfl_xor_sync(0xffffffffu, a1, o, 8);
    a2 += __shfl_xor_sync(0xffffffffu, a2, o, 8);
  }
  if (row && sub == 0) {
    const float2 x = xs[p];
    if (parts & AFMPB_PART_DIAG) {
      a1 += alpha * x.x;
      a2 += alpha * x.y;
    }
    if (parts & AFMPB_PART_FAR) {
      const float4 u = pfar[p], v = pnear[p];
      a1 += -(u.x + v.x) + (u.z + v.z);
      a2 += -(u.y + v.y) + (u.w + v.w) * inv_ebar;
    }
    ys[p] = a1;
    ys[n + p] = a2;
  }
}

// ------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------
namespace {

double cheb_s(int n, int m, double x) {   // s_m(x) in double (host tables)
  double xm = std::cos((2.0 * m + 1.0) * kPi / (2.0 * n));
  double v = 1.0 / n;
  for (int k = 1; k < n; ++k) v += 2.0 / n * std::cos(k * std::acos(xm)) * std::cos(k * std::acos(std::max(-1.0, std::min(1.0, x))));
  return v;
}

// Chebyshev tables of every order, uploaded once per device (host double -> float).
Err init_cheb_tables() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  AFMPB_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return make_err(AFMPB_EINVAL, "device index out of range");
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return Err{};
  static float cheb[kMaxOrder + 1][kMaxOrder * kMaxOrder], nodes[kMaxOrder + 1][kMaxOrder],
      m2m[kMaxOrder + 1][2 * kMaxOrder * kMaxOrder];
  for (int n = 2; n <= kMaxOrder; ++n) {
    for (int m = 0; m < n; ++m) {
      nodes[n][m] = (float)std::cos((2.0 * m + 1.0) * kPi / (2.0 * n));
      for (int k = 0; k < n; ++k)
        cheb[n][m * kMaxOrder + k] = (float)((k == 0 ? 1.0 : 2.0) / n * std::cos(k * (2.0 * m + 1.0) * kPi / (2.0 * n)));
    }
    for (int c = 0; c < 2; ++c)
      for (int m = 0; m < n; ++m)
        for (int mp = 0; mp < n; ++mp) {
          const double xmp = std::cos((2.0 * mp + 1.0) * kPi / (2.0 * n));
          const double xi = (c == 0 ? -0.5 : 0.5) + 0.5 * xmp;
          m2m[n][c * kMaxOrder * kMaxOrder + m * kMaxOrder + mp] = (float)cheb_s(n, m, xi);
        }
  }
  AFMPB_CUDA(cudaMemcpyToSymbol(c_cheb, cheb, sizeof(cheb)));
  AFMPB_CUDA(cudaMemcpyToSymbol(c_nodes, nodes, sizeof(nodes)));
  AFMPB_CUDA(cudaMemcpyToSymbol(c_m2m, m2m, sizeof(m2m)));
  done[dev] = true;
  return Err{};
}

// L and the compressed locals, beside the upward pass.  A kernel, since a memset node has no
// priority and its blocks wait behind those of P2P (products of 163,842 nodes 416 us so, 400
// with the kernel); half a block per SM, which leaves room to the chain (on 152 SMs 608 in
// place of 76: a protein surface of 191,944 nodes 570 against 561 us; 24: 570).
__global__ void __launch_bounds__(256) k_zero(int64_t na, float2 *__restrict__ a, int64_t nb, float2 *__restrict__ b) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < na + nb; i += (int64_t)gridDim.x * blockDim.x)
    (i < na ? a[i] : b[i - na]) = make_float2(0.f, 0.f);
}

template <int N>
Err launch_far(afmpb_t *h, cudaStream_t s, StageTimer *tm, int parts, const FarOut *out) {
  constexpr int N3 = N * N * N;
  const auto &T = h->shape;
  const float inv_ebar = (float)(1.0 / h->ebar);
  const float inv_w0 = (float)(1.0 / T.w0);
  const bool plane_wave = h->opt.m2l_method == AFMPB_M2L_PLANE_WAVE;
  const bool compressed = !h->m2l_groups.empty() && h->m2l_rank > 0 && !plane_wave;
  // P2L adds into L, which the compressed M2L does not touch (it writes Lc; the expansion
  // adds Lc into L afterwards): in a whole product it runs on a branch of its own from the
  // zeroed L to just before the expansion, beside the upward pass and the M2L.
  const bool p2l_beside = compressed && parts == kFarAll && !tm && h->side2 && h->n_xbox > 0;
  auto launch_p2l = [&](cudaStream_t st) -> Err {
    k_p2l<N><<<(unsigned)h->n_xbox, 256, 0, st>>>(h->d_xbox, h->d_x_ptr, h->d_x_idx, h->d_box_begin, h->d_box_end,
                                                  h->d_box_center, h->d_pos, h->d_nrm, h->d_xs, inv_ebar,
                                                  (float)h->kappa, h->d_L);
    return check_launch("k_p2l");
  };
  if (parts & kFarUp) {
  // (in the chain the two memsets cost a product of 2,562 nodes 6 us of 51)
  const bool beside = !tm && h->side2;
  cudaStream_t z = beside ? h->side2 : s;
  if (beside) {
    AFMPB_CUDA(cudaEventRecord(h->ev_fork2, s));
    AFMPB_CUDA(cudaStreamWaitEvent(z, h->ev_fork2, 0));
  }
  int dev = 0, sms = 0;
  AFMPB_CUDA(cudaGetDevice(&dev));
  AFMPB_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  {
    const int64_t nl = (int64_t)T.nbox * N3, nc = compressed ? (int64_t)T.nbox * h->m2l_rank : 0;
    k_zero<<<(unsigned)std::min(div_up(nl + nc, 4 * 256), std::max(1, sms / 2)), 256, 0, z>>>(
        nl, reinterpret_cast<float2 *>(h->d_L), nc, reinterpret_cast<float2 *>(h->d_Lc));
    AFMPB_TRY(check_launch("k_zero"));
  }
  if (beside) AFMPB_CUDA(cudaEventRecord(h->ev_zero, z));
  if (p2l_beside) {
    AFMPB_TRY(launch_p2l(z));
    AFMPB_CUDA(cudaEventRecord(h->ev_join2, z));
  }
  const bool wide = kP2MHasWide<N> && T.nleaf <= kP2MWideWarps * P2MShape<N, false>::Leaves * sms;
  AFMPB_TRY(launch_next(beside, "k_p2m", wide ? k_p2m<N, kP2MHasWide<N>> : k_p2m<N, false>,
                        div_up(T.nleaf, kP2MWarps * (wide ? 1 : P2MShape<N, false>::Leaves)), 32 * kP2MWarps, 0, s, T.nleaf,
                        h->d_leaf_rec, inv_w0, h->d_pos, h->d_nrm, h->d_xs, inv_ebar, h->d_M));
  if (tm) tm->mark("p2m", 1);
  for (int level = T.nlevel - 2; level >= 2; --level) {
    const int p0 = T.par_start[level], np = T.par_start[level + 1] - p0;
    if (np == 0) continue;
    AFMPB_TRY(launch_next(true, "k_m2m", k_m2m<N>, dim3(np, 2), kAxisThreads<N>, 0, s, h->d_par + p0,
                          h->d_par_child + 8 * (size_t)p0, h->d_M));
  }
  if (tm) tm->mark("m2m", std::max(0, T.nlevel - 3));
  if (beside) AFMPB_CUDA(cudaStreamWaitEvent(s, h->ev_zero, 0));
  }
  if (compressed && p2l_beside) {
    AFMPB_TRY(enqueue_m2l_svd(h, s, tm, kFarUp | kFarM2L));
    AFMPB_CUDA(cudaStreamWaitEvent(s, h->ev_join2, 0));
    AFMPB_TRY(enqueue_m2l_svd(h, s, tm, kFarDown));
  } else if (compressed) {
    AFMPB_TRY(enqueue_m2l_svd(h, s, tm, parts));  // marks compress, m2l, expand itself
  } else if (!h->m2l_groups.empty() && (parts & kFarM2L)) {
    if (out && out->before_m2l) AFMPB_CUDA(cudaStreamWaitEvent(s, out->before_m2l, 0));
    if (plane_wave) {
      AFMPB_TRY(enqueue_m2l_pw(h, s));
    } else if (h->opt.precision == 1) {
      AFMPB_TRY(enqueue_m2l_tc(h, s));
    } else {
      constexpr int RT = 64, PC = 32;
      const size_t smem = sizeof(float) * (RT * (N3 + 1) + N3 * PC);
      dim3 grid((N3 + RT - 1) / RT, (unsigned)h->m2l_groups.size(), 2);
      k_m2l<N><<<grid, 256, smem, s>>>(h->d_m2l_groups, h->d_m2l_pairs, h->d_K_lap, h->d_K_yuk, h->d_box_center,
                                       h->m2l_yuk_levels, h->d_M, h->d_L);
      AFMPB_TRY(check_launch("k_m2l"));
    }
  }
  if (tm && !compressed) tm->mark("m2l", h->m2l_groups.empty() ? 0 : 1);
  if (!(parts & kFarDown)) return Err{};
  bool chained = compressed ? h->m2l_nchunks > 0 : !h->m2l_groups.empty() && (parts & kFarM2L) && !plane_wave;
  if (h->n_xbox > 0 && !p2l_beside) {
    AFMPB_TRY(launch_p2l(s));
    chained = true;
  }
  if (tm) tm->mark("p2l", h->n_xbox > 0 ? 1 : 0);
  for (int level = 2; level + 1 < T.nlevel; ++level) {
    const int p0 = T.par_start[level], np = T.par_start[level + 1] - p0;
    if (np == 0) continue;
    AFMPB_TRY(launch_next(chained, "k_l2l", k_l2l<N>, dim3(np, 2), kAxisThreads<N>, 0, s, h->d_par + p0,
                          h->d_par_child + 8 * (size_t)p0, h->d_L));
    chained = true;
  }
  if (tm) tm->mark("l2l", std::max(0, T.nlevel - 3));
  const int nblk = div_up(h->n, kL2PNodes);
  const float alpha = out && out->diag ? (float)h->alpha : 0.f;
  if (out) {
    if (out->join) AFMPB_CUDA(cudaStreamWaitEvent(s, out->join, 0));
    if (out->fold) AFMPB_TRY(enqueue_near_fold(h, s));
  }
  if (!out)
    k_l2p<N, 0><<<nblk, kL2PNodes, 0, s>>>(h->n, h->d_l2p_blk, h->d_leaf_rec, inv_w0, h->d_pos, h->d_nrm, h->d_L,
                                           h->d_phi_far, nullptr, nullptr, nullptr, 0.f, 0.f, 0, nullptr);
  else if (out->y)
    k_l2p<N, 2><<<nblk, kL2PNodes, 0, s>>>(h->n, h->d_l2p_blk, h->d_leaf_rec, inv_w0, h->d_pos, h->d_nrm, h->d_L,
                                           nullptr, h->d_xs, h->d_phi_near, h->d_perm, alpha, inv_ebar, h->n, out->y);
  else
    k_l2p<N, 1><<<nblk, kL2PNodes, 0, s>>>(h->n, h->d_l2p_blk, h->d_leaf_rec, inv_w0, h->d_pos, h->d_nrm, h->d_L,
                                           nullptr, h->d_xs, h->d_phi_near, nullptr, alpha, inv_ebar, h->n, h->d_ys);
  AFMPB_TRY(check_launch("k_l2p"));
  if (tm) tm->mark("l2p", 1);
  return Err{};
}

template <int N>
Err set_m2l_smem() {
  constexpr int N3 = N * N * N;
  const size_t smem = sizeof(float) * (64 * (N3 + 1) + N3 * 32);
  AFMPB_TRY(raise_smem_limit((const void *)k_m2l<N>, (int)smem));
  return Err{};
}

}  // namespace

Err enqueue_far(afmpb_t *h, cudaStream_t s, StageTimer *tm, int parts, const FarOut *out) {
  switch (h->order) {
    case 2: return launch_far<2>(h, s, tm, parts, out);
    case 3: return launch_far<3>(h, s, tm, parts, out);
    case 4: return launch_far<4>(h, s, tm, parts, out);
    case 5: return launch_far<5>(h, s, tm, parts, out);
    case 6: return launch_far<6>(h, s, tm, parts, out);
    case 7: return launch_far<7>(h, s, tm, parts, out);
    case 8: return launch_far<8>(h, s, tm, parts, out);
    default: return make_err(AFMPB_EINVAL, "fmm_order must be in [2, 8]");
  }
}

const void *far_out_kernel(int order) {
  switch (order) {
    case 2: return (const void *)k_l2p<2, 2>;
    case 3: return (const void *)k_l2p<3, 2>;
    case 4: return (const void *)k_l2p<4, 2>;
    case 5: return (const void *)k_l2p<5, 2>;
    case 6: return (const void *)k_l2p<6, 2>;
    case 7: return (const void *)k_l2p<7, 2>;
    default: return (const void *)k_l2p<8, 2>;
  }
}

Err enqueue_p2p(afmpb_t *h, cudaStream_t s) {
  // Beside the far-field chain the graph's node priorities let the chain's blocks in first
  // as P2P blocks finish.  Against a static deal to six resident blocks per SM, products of
  // 163,842 nodes 0.429 / 0.426 ms, 191,944 0.572 / 0.592, 655,362 1.306 / 1.399.
  AFMPB_CUDA(cudaMemsetAsync(h->d_phi_near, 0, sizeof(float4) * h->n, s));   // split leaves add into it
  if (h->p2p_nunits == 0) return Err{};
  k_p2p<<<h->p2p_nunits, kP2PThreads, 0, s>>>(h->d_p2p_units, h->d_leaf_rec, h->d_p2p_src, h->d_p2p_slot, h->d_pos,
                                     h->d_nrm, h->d_xs, (float)(1.0 / h->ebar), (float)h->kappa_p2p,
                                     (float)(kP2PSkip * h->opt.near_c), h->d_phi_near);
  return check_launch("k_p2p");
}

P2PReq p2p_req_of(const afmpb_t *h, const int *active) {
  P2PReq q{};
  q.leaf_rec = h->d_leaf_rec;
  q.src = h->d_p2p_src;
  q.slot = h->d_p2p_slot;
  q.pos = h->d_pos;
  q.nrm = h->d_nrm;
  q.xs = h->d_xs;
  q.phi = h->d_phi_near;
  q.active = active;
  q.inv_ebar = (float)(1.0 / h->ebar);
  q.kappa = (float)h->kappa_p2p;
  q.skip_scale = (float)(kP2PSkip * h->opt.near_c);
  return q;
}

Err enqueue_p2p_batch(const P2PReq *d_reqs, const P2PUnit *d_units, int nunits, cudaStream_t s) {
  if (nunits == 0) return Err{};
  k_p2p_batch<<<nunits, kP2PThreads, 0, s>>>(d_units, d_reqs);
  return check_launch("k_p2p_batch");
}

// The near-field correction of Eq. 5 folded into the P2P sums, on the P2P branch right
// after P2P, so that it overlaps the rest of the far-field chain instead of following it:
//   PhiL <- PhiL - sum_near (dB f - dA h),   dn PhiL <- dn PhiL - sum_near (dD f - dC h)
// (the assembly subtracts PhiL and dn PhiL, so the correction enters with its own sign).
// Eight lanes per row walk the near-field CSR, as in k_combine.
__global__ void __launch_bounds__(256) k_near_fold(int64_t n, const float2 *__restrict__ xs,
                                                   const int64_t *__restrict__ nptr, const int32_t *__restrict__ ncol,
                                                   const float4 *__restrict__ ncoef, float4 *__restrict__ pnear) {
  const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t p = gid >> 3;
  const int sub = threadIdx.x & 7;
  const bool row = p < n;           // every lane stays for the shuffles below
  float a1 = 0.f, a2 = 0.f;
  if (row) {
    for (int64_t j = nptr[p] + sub; j < nptr[p + 1]; j += 8) {
      const float4 c = ncoef[j];
      const float2 x = xs[ncol[j]];
      a1 = fmaf(c.y, x.x, fmaf(-c.x, x.y, a1));
      a2 = fmaf(c.w, x.x, fmaf(-c.z, x.y, a2));
    }
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    a1 += __shfl_xor_sync(0xffffffffu, a1, o, 8);
    a2 += __shfl_xor_sync(0xffffffffu, a2, o, 8);
  }
  if (row && sub == 0) {
    float4 v = pnear[p];
    v.x -= a1;
    v.y -= a2;
    pnear[p] = v;
  }
}

Err enqueue_near_fold(afmpb_t *h, cudaStream_t s) {
  if (h->n == 0) return Err{};
  k_near_fold<<<div_up(h->n * 8, 256), 256, 0, s>>>(h->n, h->d_xs, h->d_near_ptr, h->d_near_col, h->d_near_coef,
                                                     h->d_phi_near);
  return check_launch("k_near_fold");
}

Err enqueue_combine(afmpb_t *h, cudaStream_t s, int parts) {
  k_combine<<<div_up(h->n * 8, 256), 256, 0, s>>>(h->n, parts, (float)h->alpha, (float)(1.0 / h->ebar), h->d_xs,
                                                   h->d_phi_far, h->d_phi_near, h->d_near_ptr, h->d_near_col,
                                                   h->d_near_coef, h->d_ys);
  return check_launch("k_combine");
}

Err build_fmm(afmpb_t *h) {
  const int n = h->order;
  const int N3 = n * n * n;
  cudaStream_t s = h->stream;
  auto &A = h->arena;
  const auto &T = h->shape;
  AFMPB_TRY(init_cheb_tables());
  // offset slots: [-3,3]^3 minus [-1,1]^3
  std::vector<int> code_to_slot(343, -1);
  std::vector<int3> offs;
  for (int ox = -3; ox <= 3; ++ox)
    for (int oy = -3; oy <= 3; ++oy)
      for (int oz = -3; oz <= 3; ++oz) {
        if (std::abs(ox) <= 1 && std::abs(oy) <= 1 && std::abs(oz) <= 1) continue;
        code_to_slot[(ox + 3) * 49 + (oy + 3) * 7 + (oz + 3)] = (int)offs.size();
        offs.push_back(make_int3(ox, oy, oz));
      }
  int3 *d_offs = nullptr;
  AFMPB_TRY(A.alloc(&d_offs, offs.size(), "m2l offsets"));
  AFMPB_CUDA(cudaMemcpyAsync(d_offs, offs.data(), sizeof(int3) * offs.size(), cudaMemcpyHostToDevice, s));
  for (auto &g : h->m2l_groups) g.offset = code_to_slot[g.offset];
  if (!h->m2l_groups.empty()) {
    AFMPB_TRY(A.alloc(&h->d_m2l_groups, h->m2l_groups.size(), "m2l groups"));
    AFMPB_CUDA(cudaMemcpyAsync(h->d_m2l_groups, h->m2l_groups.data(), sizeof(M2LGroup) * h->m2l_groups.size(),
                               cudaMemcpyHostToDevice, s));
  }
  // Yukawa M2L is skipped on coarse levels where the screened kernel across the one-box
  // gap of a list-2 pair (distance >= 2 w) is below e^-40 of its unscreened value.
  int maxlev = 0;
  for (auto &g : h->m2l_groups) maxlev = std::max(maxlev, g.level + 1);
  h->m2l_yuk_levels = 0;
  while (h->m2l_yuk_levels < maxlev && h->kappa * 2.0 * std::ldexp(T.w0, -h->m2l_yuk_levels) > 40.0)
    ++h->m2l_yuk_levels;
  if (h->laplace_only) h->m2l_yuk_levels = maxlev;
  bool compressed = false;
  AFMPB_TRY(build_m2l_svd(h, &compressed));
  if (compressed) {
    A.release(d_offs);
    AFMPB_TRY(A.alloc(&h->d_M, (size_t)T.nbox * 2 * N3, "M"));
    AFMPB_TRY(A.alloc(&h->d_L, (size_t)T.nbox * 2 * N3, "L"));
    AFMPB_CUDA(cudaMemsetAsync(h->d_M, 0, sizeof(float) * (size_t)T.nbox * 2 * N3, s));
    if (h->opt.precision == 1) AFMPB_TRY(build_m2l_tc(h));
    if (h->opt.m2l_method == AFMPB_M2L_PLANE_WAVE) AFMPB_TRY(build_m2l_pw(h));
    return Err{};
  }
  const size_t N6 = (size_t)N3 * N3;
  AFMPB_TRY(A.alloc(&h->d_K_lap, kNumOffsets * N6, "K laplace"));
  AFMPB_TRY(A.alloc(&h->d_K_yuk, h->laplace_only ? 1 : (size_t)std::max(maxlev, 1) * kNumOffsets * N6, "K yukawa"));
  k_m2l_table<<<1024, 256, 0, s>>>(n, kNumOffsets, d_offs, -1.0, 1.0, h->d_K_lap);
  AFMPB_TRY(check_launch("k_m2l_table lap"));
  for (int l = std::max(2, h->m2l_yuk_levels); l < maxlev; ++l) {
    double w = std::ldexp(T.w0, -l);
    k_m2l_table<<<1024, 256, 0, s>>>(n, kNumOffsets, d_offs, h->kappa * w, 1.0 / w,
                                     h->d_K_yuk + (size_t)l * kNumOffsets * N6);
    AFMPB_TRY(check_launch("k_m2l_table yuk"));
  }
  AFMPB_CUDA(cudaStreamSynchronize(s));
  A.release(d_offs);
  AFMPB_TRY(A.alloc(&h->d_M, (size_t)T.nbox * 2 * N3, "M"));
  AFMPB_TRY(A.alloc(&h->d_L, (size_t)T.nbox * 2 * N3, "L"));
  AFMPB_CUDA(cudaMemsetAsync(h->d_M, 0, sizeof(float) * (size_t)T.nbox * 2 * N3, s));
  switch (n) {
    case 2: AFMPB_TRY(set_m2l_smem<2>()); break;
    case 3: AFMPB_TRY(set_m2l_smem<3>()); break;
    case 4: AFMPB_TRY(set_m2l_smem<4>()); break;
    case 5: AFMPB_TRY(set_m2l_smem<5>()); break;
    case 6: AFMPB_TRY(set_m2l_smem<6>()); break;
    case 7: AFMPB_TRY(set_m2l_smem<7>()); break;
    case 8: AFMPB_TRY(set_m2l_smem<8>()); break;
    default: return make_err(AFMPB_EINVAL, "fmm_order must be in [2, 8]");
  }
  if (h->opt.precision == 1) AFMPB_TRY(build_m2l_tc(h));
  if (h->opt.m2l_method == AFMPB_M2L_PLANE_WAVE) AFMPB_TRY(build_m2l_pw(h));
  return Err{};
}

}  // namespace afmpb
