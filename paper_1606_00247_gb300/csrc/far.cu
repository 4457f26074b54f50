// far.cu -- the far field (Sec. 2 steps 1-2 and 4-5; the M2L is m2l32.cu and
// m2l_tc.cu): P2M, M2M, L2L and L2P on per-level scaled, trace-free expansions,
// in FP64 (FP64 plans) or FP32 (mixed precision).
//
// With s the side of a cell, the stored coefficients are
//   Qt_n = Qhat_n / s^|n|      Lt_m = L_m s^|m|
// (Qhat_n = Q_n/n!, Q_n the moments of Sec. 2.2, L_m = d^m u), kept in the trace-free form of
// common.cuh (nq = (p+1)^2 - 1 moments, nl = p^2 local coefficients: 80 and 64
// instead of 165 at p = 8).  All of them are O(1) whatever the mesh scale, so
// FP32 neither overflows nor underflows, and the octree translations become
// level independent.  With F[n -> r] the folding weights of common.cuh:
//   P2M: Qt_r = sum_j sum_c G_j[r, c] M_c(j),
//        G_j[r, c] = sum_{n -> r} F Ghat_j[n - e_c] / s^|n|               (plan time, FP64)
//   M2M: Qt^P_r = sum_k [sum_{n -> r} F s_{n-k}(+-1/4)] 2^-|k| Qt^C_k      (child centre - parent centre = +-s_P/4)
//   M2L: Lt^T_m = (-1)^|m| / (4 pi s_T) sum_n b_{n+m}(v) (s_S/s_T)^|n| Qt^S_n,  v = (c_T - c_S)/s_T
//   L2L: Lt^C_m = sum_r [sum_{k -> r, k >= m} F s_{k-m}(+-1/2) 2^-|k|] Lt^P_r  (= +-s_C/2)
//   L2P: u(c + z) = sum_m h_m(z/s) Lt_m,  h_m = sum_{n -> m} F s_n           (plan time, FP64)
// (s_j(d) = d^j/j!; b_k(x) = (-1)^|k| d^k (1/|x|), so that 1/|x - y| = sum_k
// b_k(x) y^k / k!).  All arrays keep the state index innermost: X[item][coefficient][state].
#include <algorithm>
#include <array>
#include <cmath>
#include <type_traits>

#include "common.cuh"

namespace demag {

static inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

namespace {

// P2M operator of every support node, [moment q][component] (rows of `gs`
// values): the exact-moment operator Ghat folded onto the trace-free moments
template <class T>
__global__ void k_p2m_op(const int32_t* __restrict__ leaves, const int32_t* __restrict__ level,
                         const int64_t* __restrict__ sup_off, const double* __restrict__ Ghat, double side, int nc1,
                         int nq, int gs, T* G) {
  const int32_t c = leaves[blockIdx.x];
  const double inv_s = 1.0 / ldexp(side, -level[c]);
  const int64_t so = sup_off[c], ne = sup_off[c + 1] - so;
  for (int64_t it = threadIdx.x; it < ne * gs; it += blockDim.x) {
    const int64_t e = so + it / gs;
    const int q = (int)(it % gs), r = q / 3, comp = q - 3 * r;
    double v = 0.0;
    if (r < nq) {
      int ra, rb, rc;
      h_decode(r + 1, ra, rb, rc);
      const double* gh = Ghat + e * nc1;
      v = h_fold(ra, rb, rc, [&](int na, int nb, int nz) {
        if (comp == 0) return na ? gh[mi_index(na - 1, nb, nz)] : 0.0;
        if (comp == 1) return nb ? gh[mi_index(na, nb - 1, nz)] : 0.0;
        return nz ? gh[mi_index(na, nb, nz - 1)] : 0.0;
      });
      for (int t = ra + rb + rc; t > 0; t--) v *= inv_s;
    }
    G[e * gs + q] = (T)v;
  }
}

// L2P polynomials h_m(z/s) of every node at its leaf, rows of nl values: block per
// NODE_H nodes, whose scaled monomials z^e/e! are formed once
constexpr int NODE_H = 16;
template <class T>
__global__ void __launch_bounds__(256) k_node_h(int64_t nn, const int32_t* __restrict__ node_leaf,
                                                const int32_t* __restrict__ level, const double* __restrict__ nodes_s,
                                                const double* __restrict__ centre, double side, int p, int nl, T* h) {
  __shared__ double s[NODE_H][3][MAX_P];  // degrees below p
  const int64_t i0 = blockIdx.x * (int64_t)NODE_H;
  const int nb = (int)min((int64_t)NODE_H, nn - i0);
  if (threadIdx.x < 3 * nb) {
    const int k = threadIdx.x / 3, x = threadIdx.x - 3 * k;
    const int64_t i = i0 + k;
    const int32_t c = node_leaf[i];
    const double z = (nodes_s[3 * i + x] - centre[3 * c + x]) * (1.0 / ldexp(side, -level[c]));
    double v = 1.0;
    for (int e = 0; e < p; e++) {
      s[k][x][e] = v;
      v = v * z / (e + 1);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < nb * nl; q += blockDim.x) {
    const int k = q / nl, m = q - k * nl;
    int a, b, g;
    h_decode(m, a, b, g);
    h[i0 * nl + q] =
        (T)h_fold(a, b, g, [&](int na, int nb_, int nz) { return s[k][0][na] * s[k][1][nb_] * s[k][2][nz]; });
  }
}

// P2M: one block per (source leaf, NN moments, 128 SPT states), 128 threads,
// thread = SPT states (bl, bl + 128).  Support nodes come in chunks of P2M_NE,
// double-buffered in shared memory by asynchronous copies (cp.async), the next
// chunk in flight while the current one is applied: per node the operator
// values of the block's NN moments (3 NN, in the order of use) and M of the
// states.  One node costs 3 NN / 4 broadcast 16-byte reads for 3 NN SPT FMAs
// (two states per thread halve the shared-memory reads per FMA).  NN = 80 holds
// all moments of p <= 8 in registers, so M is read once per leaf.
constexpr int P2M_NE = 8, P2M_B = 128;
template <int SPT, int NN>
constexpr size_t p2m_smem() {  // two chunk buffers
  return sizeof(float) * 2 * P2M_NE * (NN * 3 + 3 * SPT * P2M_B);
}

__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 4 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}

template <int SPT, int NN>
__global__ void __launch_bounds__(P2M_B) k_p2m32(const int32_t* __restrict__ leaves,
                                                 const int64_t* __restrict__ sup_off,
                                                 const int32_t* __restrict__ sup_node, const float* __restrict__ G,
                                                 int gs, const float* __restrict__ Ms, int nq, int B, float* Q) {
  constexpr int NS = SPT * P2M_B, NN3 = 3 * NN;  // states per block, operator values per node
  static_assert(NN % 4 == 0, "operator rows are copied and read 16 bytes at a time");
  extern __shared__ __align__(16) float p2m_smem_[];
  float(*sG)[P2M_NE][NN3] = (float(*)[P2M_NE][NN3])p2m_smem_;                              // [2][node][(q, c)]
  float(*sM)[P2M_NE][3][NS] = (float(*)[P2M_NE][3][NS])(p2m_smem_ + 2 * P2M_NE * NN3);     // [2][node][c][state]
  const int32_t c = leaves[blockIdx.x];
  const int n0 = blockIdx.y * NN;
  const int tid = threadIdx.x, bb = blockIdx.z * NS;
  const int64_t so = sup_off[c], eo = sup_off[c + 1];
  auto stage = [&](int64_t e0, int buf) {  // one chunk of support nodes into buffer buf
    const int ne = (int)min((int64_t)P2M_NE, eo - e0);
    for (int q = tid; q < P2M_NE * NN3 / 4; q += P2M_B) {
      const int r = q / (NN3 / 4), j = 4 * (q - r * (NN3 / 4));
      const bool ok = r < ne && 3 * n0 + j < gs;
      cp_async16(&sG[buf][r][j], ok ? G + (e0 + r) * gs + 3 * n0 + j : G, ok);
    }
    for (int r = 0; r < P2M_NE; r++) {
      const int64_t node = r < ne ? sup_node[e0 + r] : 0;
#pragma unroll
      for (int s2 = 0; s2 < SPT; s2++) {
        const int b = bb + s2 * P2M_B + tid;
        const bool ok = r < ne && b < B;
        const float* mp = Ms + (ok ? node * 3 * B + b : 0);
#pragma unroll
        for (int cc = 0; cc < 3; cc++) cp_async4(&sM[buf][r][cc][s2 * P2M_B + tid], ok ? mp + (int64_t)cc * B : Ms, ok);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[SPT][NN];
#pragma unroll
  for (int s2 = 0; s2 < SPT; s2++)
#pragma unroll
    for (int j = 0; j < NN; j++) acc[s2][j] = 0.f;
  if (so < eo) stage(so, 0);
  int buf = 0;
  for (int64_t e0 = so; e0 < eo; e0 += P2M_NE, buf ^= 1) {
    const int ne = (int)min((int64_t)P2M_NE, eo - e0);
    if (e0 + P2M_NE < eo) {
      stage(e0 + P2M_NE, buf ^ 1);  // the other buffer was released by the barrier that ended the last chunk
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();  // this chunk complete in shared memory for every thread
    for (int r = 0; r < ne; r++) {
      float m[SPT][3];
#pragma unroll
      for (int s2 = 0; s2 < SPT; s2++)
#pragma unroll
        for (int cc = 0; cc < 3; cc++) m[s2][cc] = sM[buf][r][cc][s2 * P2M_B + tid];
      const float4* g4 = (const float4*)sG[buf][r];
#pragma unroll
      for (int q = 0; q < NN3 / 4; q++) {
        const float4 g = g4[q];  // values 4q .. 4q+3 = (j, comp) pairs in order
        const float gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int u = 0; u < 4; u++) {
          const int jc = 4 * q + u, j = jc / 3, comp = jc % 3;
#pragma unroll
          for (int s2 = 0; s2 < SPT; s2++) acc[s2][j] = fmaf(gv[u], m[s2][comp], acc[s2][j]);
        }
      }
    }
    __syncthreads();  // the buffer may be refilled
  }
#pragma unroll
  for (int s2 = 0; s2 < SPT; s2++) {
    const int b = bb + s2 * P2M_B + tid;
    if (b < B)
#pragma unroll
      for (int j = 0; j < NN; j++)
        if (n0 + j < nq) Q[((int64_t)c * nq + n0 + j) * B + b] = acc[s2][j];
  }
}

// P2M of small batches: block per (source leaf, SB states).  The tiles of
// k_p2m32 hold 128 states; here a thread is (moment q, node group g) and keeps
// SB states, the operator rows are read once, coalesced (12 bytes a thread), M
// of the chunk's nodes is a shared-memory broadcast.  The groups' sums are added
// in order.
constexpr int P2MS_THREADS = 256, P2MS_NE = 64;
template <class T, int SB>
__global__ void __launch_bounds__(P2MS_THREADS) k_p2m_small(const int32_t* __restrict__ leaves,
                                                              const int64_t* __restrict__ sup_off,
                                                              const int32_t* __restrict__ sup_node,
                                                              const T* __restrict__ G, int gs,
                                                              const T* __restrict__ Ms, int nq, int B, T* Q) {
  __shared__ T sM[P2MS_NE][3][SB];
  __shared__ T red[P2MS_THREADS][SB];
  const int32_t c = leaves[blockIdx.x];
  const int tid = threadIdx.x, b0 = blockIdx.y * SB;
  const int64_t so = sup_off[c];
  const int ns = (int)(sup_off[c + 1] - so);
  const int ng = min(8, P2MS_THREADS / nq), g = tid / nq, q = tid - g * nq;
  T acc[SB];
#pragma unroll
  for (int v = 0; v < SB; v++) acc[v] = (T)0;
  for (int e0 = 0; e0 < ns; e0 += P2MS_NE) {
    const int ne = min(P2MS_NE, ns - e0);
    __syncthreads();  // the previous chunk is no longer read
    for (int t = tid; t < ne * 3 * SB; t += P2MS_THREADS) {
      const int e = t / (3 * SB), r = t - e * 3 * SB, cc = r / SB, v = r - cc * SB;
      sM[e][cc][v] = b0 + v < B ? Ms[((int64_t)sup_node[so + e0 + e] * 3 + cc) * B + b0 + v] : (T)0;
    }
    __syncthreads();
    if (g < ng) {
      const T* gp = G + (so + e0) * gs + 3 * q;
#pragma unroll 4
      for (int e = g; e < ne; e += ng) {
        const T g0 = gp[(int64_t)e * gs], g1 = gp[(int64_t)e * gs + 1], g2 = gp[(int64_t)e * gs + 2];
#pragma unroll
        for (int v = 0; v < SB; v++) acc[v] = fma(g0, sM[e][0][v], fma(g1, sM[e][1][v], fma(g2, sM[e][2][v], acc[v])));
      }
    }
  }
#pragma unroll
  for (int v = 0; v < SB; v++) red[tid][v] = acc[v];
  __syncthreads();
  for (int t = tid; t < nq * SB; t += P2MS_THREADS) {
    const int qq = t / SB, v = t - qq * SB;
    if (b0 + v >= B) continue;
    T sum = (T)0;
    for (int gg = 0; gg < ng; gg++) sum += red[gg * nq + qq][v];
    Q[((int64_t)c * nq + qq) * B + b0 + v] = sum;
  }
}

// Largest batches of the small-batch P2M and L2P (slices of 8 states), whose time
// grows with the slices; the tiles cost the same up to 128 states.  P2M, small
// against tiles: 2,360 leaves (68k-tet ball, leaf 128) p = 8 32 states 81 / 123 us, p =
// 6 63 / 82, p = 4 24 states 46 / 51 and 32 states 55 / 50; 2,571 leaves (224k tets) p =
// 8 162 / 239, p = 6 115 / 155; 16,941 leaves of 13 tets, where a slice costs most, p =
// 8 24 states 391 / 481 and 32 states 520 / 489, p = 6 16 states 234 / 288 and 24 states
// 352 / 292, p = 4 8 states 95 / 165 and 16 states 183 / 167.  L2P, 24 and 32 states: p =
// 8 41 / 45 and 53 / 45 us; leaf 64, p = 6 59 / 98 and 87 / 98, p = 4 45 / 55 and 55 /
// 56; 29k tets, p = 8 12 / 16 and 14 / 16.
inline int p2m_small_batch(const Plan& P) {
  const bool many = P.h_src_leaves.size() > 8192;
  return P.nq <= 24 ? (many ? 8 : 24) : P.nq <= 48 ? (many ? 16 : 32) : (many ? 24 : 32);
}
constexpr int L2P_SMALL_BATCH = 32;

template <int SPT, int NN>
void launch_p2m_tile(Plan& P, int B, const float* Ms, float* Q, cudaStream_t s) {
  smem_opt_in((const void*)k_p2m32<SPT, NN>, p2m_smem<SPT, NN>());
  const dim3 grid((unsigned)P.h_src_leaves.size(), (unsigned)((P.nq + NN - 1) / NN),
                  (unsigned)((B + SPT * P2M_B - 1) / (SPT * P2M_B)));
  k_p2m32<SPT, NN><<<grid, P2M_B, p2m_smem<SPT, NN>(), s>>>(P.src_leaves, P.sup_off, P.sup_node, (const float*)P.far_G,
                                                           P.g_stride, Ms, P.nq, B, Q);
}

template <class T, int SB>
void launch_p2m_small(Plan& P, int B, const T* Ms, T* Q, cudaStream_t s) {
  const dim3 grid((unsigned)P.h_src_leaves.size(), (unsigned)((B + SB - 1) / SB));
  k_p2m_small<T, SB><<<grid, P2MS_THREADS, 0, s>>>(P.src_leaves, P.sup_off, P.sup_node, (const T*)P.far_G, P.g_stride,
                                                   Ms, P.nq, B, Q);
}

// Octree translations.  The child centres are at (+-h, +-h, +-h) of the parent's,
// so a term of index difference j takes the sign prod_a (+-1)^{j_a} of the
// child's octant o: (-1)^popcount(c & ~o) with c = (j_x, j_y, j_z) mod 2, the
// term's parity class.  Eight children therefore need every coefficient once:
//   M2M: T_c = sum_o (-1)^popcount(c & ~o) Qt_o  (Walsh-Hadamard transform over
//        the octants, 24 additions per moment), Qt^P_n = sum_e c_e T_{class e, k_e};
//   L2L: S_c = sum of the terms of class c, then the same transform gives the
//        eight children.
// At p = 8 ~1,800 products per parent and state instead of ~1,800 per child.
// Block per (parent, SW states), thread = (row, state); the transformed moments
// (the parent's coefficients) are staged in shared memory.  Measured against a
// thread per (parent, row, state) walking all children's terms through L2, one
// term after another (224k-tet ball): M2M 150 -> 45 us for one state, 777 -> 199
// us for 256; L2L 87 -> 49 us for one state, 330 -> 267 us for 256.
constexpr int TR_THREADS = 256;

// x_c = sum_o (-1)^popcount(c & ~o) x_o
template <class T>
__device__ __forceinline__ void octant_transform(T (&x)[8]) {
#pragma unroll
  for (int d = 1; d < 8; d <<= 1)
#pragma unroll
    for (int o = 0; o < 8; o++)
      if (!(o & d)) {
        const T lo = x[o], hi = x[o | d];
        x[o] = hi + lo;
        x[o | d] = hi - lo;
      }
}

// x_o = sum_c (-1)^popcount(c & ~o) x_c
template <class T>
__device__ __forceinline__ void classes_to_octants(T (&x)[8]) {
#pragma unroll
  for (int d = 1; d < 8; d <<= 1)
#pragma unroll
    for (int c = 0; c < 8; c++)
      if (!(c & d)) {
        const T even = x[c], odd = x[c | d];
        x[c] = even - odd;  // octant bit 0: the odd terms change sign
        x[c | d] = even + odd;
      }
}

template <class T, int SW>
__global__ void __launch_bounds__(TR_THREADS) k_m2m(const int32_t* __restrict__ parents,
                                                    const int32_t* __restrict__ child0,
                                                    const int32_t* __restrict__ nchild,
                                                    const uint64_t* __restrict__ prefix,
                                                    const int32_t* __restrict__ cnt, const TEnt<T>* __restrict__ ent,
                                                    int nq, int B, T* Q) {
  extern __shared__ __align__(16) unsigned char tr_smem[];
  T* sq = (T*)tr_smem;  // [class][moment][state]
  const int64_t P = parents[blockIdx.x];
  const int v = threadIdx.x % SW, r0 = threadIdx.x / SW, b = blockIdx.y * SW + v;
  const int nch = nchild[P];
  const int32_t c0 = child0[P];
  int pos[8];  // child of every octant, -1 = none
#pragma unroll
  for (int o = 0; o < 8; o++) pos[o] = -1;
  for (int k = 0; k < nch; k++) {
    const int o = (int)(prefix[c0 + k] & 7ull);
#pragma unroll
    for (int q = 0; q < 8; q++)
      if (q == o) pos[q] = c0 + k;
  }
  for (int n = r0; n < nq; n += TR_THREADS / SW) {
    T x[8];
#pragma unroll
    for (int o = 0; o < 8; o++) x[o] = pos[o] >= 0 && b < B ? Q[((int64_t)pos[o] * nq + n) * B + b] : (T)0;
    octant_transform(x);
#pragma unroll
    for (int o = 0; o < 8; o++) sq[(o * nq + n) * SW + v] = x[o];
  }
  __syncthreads();
  for (int n = r0; n < nq; n += TR_THREADS / SW) {
    const int ne = cnt[n];
    T a0 = (T)0, a1 = (T)0;
    int e = 0;
#pragma unroll 4
    for (; e + 1 < ne; e += 2) {
      const TEnt<T> E = ent[(int64_t)e * nq + n], F = ent[(int64_t)(e + 1) * nq + n];
      a0 = fma(E.c, sq[E.k * SW + v], a0);
      a1 = fma(F.c, sq[F.k * SW + v], a1);
    }
    if (e < ne) {
      const TEnt<T> E = ent[(int64_t)e * nq + n];
      a0 = fma(E.c, sq[E.k * SW + v], a0);
    }
    if (b < B) Q[(P * nq + n) * B + b] = a0 + a1;
  }
}

// bytes of the parent's coefficients and the class sums, to whole 16 bytes (the
// staged lists that follow hold 8- and 16-byte items)
template <class T>
__host__ __device__ constexpr size_t l2l_smem_base(int nl, int sw) {
  return (sizeof(T) * 9 * nl * sw + 15) / 16 * 16;
}

// added to the children's own M2L results
template <class T, int SW>
__global__ void __launch_bounds__(TR_THREADS) k_l2l(const int32_t* __restrict__ parents,
                                                    const int32_t* __restrict__ child0,
                                                    const int32_t* __restrict__ nchild, const int4* __restrict__ range,
                                                    const uint64_t* __restrict__ prefix,
                                                    const int2* __restrict__ cls, const TEnt<T>* __restrict__ ent,
                                                    int nent, bool staged, int nl, int B, T* L) {
  extern __shared__ __align__(16) unsigned char tr_smem[];
  T* sl = (T*)tr_smem;  // [coefficient][state]
  static_assert(2 * sizeof(TEnt<T>) % 16 == 0, "pairs of entries keep the 16-byte alignment");
  const int64_t P = parents[blockIdx.x];
  if (range[P].w == range[P].z) return;  // no target node below this cell
  const int v = threadIdx.x % SW, r0 = threadIdx.x / SW, b = blockIdx.y * SW + v;
  const int nch = nchild[P];
  const int32_t c0 = child0[P];
  for (int m = r0; m < nl; m += TR_THREADS / SW) sl[m * SW + v] = b < B ? L[(P * nl + m) * B + b] : (T)0;
  int pos[8];  // child with target nodes of every octant, -1 = none
#pragma unroll
  for (int o = 0; o < 8; o++) pos[o] = -1;
  for (int k = 0; k < nch; k++) {
    const int o = (int)(prefix[c0 + k] & 7ull);
    const int4 rg = range[c0 + k];
#pragma unroll
    for (int q = 0; q < 8; q++)
      if (q == o && rg.w > rg.z) pos[q] = c0 + k;
  }
  T* sc = sl + nl * SW;  // [row][class][state]: the classes of a row are short chains of their own
  // the entries too, where they fit (short chains of global loads were what this kernel waited for)
  const int2* cl = cls;
  const TEnt<T>* en = ent;
  if (staged) {
    TEnt<T>* se = (TEnt<T>*)(tr_smem + l2l_smem_base<T>(nl, SW));
    int2* scl = (int2*)(se + (nent + 1) / 2 * 2);  // both start on 16 bytes
    for (int e = threadIdx.x; e < nent; e += TR_THREADS) se[e] = ent[e];
    for (int q = threadIdx.x; q < 8 * nl; q += TR_THREADS) scl[q] = cls[q];
    en = se;
    cl = scl;
  }
  __syncthreads();
  for (int q = r0; q < 8 * nl; q += TR_THREADS / SW) {
    const int2 range_ = cl[q];
    T a = (T)0;
#pragma unroll 2
    for (int e = range_.x; e < range_.y; e++) {
      const TEnt<T> E = en[e];
      a = fma(E.c, sl[E.k * SW + v], a);
    }
    sc[q * SW + v] = a;
  }
  __syncthreads();
  for (int m = r0; m < nl; m += TR_THREADS / SW) {
    T y[8];
#pragma unroll
    for (int c = 0; c < 8; c++) y[c] = sc[(8 * m + c) * SW + v];
    classes_to_octants(y);
#pragma unroll
    for (int o = 0; o < 8; o++)
      if (pos[o] >= 0 && b < B) L[((int64_t)pos[o] * nl + m) * B + b] += y[o];
  }
}

// L2L of larger batches: thread per (parent, row, state), the states of a row
// side by side (whole lines of the children's rows; above 8 states 16-state
// slices in shared memory were up to 1.7x slower)
template <class T>
__global__ void __launch_bounds__(256) k_l2l_rows(const int32_t* __restrict__ parents, int64_t npar,
                                                  const int32_t* __restrict__ child0,
                                                  const int32_t* __restrict__ nchild, const int4* __restrict__ range,
                                                  const uint64_t* __restrict__ prefix, const int2* __restrict__ cls,
                                                  const TEnt<T>* __restrict__ ent, int nl, int B, T* L) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t per = (int64_t)nl * B;
  if (idx >= npar * per) return;
  const int64_t P = parents[idx / per];
  const int4 rp = range[P];
  if (rp.w == rp.z) return;  // no target node below this cell
  const int rem = (int)(idx % per), m = rem / B, b = rem - m * B;
  const T* Lp = L + P * per + b;
  T x[8];
#pragma unroll
  for (int c = 0; c < 8; c++) {
    const int2 e = cls[8 * m + c];
    T a = (T)0;
#pragma unroll 4
    for (int q = e.x; q < e.y; q++) a = fma(ent[q].c, Lp[(int64_t)ent[q].k * B], a);
    x[c] = a;
  }
  classes_to_octants(x);
  const int nch = nchild[P];
  const int32_t c0 = child0[P];
  for (int k = 0; k < nch; k++) {
    const int4 r = range[c0 + k];
    if (r.w == r.z) continue;  // only cells with target nodes
    const int o = (int)(prefix[c0 + k] & 7ull);
    T y = x[0];
#pragma unroll
    for (int q = 1; q < 8; q++) y = o == q ? x[q] : y;
    L[(int64_t)(c0 + k) * per + (int64_t)m * B + b] += y;
  }
}

// L2P: block per (leaf holding nodes, 128 states), 256 threads.  The leaf's
// local expansion (nl coefficients x 128 states, 32 KB at p = 8) is staged once
// in shared memory by asynchronous copies (coalesced over states); the nodes
// follow in chunks of 16, their polynomials transposed into [m][16 nodes], and
// thread (group g, states 2s and 2s + 1) accumulates the potentials of nodes
// 4g .. 4g + 3: per m one 8-byte and one broadcast 16-byte read for 8 FMAs.
constexpr int L2P_NCH = 16, L2P_THREADS = 256;

__global__ void __launch_bounds__(L2P_THREADS) k_l2p32(const int32_t* __restrict__ leaves,
                                                       const int4* __restrict__ range, const float* __restrict__ nodeh,
                                                       int nl, int B, const float* __restrict__ L, float* u) {
  extern __shared__ __align__(16) float l2p_smem[];
  float* sL = l2p_smem;              // [m][128 states]
  float* sh = l2p_smem + nl * 128;   // [m][16 nodes]
  const int32_t c = leaves[blockIdx.x];
  const int4 r = range[c];
  const int tid = threadIdx.x, sp = tid & 63, grp = tid >> 6, b0 = blockIdx.y * 128, b = b0 + 2 * sp;
  const float* Lc = L + (int64_t)c * nl * B + b0;
  if (B % 4 == 0) {  // rows of 16-byte vectors, whole within B
    for (int q = tid; q < nl * 32; q += L2P_THREADS) {
      const int m = q >> 5, v = 4 * (q & 31);
      const bool ok = b0 + v < B;
      cp_async16(sL + m * 128 + v, ok ? Lc + (int64_t)m * B + v : L, ok);
    }
  } else {
    for (int q = tid; q < nl * 128; q += L2P_THREADS) {
      const int m = q >> 7, v = q & 127;
      const bool ok = b0 + v < B;
      cp_async4(sL + q, ok ? Lc + (int64_t)m * B + v : L, ok);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  for (int32_t i0 = r.z; i0 < r.w; i0 += L2P_NCH) {
    const int nk = min(L2P_NCH, r.w - i0);
    __syncthreads();  // sL complete (first chunk); the previous chunk's polynomials are read
    for (int q = tid; q < L2P_NCH * nl; q += L2P_THREADS) {
      const int k = q / nl, m = q - k * nl;
      sh[m * L2P_NCH + k] = k < nk ? nodeh[(int64_t)(i0 + k) * nl + m] : 0.f;
    }
    __syncthreads();
    float a[2][4] = {};
#pragma unroll 4
    for (int m = 0; m < nl; m++) {
      const float2 l = *(const float2*)(sL + m * 128 + 2 * sp);
      const float4 w = *(const float4*)(sh + m * L2P_NCH + 4 * grp);
      const float wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        a[0][k] = fmaf(l.x, wv[k], a[0][k]);
        a[1][k] = fmaf(l.y, wv[k], a[1][k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (4 * grp + k >= nk) break;
      float* o = u + (int64_t)(i0 + 4 * grp + k) * B + b;
      if (b < B) o[0] = a[0][k];
      if (b + 1 < B) o[1] = a[1][k];
    }
  }
}

// L2P of small batches: block per (leaf holding nodes, SB states), the leaf's
// coefficients in shared memory, one warp per node: lanes stride the node's
// polynomials (coalesced), the states are added over the lanes by a fixed
// shuffle tree
constexpr int L2PS_THREADS = 128;
template <class T, int SB>
__global__ void __launch_bounds__(L2PS_THREADS) k_l2p_small(const int32_t* __restrict__ leaves,
                                                              const int4* __restrict__ range,
                                                              const T* __restrict__ nodeh, int nl, int B,
                                                              const T* __restrict__ L, T* u) {
  __shared__ T sL[MAX_P * MAX_P * SB];
  const int32_t c = leaves[blockIdx.x];
  const int4 r = range[c];
  const int b0 = blockIdx.y * SB, lane = threadIdx.x & 31;
  for (int q = threadIdx.x; q < nl * SB; q += L2PS_THREADS) {
    const int m = q / SB, v = q - m * SB;
    sL[q] = b0 + v < B ? L[((int64_t)c * nl + m) * B + b0 + v] : (T)0;
  }
  __syncthreads();
  for (int32_t i = r.z + (int)(threadIdx.x >> 5); i < r.w; i += L2PS_THREADS / 32) {
    T a[SB];
#pragma unroll
    for (int v = 0; v < SB; v++) a[v] = (T)0;
    for (int m = lane; m < nl; m += 32) {
      const T h = nodeh[(int64_t)i * nl + m];
#pragma unroll
      for (int v = 0; v < SB; v++) a[v] = fma(h, sL[m * SB + v], a[v]);
    }
#pragma unroll
    for (int v = 0; v < SB; v++) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a[v] += __shfl_xor_sync(0xffffffffu, a[v], o);
      if (lane == 0 && b0 + v < B) u[(int64_t)i * B + b0 + v] = a[v];
    }
  }
}

template <class T, int SB>
void launch_l2p_small(Plan& P, int B, const T* L, T* u, cudaStream_t s) {
  const dim3 grid((unsigned)P.n_node_leaves, (unsigned)((B + SB - 1) / SB));
  k_l2p_small<T, SB><<<grid, L2PS_THREADS, 0, s>>>(P.node_leaves, P.cell_range, (const T*)P.far_h, P.nl, B, L, u);
}

// coefficient lists of the translations on the trace-free coefficients
// (formulas in the file header) for the octant (+h, +h, +h); bit i of an octant
// is set where d_i = +h.  A fold moves n_x by multiples of two into n_y and
// n_z, so the parity class of a term is that of the folded index difference.
template <class T>
void build_translations(Plan& P) {
  const int p = P.p, nq = P.nq, nl = P.nl;
  double fact[MAX_P + 1] = {1.0};
  for (int i = 1; i <= MAX_P; i++) fact[i] = i * fact[i - 1];
  auto mono = [&](int e, int ja, int jb, int jc) {  // s_j(h, h, h) at h = 2^e, 0 below the index range
    if (ja < 0 || jb < 0 || jc < 0) return 0.0;
    return std::ldexp(1.0, e * (ja + jb + jc)) / (fact[ja] * fact[jb] * fact[jc]);
  };
  auto parity = [](int ja, int jb, int jc) { return (ja & 1) | ((jb & 1) << 1) | ((jc & 1) << 2); };
  std::vector<std::vector<TEnt<T>>> mrow(nq);
  std::vector<TEnt<T>> lent;
  std::vector<int2> lcls(8 * nl);
  for (int r = 0; r < nq; r++) {
    int ra, rb, rc;
    h_decode(r + 1, ra, rb, rc);
    for (int k = 0; k < nq; k++) {
      int ka, kb, kc;
      h_decode(k + 1, ka, kb, kc);
      const double cf = h_fold(ra, rb, rc, [&](int na, int nb, int nz) { return mono(-2, na - ka, nb - kb, nz - kc); }) *
                        std::ldexp(1.0, -(ka + kb + kc));
      if (cf != 0.0) mrow[r].push_back(TEnt<T>{(uint16_t)(parity(ra + ka, rb + kb, rc + kc) * nq + k), (T)cf});
    }
  }
  for (int m = 0; m < nl; m++) {
    int ma, mb, mc;
    h_decode(m, ma, mb, mc);
    for (int cls = 0; cls < 8; cls++) {  // entries by parity class
      lcls[8 * m + cls].x = (int)lent.size();
      for (int r = 0; r < nl; r++) {     // parent coefficients of degree p are zero
        int ra, rb, rc;
        h_decode(r, ra, rb, rc);
        if (parity(ra + ma, rb + mb, rc + mc) != cls) continue;
        const double cf = h_fold(ra, rb, rc, [&](int ka, int kb, int kz) { return mono(-1, ka - ma, kb - mb, kz - mc); }) *
                          std::ldexp(1.0, -(ra + rb + rc));
        if (cf != 0.0) lent.push_back(TEnt<T>{(uint16_t)r, (T)cf});
      }
      lcls[8 * m + cls].y = (int)lent.size();
    }
  }
  cudaStream_t s = P.stream;
  size_t width = 1;
  std::vector<int32_t> mcnt(nq);
  for (int r = 0; r < nq; r++) {
    mcnt[r] = (int32_t)mrow[r].size();
    width = std::max(width, mrow[r].size());
  }
  std::vector<TEnt<T>> ment(width * nq, TEnt<T>{0, (T)0});
  for (int r = 0; r < nq; r++)
    for (size_t j = 0; j < mrow[r].size(); j++) ment[j * nq + r] = mrow[r][j];
  P.m2m_width = (int)width;
  P.l2l_nent = (int)lent.size();
  P.m2m_cnt = dalloc<int32_t>(P, nq);
  P.m2m_ent = dalloc<TEnt<T>>(P, ment.size());
  P.l2l_cls = dalloc<int2>(P, lcls.size());
  P.l2l_ent = dalloc<TEnt<T>>(P, lent.size());
  DM_CUDA(cudaMemcpyAsync(P.m2m_cnt, mcnt.data(), nq * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaMemcpyAsync(P.m2m_ent, ment.data(), ment.size() * sizeof(TEnt<T>), cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaMemcpyAsync(P.l2l_cls, lcls.data(), lcls.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaMemcpyAsync(P.l2l_ent, lent.data(), lent.size() * sizeof(TEnt<T>), cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaStreamSynchronize(s));
}

// cells with children, level by level (the M2M and L2L launches run over these only)
void build_parent_lists(Plan& P) {
  cudaStream_t s = P.stream;
  std::vector<int32_t> nch(P.ncells), list;
  DM_CUDA(cudaMemcpyAsync(nch.data(), P.cell_nchild, sizeof(int32_t) * P.ncells, cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaStreamSynchronize(s));
  P.par_start.assign(1, 0);
  for (int l = 0; l < P.nlevels; l++) {
    for (int64_t c = P.level_start[l]; c < P.level_start[l + 1]; c++)
      if (nch[c] > 0) list.push_back((int32_t)c);
    P.par_start.push_back((int64_t)list.size());
  }
  P.par_list = dalloc<int32_t>(P, std::max<size_t>(list.size(), 1));
  if (!list.empty())
    DM_CUDA(cudaMemcpyAsync(P.par_list, list.data(), sizeof(int32_t) * list.size(), cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaStreamSynchronize(s));
}

template <class T>
void build_operators(Plan& P) {
  build_translations<T>(P);
  cudaStream_t s = P.stream;
  P.g_stride = (3 * P.nq + 3) / 4 * 4;
  T* G = dalloc<T>(P, std::max<int64_t>(P.n_sup, 1) * P.g_stride);
  T* h = dalloc<T>(P, P.nn * P.nl);
  P.far_G = G;
  P.far_h = h;
  if (!P.h_src_leaves.empty()) {
    k_p2m_op<T><<<(unsigned)P.h_src_leaves.size(), 256, 0, s>>>(P.src_leaves, P.cell_level, P.sup_off, P.Ghat, P.side,
                                                                P.nc1, P.nq, P.g_stride, G);
    DM_LAUNCH("k_p2m_op");
  }
  k_node_h<T><<<nblk(P.nn, NODE_H), 256, 0, s>>>(P.nn, P.node_leaf, P.cell_level, P.nodes_s, P.cell_centre, P.side, P.p,
                                                 P.nl, h);
  DM_LAUNCH("k_node_h");
}

}  // namespace

void build_far_operators(Plan& P) {
  build_parent_lists(P);
  if (P.opt.precision == DEMAG_FP64)
    build_operators<double>(P);
  else
    build_operators<float>(P);
  if (P.n_m2l == 0) return;
  const bool fp64 = P.opt.precision == DEMAG_FP64;
  if (fp64 && P.opt.m2l_table_batch < 0) return;  // FP64 without a table
  const M2lKeys K = build_m2l_keys(P);
  if (!fp64) build_m2l_tc(P, K);
  build_m2l_tab(P, K);
}

template <class T>
int launch_p2m(Plan& P, int B, const T* Ms, T* Q, cudaStream_t s) {
  if (P.h_src_leaves.empty()) return 0;
  if (B == 1)
    launch_p2m_small<T, 1>(P, B, Ms, Q, s);
  else if (B == 2)
    launch_p2m_small<T, 2>(P, B, Ms, Q, s);
  else if (B <= 4)
    launch_p2m_small<T, 4>(P, B, Ms, Q, s);
  else if (B <= p2m_small_batch(P) || std::is_same<T, double>::value)
    launch_p2m_small<T, 8>(P, B, Ms, Q, s);
  else if constexpr (std::is_same<T, float>::value) {
    if (P.nq <= 24)
      B > P2M_B ? launch_p2m_tile<2, 24>(P, B, Ms, Q, s) : launch_p2m_tile<1, 24>(P, B, Ms, Q, s);
    else if (P.nq <= 48)
      B > P2M_B ? launch_p2m_tile<2, 48>(P, B, Ms, Q, s) : launch_p2m_tile<1, 48>(P, B, Ms, Q, s);
    else
      B > P2M_B ? launch_p2m_tile<2, 80>(P, B, Ms, Q, s) : launch_p2m_tile<1, 80>(P, B, Ms, Q, s);
  }
  DM_LAUNCH("k_p2m");
  return 1;
}

namespace {

template <class T, int SW>
void launch_m2m_level(Plan& P, int64_t pb, int64_t np, int B, T* Q, cudaStream_t s) {
  const size_t smem = sizeof(T) * SW * 8 * P.nq;
  smem_opt_in((const void*)k_m2m<T, SW>, smem);
  k_m2m<T, SW><<<dim3((unsigned)np, (unsigned)((B + SW - 1) / SW)), TR_THREADS, smem, s>>>(
      P.par_list + pb, P.cell_child0, P.cell_nchild, P.cell_prefix, P.m2m_cnt, (const TEnt<T>*)P.m2m_ent, P.nq, B, Q);
  DM_LAUNCH("k_m2m");
}

template <class T, int SW>
void launch_l2l_level(Plan& P, int64_t pb, int64_t np, int B, T* L, cudaStream_t s) {
  const size_t base = l2l_smem_base<T>(P.nl, SW);
  const size_t ents = sizeof(TEnt<T>) * ((P.l2l_nent + 1) / 2 * 2) + sizeof(int2) * 8 * P.nl;
  const bool staged = base + ents <= 100 * 1024;  // two blocks per SM
  const size_t smem = base + (staged ? ents : 0);
  smem_opt_in((const void*)k_l2l<T, SW>, smem);
  k_l2l<T, SW><<<dim3((unsigned)np, (unsigned)((B + SW - 1) / SW)), TR_THREADS, smem, s>>>(
      P.par_list + pb, P.cell_child0, P.cell_nchild, P.cell_range, P.cell_prefix, P.l2l_cls,
      (const TEnt<T>*)P.l2l_ent, P.l2l_nent, staged, P.nl, B, L);
  DM_LAUNCH("k_l2l");
}

}  // namespace

template <class T>
int launch_m2m(Plan& P, int B, T* Q, cudaStream_t s) {
  int n = 0;
  for (int l = P.nlevels - 2; l >= 0; l--) {
    const int64_t pb = P.par_start[l], np = P.par_start[l + 1] - pb;
    if (np == 0) continue;
    if (B == 1)
      launch_m2m_level<T, 1>(P, pb, np, B, Q, s);
    else if (B == 2)
      launch_m2m_level<T, 2>(P, pb, np, B, Q, s);
    else if (B <= 4)
      launch_m2m_level<T, 4>(P, pb, np, B, Q, s);
    else if (B <= 8)
      launch_m2m_level<T, 8>(P, pb, np, B, Q, s);
    else
      launch_m2m_level<T, 16>(P, pb, np, B, Q, s);
    n++;
  }
  return n;
}

template <class T>
int launch_l2l(Plan& P, int B, T* L, cudaStream_t s) {
  int n = 0;
  for (int l = 0; l + 1 < P.nlevels; l++) {  // parents at level l, children at l + 1
    const int64_t pb = P.par_start[l], np = P.par_start[l + 1] - pb;
    if (np == 0) continue;
    if (B == 1)
      launch_l2l_level<T, 1>(P, pb, np, B, L, s);
    else if (B == 2)
      launch_l2l_level<T, 2>(P, pb, np, B, L, s);
    else if (B <= 4)
      launch_l2l_level<T, 4>(P, pb, np, B, L, s);
    else if (B <= 8)
      launch_l2l_level<T, 8>(P, pb, np, B, L, s);
    else {
      k_l2l_rows<T><<<nblk(np * P.nl * B, 256), 256, 0, s>>>(P.par_list + pb, np, P.cell_child0, P.cell_nchild,
                                                             P.cell_range, P.cell_prefix, P.l2l_cls,
                                                             (const TEnt<T>*)P.l2l_ent, P.nl, B, L);
      DM_LAUNCH("k_l2l_rows");
    }
    n++;
  }
  return n;
}

template <class T>
int launch_l2p(Plan& P, int B, const T* L, T* u, cudaStream_t s) {
  if (P.n_node_leaves == 0) return 0;
  if (B == 1)
    launch_l2p_small<T, 1>(P, B, L, u, s);
  else if (B == 2)
    launch_l2p_small<T, 2>(P, B, L, u, s);
  else if (B <= 4)
    launch_l2p_small<T, 4>(P, B, L, u, s);
  else if (B <= L2P_SMALL_BATCH || std::is_same<T, double>::value)
    launch_l2p_small<T, 8>(P, B, L, u, s);
  else if constexpr (std::is_same<T, float>::value) {
    const size_t smem = sizeof(float) * (size_t)P.nl * (128 + L2P_NCH);
    smem_opt_in((const void*)k_l2p32, smem);
    const dim3 grid((unsigned)P.n_node_leaves, (unsigned)((B + 127) / 128));
    k_l2p32<<<grid, L2P_THREADS, smem, s>>>(P.node_leaves, P.cell_range, (const float*)P.far_h, P.nl, B, L, u);
  }
  DM_LAUNCH("k_l2p");
  return 1;
}

template int launch_p2m<float>(Plan&, int, const float*, float*, cudaStream_t);
template int launch_p2m<double>(Plan&, int, const double*, double*, cudaStream_t);
template int launch_m2m<float>(Plan&, int, float*, cudaStream_t);
template int launch_m2m<double>(Plan&, int, double*, cudaStream_t);
template int launch_l2l<float>(Plan&, int, float*, cudaStream_t);
template int launch_l2l<double>(Plan&, int, double*, cudaStream_t);
template int launch_l2p<float>(Plan&, int, const float*, float*, cudaStream_t);
template int launch_l2p<double>(Plan&, int, const double*, double*, cudaStream_t);

}  // namespace demag
