// p2p.cu -- near field (Sec. 2.1): per-tet geometry, and the FP64 near field
// integrated at every evaluation (near_mode 0), by the faces of the source tets.
//
// The potential of a tet with affine M is a sum over its faces (p2p.cuh),
//   4 pi u = sum_F h_F (M(r).A_F + (1/2) T_F:J),   h_F = n_F.(r - a_F),  J = dM/dx,
// M(r) the tet's affine M continued to the target.  A_F and T_F belong to the
// face, h_F changes sign with the side.  M is nodal, so across a face shared by
// two tets it is continuous: the difference of the two affine functions is
// (dM/dn)_jump n.(r' - a), its J difference is of rank one, T_F n = -h_F A_F, and
// an interior face of a set of tets leaves
//   h (h j.A - (1/2) h j.A) = (1/2) h^2 j.A_F,   j = jump of dM/dn.
// The source leaves are cut, in their sorted (Morton) order, into clusters of at
// most CL_TETS tets; a cluster keeps its distinct vertices, edges and faces, and
// per target
//   R_v      once per vertex  (0.5 - 0.7 per tet, 4 in the tet-wise form),
//   Lam_e    once per edge    (1.8 - 2.2 per tet instead of 6 logarithms),
//   Omega_F  once per face    (2.6 - 2.9 per tet instead of 4 solid angles).
// The cluster's boundary faces (one tet in the cluster) take the whole sum.  In
// the face's frame (t along edge 0, m = t x n, n), with foot (x, y) of r from
// vertex 0, edge normals m_e = c_e t + d_e m, w_e = P0_e Lam_e, dR_e = R_end -
// R_start and I = sum_e w_e + h Omega (p2p.cuh has the derivation):
//   A = (P_t, P_m, Omega),  P_t = -sum c_e Lam_e,  P_m = -sum d_e Lam_e
//   S_tt = I - sum (w c^2 + dR c d),  S_mm = I - sum (w d^2 - dR c d),
//   S_tm = -sum (w c d + dR (d^2 - c^2) / 2)     (the in-plane part of T)
//   4 pi u_F = h [M_0.A + G_t.(x A + (S_tt, S_tm, -h P_t)/2)
//                       + G_m.(y A + (S_tm, S_mm, -h P_m)/2)] + (1/2) h^2 dM/dn.A
// M_0 at vertex 0, G the in-plane derivatives of M.
//
// Rounding.  The terms are those of the tet-wise form, and so is the error: every
// one carries the height h, no term is divided by a height of the triangle, and
// M enters by its derivatives.  (Face charges n.M and jumps of div M need fewer
// products per state, but int_F (n.M)/R dA carries an error of eps R L per
// derivative of M where this form has eps h L: 5 to 20 times the error on
// flattened tets.)  Against 80-bit arithmetic, theta -> 0, smooth M | Gaussian M
// per node, here (tet-wise kernels for one state / batched in parentheses):
//   balls of 0.2 - 2k tets (14, means)  3.3e-15 (5.1e-15 / 2.7e-15) | 1.7e-14 (2.6e-14 / 1.4e-14)
//   film, cells of 6.7:1                3.9e-15 (5.8e-15 / 4.4e-15) | 3.2e-14 (3.4e-14 / 3.3e-14)
//   film, cells of 20:1                 1.2e-14 (1.5e-14 / 1.1e-14) | 2.2e-13 (3.0e-13 / 2.2e-13)
//   film, cells of 100:1                1.5e-13 (2.0e-13 / 1.6e-13) | 3.4e-12 (4.0e-12 / 3.5e-12)
//   ball squeezed to 1:20               1.1e-14 (1.2e-14 / 1.2e-14) | 1.1e-13 (1.2e-13 / 1.0e-13)
//   ball stretched to 20:1              8.6e-15 (1.1e-14 / 8.7e-15) | 1.3e-13 (1.6e-13 / 1.3e-13)
#include <algorithm>
#include <utility>
#include <vector>

#include "common.cuh"
#include "p2p.cuh"

namespace demag {

static inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

// ---------------------------------------------------------------------------
// per-tet geometry (plan time)
// ---------------------------------------------------------------------------
__global__ void k_tet_geometry(int64_t nt, const double* __restrict__ nodes_s, int32_t* tets_s, double* geo,
                               double* grad, double* vol) {
  int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= nt) return;
  int32_t g[4];
  double v[4][3];
  for (int k = 0; k < 4; k++) {
    g[k] = tets_s[4 * j + k];
    for (int c = 0; c < 3; c++) v[k][c] = nodes_s[3 * (int64_t)g[k] + c];
  }
  double e1[3], e2[3], e3[3];
  for (int c = 0; c < 3; c++) {
    e1[c] = v[1][c] - v[0][c];
    e2[c] = v[2][c] - v[0][c];
    e3[c] = v[3][c] - v[0][c];
  }
  double c23[3] = {e2[1] * e3[2] - e2[2] * e3[1], e2[2] * e3[0] - e2[0] * e3[2], e2[0] * e3[1] - e2[1] * e3[0]};
  double det = e1[0] * c23[0] + e1[1] * c23[1] + e1[2] * c23[2];
  if (det < 0) {  // store positively oriented: swap vertices 2 and 3
    int32_t t = g[2];
    g[2] = g[3];
    g[3] = t;
    tets_s[4 * j + 2] = g[2];
    tets_s[4 * j + 3] = g[3];
    for (int c = 0; c < 3; c++) {
      double x = v[2][c];
      v[2][c] = v[3][c];
      v[3][c] = x;
      x = e2[c];
      e2[c] = e3[c];
      e3[c] = x;
    }
    det = -det;
    c23[0] = e2[1] * e3[2] - e2[2] * e3[1];
    c23[1] = e2[2] * e3[0] - e2[0] * e3[2];
    c23[2] = e2[0] * e3[1] - e2[1] * e3[0];
  }
  double c31[3] = {e3[1] * e1[2] - e3[2] * e1[1], e3[2] * e1[0] - e3[0] * e1[2], e3[0] * e1[1] - e3[1] * e1[0]};
  double c12[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
  double inv = 1.0 / det;
  double* gr = grad + 12 * j;
  for (int c = 0; c < 3; c++) {
    gr[3 + c] = c23[c] * inv;
    gr[6 + c] = c31[c] * inv;
    gr[9 + c] = c12[c] * inv;
    gr[c] = -(gr[3 + c] + gr[6 + c] + gr[9 + c]);
  }
  vol[j] = det / 6.0;
  double* G = geo + (int64_t)TET_GEO * j;
  for (int k = 0; k < 4; k++)
    for (int c = 0; c < 3; c++) G[3 * k + c] = v[k][c];
  for (int F = 0; F < 4; F++) {
    int p = face_vertex(F, 0), q = face_vertex(F, 1), s = face_vertex(F, 2);
    double u1[3], u2[3];
    for (int c = 0; c < 3; c++) {
      u1[c] = v[q][c] - v[p][c];
      u2[c] = v[s][c] - v[p][c];
    }
    double n[3] = {u1[1] * u2[2] - u1[2] * u2[1], u1[2] * u2[0] - u1[0] * u2[2], u1[0] * u2[1] - u1[1] * u2[0]};
    double ln = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    for (int c = 0; c < 3; c++) n[c] /= ln;
    for (int c = 0; c < 3; c++) G[12 + 3 * F + c] = n[c];
    for (int e = 0; e < 3; e++) {
      int a0 = face_vertex(F, e), a1 = face_vertex(F, (e + 1) % 3);
      double t[3];
      for (int c = 0; c < 3; c++) t[c] = v[a1][c] - v[a0][c];
      double lt = sqrt(t[0] * t[0] + t[1] * t[1] + t[2] * t[2]);
      for (int c = 0; c < 3; c++) t[c] /= lt;
      double m[3] = {t[1] * n[2] - t[2] * n[1], t[2] * n[0] - t[0] * n[2], t[0] * n[1] - t[1] * n[0]};
      for (int c = 0; c < 3; c++) G[24 + 9 * F + 3 * e + c] = m[c];
    }
  }
  for (int e = 0; e < 6; e++) {
    int a0 = edge_v0(e), a1 = edge_v1(e);
    double dx = v[a1][0] - v[a0][0], dy = v[a1][1] - v[a0][1], dz = v[a1][2] - v[a0][2];
    G[60 + e] = sqrt(dx * dx + dy * dy + dz * dz);
  }
}

void build_tet_geometry(Plan& P) {
  P.tet_geo = dalloc<double>(P, (size_t)TET_GEO * P.nt);
  P.tet_grad = dalloc<double>(P, 12 * (size_t)P.nt);
  P.tet_vol = dalloc<double>(P, P.nt);
  k_tet_geometry<<<nblk(P.nt, 128), 128, 0, P.stream>>>(P.nt, P.nodes_s, P.tets_s, P.tet_geo, P.tet_grad, P.tet_vol);
  DM_LAUNCH("k_tet_geometry");
}

// ---------------------------------------------------------------------------
// clusters of source tets (plan time)
// ---------------------------------------------------------------------------
namespace {

constexpr int PF_GMIN = 4;               // target nodes of a block of a split leaf, at least
constexpr double PF_SPLIT = 4.0;
constexpr int FACE_REC = 16;             // doubles per face: n, t, m (9), 2 area, c_1, d_1, c_2, d_2, 1 / length of edge 0, (v2 - v0).t
static_assert(CL_V <= 256 && CL_E <= 512, "8-bit vertex and 9-bit edge positions");

// sorts, returns 1 for an odd permutation; faces list their vertices counter-clockwise seen from outside
__device__ __forceinline__ int sort3(int32_t& a, int32_t& b, int32_t& c) {
  int odd = 0;
  if (a > b) { const int32_t t = a; a = b; b = t; odd ^= 1; }
  if (b > c) { const int32_t t = b; b = c; c = t; odd ^= 1; }
  if (a > b) { const int32_t t = a; a = b; b = t; odd ^= 1; }
  return odd;
}

// one block per cluster: its distinct vertices and edges, and its faces with
// the boundary faces first.  An interior face is one that exactly two tets of
// the cluster list, with opposite orientations; any other face (one tet, or
// tets overlapping) is kept once per tet as a boundary face.  FILL = false
// counts, FILL = true writes.
template <bool FILL>
__global__ void __launch_bounds__(256) k_clusters(const int2* __restrict__ range, const int32_t* __restrict__ tets_s,
                                                  const double* __restrict__ geo, int4* cnt,
                                                  const int4* __restrict__ off, int32_t* vnode, uint32_t* edge,
                                                  double* elen, double* frec, uint2* fidx, int2* ftet) {
  __shared__ int32_t vid[CL_V];                       // node of every tet corner
  __shared__ int32_t vloc[CL_V], eloc[CL_E];          // its position among the distinct ones
  __shared__ uint32_t ekey[CL_E];
  __shared__ int32_t fk[CL_F][3];
  __shared__ int fodd[CL_F], fother[CL_F], flag[CL_E];
  const int2 rg = range[blockIdx.x];
  const int nt = rg.y - rg.x, tid = threadIdx.x;
  for (int q = tid; q < 4 * nt; q += blockDim.x) vid[q] = tets_s[4ll * rg.x + q];
  __syncthreads();
  // distinct vertices: the first corner with the node owns it
  for (int q = tid; q < 4 * nt; q += blockDim.x) {
    int j = 0;
    while (vid[j] != vid[q]) j++;
    flag[q] = j;
  }
  __syncthreads();
  for (int q = tid; q < 4 * nt; q += blockDim.x) {
    int n = 0;
    for (int j = 0; j < flag[q]; j++) n += flag[j] == j;
    vloc[q] = n;
  }
  int nv = 0, ne = 0, nf = 0, nb = 0;
  for (int j = 0; j < 4 * nt; j++) nv += flag[j] == j;
  if (FILL)
    for (int q = tid; q < 4 * nt; q += blockDim.x)
      if (flag[q] == q) vnode[off[blockIdx.x].x + vloc[q]] = vid[q];
  __syncthreads();
  // distinct edges
  for (int q = tid; q < 6 * nt; q += blockDim.x) {
    const int t = q / 6, e = q - 6 * t;
    const int a = vloc[4 * t + edge_v0(e)], b = vloc[4 * t + edge_v1(e)];
    ekey[q] = (uint32_t)min(a, b) | ((uint32_t)max(a, b) << 16);
  }
  __syncthreads();
  for (int q = tid; q < 6 * nt; q += blockDim.x) {
    int j = 0;
    while (ekey[j] != ekey[q]) j++;
    flag[q] = j;
  }
  __syncthreads();
  for (int q = tid; q < 6 * nt; q += blockDim.x) {
    int n = 0;
    for (int j = 0; j < flag[q]; j++) n += flag[j] == j;
    eloc[q] = n;
  }
  for (int j = 0; j < 6 * nt; j++) ne += flag[j] == j;
  if (FILL)
    for (int q = tid; q < 6 * nt; q += blockDim.x)
      if (flag[q] == q) {
        edge[off[blockIdx.x].y + eloc[q]] = ekey[q];
        elen[off[blockIdx.x].y + eloc[q]] = geo[(int64_t)TET_GEO * (rg.x + q / 6) + 60 + q % 6];
      }
  __syncthreads();
  // faces
  for (int q = tid; q < 4 * nt; q += blockDim.x) {
    const int t = q >> 2, F = q & 3;
    int32_t a = vid[4 * t + face_vertex(F, 0)], b = vid[4 * t + face_vertex(F, 1)], c = vid[4 * t + face_vertex(F, 2)];
    fodd[q] = sort3(a, b, c);
    fk[q][0] = a;
    fk[q][1] = b;
    fk[q][2] = c;
  }
  __syncthreads();
  for (int q = tid; q < 4 * nt; q += blockDim.x) {
    int n = 0, other = -1;
    for (int j = 0; j < 4 * nt; j++)
      if (j != q && fk[j][0] == fk[q][0] && fk[j][1] == fk[q][1] && fk[j][2] == fk[q][2]) {
        n++;
        other = j;
      }
    fother[q] = n == 1 && fodd[other] != fodd[q] ? other : -1;
  }
  __syncthreads();
  for (int j = 0; j < 4 * nt; j++) {
    nb += fother[j] < 0;
    nf += fother[j] < 0 || fother[j] > j;
  }
  if (!FILL) {
    if (tid == 0) cnt[blockIdx.x] = make_int4(nv, ne, nf, nb);
    return;
  }
  for (int q = tid; q < 4 * nt; q += blockDim.x) {
    const bool bnd = fother[q] < 0;
    if (!bnd && fother[q] < q) continue;  // the other tet's copy owns it
    int k = bnd ? 0 : nb;
    for (int j = 0; j < q; j++) k += bnd ? fother[j] < 0 : fother[j] > j;
    const int t = q >> 2, F = q & 3;
    const int64_t o = off[blockIdx.x].z + k;
    // the record depends on the face alone: its vertices by node id, the frame of that order
    int cor[3];  // corners of tet t
    for (int e = 0; e < 3; e++)
      for (int c = 0; c < 3; c++)
        if (vid[4 * t + face_vertex(F, c)] == fk[q][e]) cor[e] = face_vertex(F, c);
    const double* G = geo + (int64_t)TET_GEO * (rg.x + t);
    double v[3][3];
    for (int e = 0; e < 3; e++)
      for (int c = 0; c < 3; c++) v[e][c] = G[3 * cor[e] + c];
    double* R = frec + FACE_REC * o;
    double u[3], w[3], n[3], tg[3][3], m[3][3], len0 = 0.0;
    for (int c = 0; c < 3; c++) {
      u[c] = v[1][c] - v[0][c];
      w[c] = v[2][c] - v[0][c];
    }
    n[0] = u[1] * w[2] - u[2] * w[1];
    n[1] = u[2] * w[0] - u[0] * w[2];
    n[2] = u[0] * w[1] - u[1] * w[0];
    const double a2 = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
    for (int c = 0; c < 3; c++) n[c] /= a2;
    for (int e = 0; e < 3; e++) {  // m = t x n, t the unit tangent
      for (int c = 0; c < 3; c++) tg[e][c] = v[(e + 1) % 3][c] - v[e][c];
      const double l = sqrt(tg[e][0] * tg[e][0] + tg[e][1] * tg[e][1] + tg[e][2] * tg[e][2]);
      if (e == 0) len0 = l;
      for (int c = 0; c < 3; c++) tg[e][c] /= l;
      m[e][0] = tg[e][1] * n[2] - tg[e][2] * n[1];
      m[e][1] = tg[e][2] * n[0] - tg[e][0] * n[2];
      m[e][2] = tg[e][0] * n[1] - tg[e][1] * n[0];
    }
    auto dot = [](const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
    for (int c = 0; c < 3; c++) {
      R[c] = n[c];
      R[3 + c] = tg[0][c];
      R[6 + c] = m[0][c];
    }
    R[9] = a2;
    for (int e = 1; e < 3; e++) {
      R[8 + 2 * e] = dot(m[e], tg[0]);
      R[9 + 2 * e] = dot(m[e], m[0]);
    }
    R[14] = 1.0 / len0;
    R[15] = dot(w, tg[0]);
    uint32_t es = 0, vs = fodd[q] ? 0x80000000u : 0u;  // top bit: n points into the tet
    for (int e = 0; e < 3; e++) {
      es |= (uint32_t)eloc[6 * t + edge_id(cor[e], cor[(e + 1) % 3])] << (9 * e);
      vs |= (uint32_t)vloc[4 * t + cor[e]] << (8 * e);
    }
    fidx[o] = make_uint2(vs, es);
    ftet[o] = make_int2(rg.x + t, bnd ? -1 : rg.x + (fother[q] >> 2));
  }
}

// clusters of every P2P target leaf: one per (source leaf of its list, cluster of that leaf)
template <bool FILL>
__global__ void k_cluster_lists(const int32_t* __restrict__ targets, const int64_t* __restrict__ p2p_off,
                                const int32_t* __restrict__ p2p_src, const int32_t* __restrict__ cl_off, int64_t* cnt,
                                const int64_t* __restrict__ pc_off, int32_t* pc_src) {
  __shared__ long long total;
  const int32_t T = targets[blockIdx.x];
  if (!FILL) {
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    long long n = 0;
    for (int64_t e = p2p_off[T] + threadIdx.x; e < p2p_off[T + 1]; e += blockDim.x)
      n += cl_off[p2p_src[e] + 1] - cl_off[p2p_src[e]];
    atomicAdd((unsigned long long*)&total, (unsigned long long)n);
    __syncthreads();
    if (threadIdx.x == 0) cnt[blockIdx.x] = total;
  } else if (threadIdx.x < 32) {  // one warp, in list order
    int64_t o = pc_off[blockIdx.x];
    const int lane = threadIdx.x;
    for (int64_t e0 = p2p_off[T]; e0 < p2p_off[T + 1]; e0 += 32) {
      const bool on = e0 + lane < p2p_off[T + 1];
      const int32_t S = on ? p2p_src[e0 + lane] : 0;
      const int c0 = on ? cl_off[S] : 0, n = on ? cl_off[S + 1] - c0 : 0;
      int sum = n;  // inclusive scan
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, sum, d);
        if (lane >= d) sum += v;
      }
      for (int k = 0; k < n; k++) pc_src[o + sum - n + k] = c0 + k;
      o += __shfl_sync(0xffffffffu, sum, 31);
    }
  }
}

// The near field's blocks, heaviest first: {P2P target, first target node, nodes, 0}.
// A block's time is its targets times its list, and the lists of an octree's
// leaves differ several times in length: 16 nodes per block in leaf order left
// the SMs busy for 48% of the kernel on the 16k-tet ball (708 blocks, the SMs'
// active cycles 14 to 93 million).  A target leaf whose 16 nodes cost more than
// 1/PF_SPLIT of the mean share of a resident block takes 8 or 4 at a time: an
// evaluation of three states 46.4 -> 19.9 ms (the kernel of that time).  Clusters staged for fewer targets cost little, the
// FP64 arithmetic is the bound; below 4 targets a warp would read 16 records a step.
std::vector<int4> face_blocks(const Plan& P, const std::vector<int64_t>& clusters) {
  const int64_t nT = (int64_t)clusters.size();
  double total = 0;
  for (int64_t t = 0; t < nT; t++) {
    const int4 r = P.h_range[P.h_p2p_targets[t]];
    total += (double)clusters[t] * (r.w - r.z);
  }
  const double most = total / (2.0 * P.sms * PF_SPLIT);  // two blocks per SM
  std::vector<std::pair<double, int4>> q;
  for (int64_t t = 0; t < nT; t++) {
    const int4 r = P.h_range[P.h_p2p_targets[t]];
    int g = PF_G;
    while (g > PF_GMIN && (double)clusters[t] * g > most) g /= 2;
    for (int i = r.z; i < r.w; i += g) {
      const int n = std::min(g, r.w - i);
      q.emplace_back((double)clusters[t] * n, make_int4((int)t, i, n, 0));
    }
  }
  std::stable_sort(q.begin(), q.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
  std::vector<int4> o;
  o.reserve(q.size());
  for (const auto& x : q) o.push_back(x.second);
  return o;
}

}  // namespace

void build_clusters(Plan& P) {
  cudaStream_t s = P.stream;
  const int64_t nc = P.ncells, nT = (int64_t)P.h_p2p_targets.size();
  std::vector<int32_t> off(nc + 1, 0);
  std::vector<int2> range;
  std::vector<char> is_src(nc, 0);
  for (int32_t c : P.h_src_leaves) is_src[c] = 1;
  for (int64_t c = 0; c < nc; c++) {
    if (is_src[c]) {  // equal pieces of at most CL_TETS tets
      const int4 r = P.h_range[c];
      const int n = r.y - r.x, k = (n + CL_TETS - 1) / CL_TETS;
      for (int i = 0; i < k; i++)
        range.push_back(make_int2(r.x + (int)((int64_t)n * i / k), r.x + (int)((int64_t)n * (i + 1) / k)));
    }
    off[c + 1] = (int32_t)range.size();
  }
  P.n_clusters = (int64_t)range.size();
  if (P.n_clusters == 0) return;
  int2* drange = dalloc<int2>(P, range.size());
  int4* dcnt = dalloc<int4>(P, range.size());
  P.cl_off = dalloc<int32_t>(P, nc + 1);
  DM_CUDA(cudaMemcpyAsync(drange, range.data(), range.size() * sizeof(int2), cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaMemcpyAsync(P.cl_off, off.data(), off.size() * sizeof(int32_t), cudaMemcpyHostToDevice, s));
  k_clusters<false><<<(unsigned)range.size(), 256, 0, s>>>(drange, P.tets_s, P.tet_geo, dcnt, nullptr, nullptr, nullptr,
                                                           nullptr, nullptr, nullptr, nullptr);
  DM_LAUNCH("k_clusters");
  std::vector<int4> cnt(range.size()), pos(range.size());
  DM_CUDA(cudaMemcpyAsync(cnt.data(), dcnt, cnt.size() * sizeof(int4), cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaStreamSynchronize(s));
  int64_t nv = 0, ne = 0, nf = 0, nb = 0;
  for (size_t i = 0; i < cnt.size(); i++) {
    if (nf > INT32_MAX - CL_F || ne > INT32_MAX - CL_E) fail(DEMAG_ERR_UNSUPPORTED, "mesh too large for near_mode 0");
    pos[i] = make_int4((int)nv, (int)ne, (int)nf, (int)nb);
    nv += cnt[i].x;
    ne += cnt[i].y;
    nf += cnt[i].z;
    nb += cnt[i].w;
  }
  P.n_cl_v = nv;
  P.n_cl_e = ne;
  P.n_cl_f = nf;
  P.n_cl_b = nb;
  P.cl_cnt = dcnt;
  P.cl_pos = dalloc<int4>(P, pos.size());
  P.cl_vnode = dalloc<int32_t>(P, nv);
  P.cl_edge = dalloc<uint32_t>(P, ne);
  P.cl_elen = dalloc<double>(P, ne);
  P.cl_frec = dalloc<double>(P, FACE_REC * nf);
  P.cl_fidx = dalloc<uint2>(P, nf);
  P.cl_ftet = dalloc<int2>(P, nf);
  DM_CUDA(cudaMemcpyAsync(P.cl_pos, pos.data(), pos.size() * sizeof(int4), cudaMemcpyHostToDevice, s));
  k_clusters<true><<<(unsigned)range.size(), 256, 0, s>>>(drange, P.tets_s, P.tet_geo, dcnt, P.cl_pos, P.cl_vnode,
                                                          P.cl_edge, P.cl_elen, P.cl_frec, P.cl_fidx, P.cl_ftet);
  DM_LAUNCH("k_clusters");
  if (nT) {
    int64_t* dc = dalloc<int64_t>(P, nT);
    k_cluster_lists<false><<<(unsigned)nT, 128, 0, s>>>(P.p2p_targets, P.p2p_off, P.p2p_src, P.cl_off, dc, nullptr,
                                                        nullptr);
    DM_LAUNCH("k_cluster_lists");
    std::vector<int64_t> hc(nT), po(nT + 1, 0);
    DM_CUDA(cudaMemcpyAsync(hc.data(), dc, nT * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    DM_CUDA(cudaStreamSynchronize(s));
    dfree(P, dc);
    for (int64_t i = 0; i < nT; i++) po[i + 1] = po[i] + hc[i];
    P.n_pc = po[nT];
    P.pc_off = dalloc<int64_t>(P, nT + 1);
    P.pc_src = dalloc<int32_t>(P, std::max<int64_t>(P.n_pc, 1));
    DM_CUDA(cudaMemcpyAsync(P.pc_off, po.data(), po.size() * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    k_cluster_lists<true><<<(unsigned)nT, 32, 0, s>>>(P.p2p_targets, P.p2p_off, P.p2p_src, P.cl_off, nullptr, P.pc_off,
                                                      P.pc_src);
    DM_LAUNCH("k_cluster_lists");
    const std::vector<int4> blk = face_blocks(P, hc);
    P.n_pc_blk = (int64_t)blk.size();
    P.pc_blk = dalloc<int4>(P, std::max<size_t>(blk.size(), 1));
    DM_CUDA(cudaMemcpyAsync(P.pc_blk, blk.data(), blk.size() * sizeof(int4), cudaMemcpyHostToDevice, s));
    DM_CUDA(cudaStreamSynchronize(s));  // the host lists end here
  }
  DM_CUDA(cudaStreamSynchronize(s));
  dfree(P, drange);
}

// ---------------------------------------------------------------------------
// per face and state of a slice of FS states, over 4 pi, in the face's frame,
// signs for the record's n: half the jump of dM/dn (half of dM/dn on a boundary
// face), [face][3][FS]; for the boundary faces M_0, G_t, G_m, [face][9][FS]
// ---------------------------------------------------------------------------
namespace {

template <int FS>
__global__ void k_face_state(int64_t nf, const int2* __restrict__ ftet, const uint2* __restrict__ fidx,
                             const double* __restrict__ frec, const int32_t* __restrict__ tets_s,
                             const double* __restrict__ grad, const double* __restrict__ Ms, int B, int b0, double* D) {
  const int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t f = it / FS;
  if (f >= nf) return;
  const int v = (int)(it - f * FS), b = b0 + v;
  const double* R = frec + FACE_REC * f;
  double j[3] = {0.0, 0.0, 0.0};
  if (b < B) {
    const int2 t = ftet[f];
#pragma unroll
    for (int side = 0; side < 2; side++) {
      const int64_t e = side ? t.y : t.x;
      if (e < 0) continue;
      double dn[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int64_t node = tets_s[4 * e + k];
        const double* g = grad + 12 * e + 3 * k;
        const double gn = g[0] * R[0] + g[1] * R[1] + g[2] * R[2];
#pragma unroll
        for (int c = 0; c < 3; c++) dn[c] += Ms[(node * 3 + c) * B + b] * gn;
      }
#pragma unroll
      for (int c = 0; c < 3; c++) j[c] += side ? -dn[c] : dn[c];
    }
  }
  const double sg = (fidx[f].x >> 31 ? -0.5 : 0.5) / (4.0 * M_PI);
#pragma unroll
  for (int x = 0; x < 3; x++) {  // frame (t, m, n) = records 3, 6, 0
    const double* e = R + (x == 0 ? 3 : x == 1 ? 6 : 0);
    D[(3 * f + x) * FS + v] = sg * (j[0] * e[0] + j[1] * e[1] + j[2] * e[2]);
  }
}

template <int FS>
__global__ void k_face_affine(const int4* __restrict__ cnt, const int4* __restrict__ pos,
                              const int32_t* __restrict__ vnode, const double* __restrict__ frec,
                              const uint2* __restrict__ fidx, const double* __restrict__ Ms, int B, int b0, double* S) {
  const int64_t c = blockIdx.x;
  const int4 n = cnt[c], o = pos[c];
  for (int q = threadIdx.x; q < n.w * FS; q += blockDim.x) {
    const int f = q / FS, v = q - f * FS, b = b0 + v;
    const uint32_t x = fidx[o.z + f].x;
    const double* R = frec + FACE_REC * (int64_t)(o.z + f);
    double M0[3] = {0.0, 0.0, 0.0}, Gt[3] = {0.0, 0.0, 0.0}, Gm[3] = {0.0, 0.0, 0.0};
    if (b < B) {
      const double il = R[14], ih = -1.0 / (R[9] * il);  // vertex 2 lies at (R[15], -height)
#pragma unroll
      for (int a = 0; a < 3; a++) {
        double m[3];
#pragma unroll
        for (int k = 0; k < 3; k++) m[k] = Ms[((int64_t)vnode[o.x + ((x >> (8 * k)) & 255u)] * 3 + a) * B + b];
        M0[a] = m[0];
        Gt[a] = (m[1] - m[0]) * il;
        Gm[a] = ((m[2] - m[0]) - Gt[a] * R[15]) * ih;
      }
    }
    const double sg = (x >> 31 ? -1.0 : 1.0) / (4.0 * M_PI);
    double* s = S + (9ll * (o.w + f)) * FS + v;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const double* e = R + (k == 0 ? 3 : k == 1 ? 6 : 0);
      s[k * FS] = sg * (M0[0] * e[0] + M0[1] * e[1] + M0[2] * e[2]);
      s[(3 + k) * FS] = sg * (Gt[0] * e[0] + Gt[1] * e[1] + Gt[2] * e[2]);
      s[(6 + k) * FS] = sg * (Gm[0] * e[0] + Gm[1] * e[1] + Gm[2] * e[2]);
    }
  }
}

// ---------------------------------------------------------------------------
// The near field: one block per entry of face_blocks (up to 16 nodes of a target
// leaf) and FS states.  Batches of whole clusters (as many as fit the
// shared-memory arrays) are staged; thread = (target i, subset of the entities),
// so a warp reads one or two records per step (broadcast) for 16 targets, and
// keeps its target's FS sums over all batches: distances, barrier, edge
// logarithms, barrier, faces.  The per-state values of a face are read once per
// block, so they come straight from global memory, and any FS leaves room for two
// blocks per SM.  The subsets are added in order at the end: no atomics, the
// result does not depend on timing.  FP64 arithmetic is the bound (2 FMA per
// clock and SM), so records are read from shared memory instead of being
// recomputed.  Near-field stage, against the tet-wise kernels before (4 sqrt, 6
// log1p, 4 atan2 and 6 divisions per pair): 3,072-tet cube, leaf 32, one state 5.2
// -> 0.77 ms; 16k-tet ball, leaf 128, 3 states 196 -> 17.8 ms, 16 states 26.8 ms.
// With face charges in the sum instead (less accurate on flattened tets, two
// divisions per boundary face) 0.91, 18.8 and 27.0 ms.
// ---------------------------------------------------------------------------
constexpr int PF_THREADS = 256, PF_BATCH = 32;
constexpr int PF_V = CL_V, PF_E = CL_E, PF_F = CL_F;  // capacities of a batch: any one cluster fits

constexpr size_t PF_SMEM = sizeof(double) * ((size_t)(PF_V + PF_E) * PF_G + 3 * PF_V + PF_E + FACE_REC * PF_F) +
                           sizeof(uint2) * PF_F + sizeof(int2) * PF_F + sizeof(uint32_t) * PF_E;
static_assert(PF_SMEM <= 227 * 1024 && PF_SMEM >= sizeof(double) * PF_THREADS * P2P_SLICE, "arrays, final sums");

// s[v] += f sum_k x_k q[k][v]
template <int FS>
__device__ __forceinline__ void add(double (&s)[FS], double f, const double (&x)[3], const double* __restrict__ q) {
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const double w = f * x[k];
    double y[FS];
    load_q<double, FS>(q + k * FS, y);
#pragma unroll
    for (int v = 0; v < FS; v++) s[v] += w * y[v];
  }
}

template <int FS>
__global__ void __launch_bounds__(PF_THREADS, 2) k_p2p_faces(
    const int4* __restrict__ blk, const int64_t* __restrict__ pc_off, const int32_t* __restrict__ pc_src,
    const double* __restrict__ nodes_s, const int4* __restrict__ cnt,
    const int4* __restrict__ pos, const int32_t* __restrict__ vnode, const uint32_t* __restrict__ edge,
    const double* __restrict__ elen, const double* __restrict__ frec, const uint2* __restrict__ fidx,
    const double* __restrict__ D, const double* __restrict__ S, int B, int b0, double* u_s) {
  extern __shared__ __align__(16) double pf[];
  double* sR = pf;                          // [vertex][target]
  double* sL = sR + PF_V * PF_G;            // [edge][target]
  double* sV = sL + PF_E * PF_G;            // [vertex][3]
  double* sEl = sV + 3 * PF_V;              // edge lengths
  double* sF = sEl + PF_E;                  // [face][FACE_REC], boundary faces of all clusters first
  uint2* sFi = (uint2*)(sF + FACE_REC * PF_F);
  int2* sId = (int2*)(sFi + PF_F);          // face's rows of D and (boundary faces) S
  uint32_t* sE = (uint32_t*)(sId + PF_F);
  __shared__ int4 bc[PF_BATCH], bp[PF_BATCH], bb[PF_BATCH];  // per cluster: counts, positions, bases in the batch
  __shared__ int4 tot;                                       // of the batch: vertices, edges, faces, boundary faces
  __shared__ int nb;
  const int tid = threadIdx.x, lane = tid & 31;
  const int4 bk = blk[blockIdx.x];
  const int64_t ti = bk.x;
  const int i0 = bk.y, nt = bk.z;
  int lg = 0;
  while ((1 << lg) < nt) lg++;
  const int G = 1 << lg, i = tid & (G - 1), sub = tid >> lg, nsub = PF_THREADS >> lg;
  const double* rp = nodes_s + 3ll * (i0 + min(i, nt - 1));
  const double rx = rp[0], ry = rp[1], rz = rp[2];
  double acc[FS];
#pragma unroll
  for (int v = 0; v < FS; v++) acc[v] = 0.0;
  const int64_t q1 = pc_off[ti + 1];
  for (int64_t q = pc_off[ti]; q < q1;) {
    __syncthreads();  // the previous batch is no longer read
    if (tid < 32) {   // the next clusters, as many as fit
      int4 n = make_int4(0, 0, 0, 0), p = n, e = n;
      const bool on = q + lane < q1;
      if (on) {
        const int32_t c = pc_src[q + lane];
        n = cnt[c];
        p = pos[c];
      }
      e = n;  // inclusive sums
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, e.x, d), b = __shfl_up_sync(0xffffffffu, e.y, d),
                  c = __shfl_up_sync(0xffffffffu, e.z, d), w = __shfl_up_sync(0xffffffffu, e.w, d);
        if (lane >= d) {
          e.x += a;
          e.y += b;
          e.z += c;
          e.w += w;
        }
      }
      const uint32_t fit = __ballot_sync(0xffffffffu, on && e.x <= PF_V && e.y <= PF_E && e.z <= PF_F);
      const int k = __popc(fit);  // a prefix: the sums ascend
      if (lane < k) {
        bc[lane] = n;
        bp[lane] = p;
        bb[lane] = make_int4(e.x - n.x, e.y - n.y, (e.z - e.w) - (n.z - n.w), e.w - n.w);  // z: interior faces
      }
      if (lane == k - 1) tot = e;
      if (lane == 0) nb = k;
    }
    __syncthreads();
    const int k1 = nb, nv = tot.x, ne = tot.y, nf = tot.z, nbf = tot.w;
    q += k1;
    for (int k = 0; k < k1; k++) {
      const int4 n = bc[k], p = bp[k], b = bb[k];
      for (int t = tid; t < n.x; t += PF_THREADS) {
        const double* x = nodes_s + 3ll * vnode[p.x + t];
        double* d = sV + 3 * (b.x + t);
        d[0] = x[0];
        d[1] = x[1];
        d[2] = x[2];
      }
      for (int t = tid; t < n.y; t += PF_THREADS) {
        sE[b.y + t] = edge[p.y + t] + (uint32_t)b.x * 0x10001u;
        sEl[b.y + t] = elen[p.y + t];
      }
      // face t of the cluster: boundary faces from b.w, interior ones behind all boundary faces
      auto slot = [&](int t) { return t < n.w ? b.w + t : nbf + b.z + t - n.w; };
      for (int t = tid; t < n.z; t += PF_THREADS) {
        const uint2 x = fidx[p.z + t];
        sFi[slot(t)] = make_uint2((x.x & 0xFFFFFFu) + (uint32_t)b.x * 0x010101u, x.y + (uint32_t)b.y * ((1u << 18) | (1u << 9) | 1u));
        sId[slot(t)] = make_int2(p.z + t, p.w + t);
      }
      for (int t = tid; t < n.z * (FACE_REC / 2); t += PF_THREADS) {
        const int f = t / (FACE_REC / 2), c = t - f * (FACE_REC / 2);
        ((double2*)(sF + FACE_REC * slot(f)))[c] = ((const double2*)(frec + FACE_REC * (int64_t)(p.z + f)))[c];
      }
    }
    __syncthreads();
    for (int t = sub; t < nv; t += nsub) {
      const double x = sV[3 * t] - rx, y = sV[3 * t + 1] - ry, z = sV[3 * t + 2] - rz;
      sR[t * PF_G + i] = sqrt(x * x + y * y + z * z);
    }
    __syncthreads();
    for (int t = sub; t < ne; t += nsub) {
      const uint32_t e = sE[t];
      const double L = sEl[t], dd = sR[(e & 0xFFFFu) * PF_G + i] + sR[(e >> 16) * PF_G + i] - L;
      sL[t * PF_G + i] = dd > 0 ? log1p(2.0 * L / dd) : 0.0;
    }
    __syncthreads();
    double part[FS];  // this batch's sums
#pragma unroll
    for (int v = 0; v < FS; v++) part[v] = 0.0;
    for (int t = sub; t < nf; t += nsub) {
      const uint2 ix = sFi[t];
      const double* F = sF + FACE_REC * t;
      const int2 id = sId[t];
      double a[3][3], R[3], lam[3], longest = 0.0, len0 = 0.0;
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const int vi = (ix.x >> (8 * k)) & 255u, ei = (ix.y >> (9 * k)) & 511u;
        a[k][0] = sV[3 * vi] - rx;
        a[k][1] = sV[3 * vi + 1] - ry;
        a[k][2] = sV[3 * vi + 2] - rz;
        R[k] = sR[vi * PF_G + i];
        lam[k] = sL[ei * PF_G + i];
        if (k == 0) len0 = sEl[ei];
        longest = fmax(longest, sEl[ei]);
      }
      const double h = -(F[0] * a[0][0] + F[1] * a[0][1] + F[2] * a[0][2]);
      if (fabs(h) <= 1e-13 * longest) continue;  // r in the plane of F
      const double d01 = a[0][0] * a[1][0] + a[0][1] * a[1][1] + a[0][2] * a[1][2];
      const double d12 = a[1][0] * a[2][0] + a[1][1] * a[2][1] + a[1][2] * a[2][2];
      const double d20 = a[2][0] * a[0][0] + a[2][1] * a[0][1] + a[2][2] * a[0][2];
      const double den = R[0] * R[1] * R[2] + d01 * R[2] + d12 * R[0] + d20 * R[1];
      const double Om = -2.0 * atan2(h * F[9], den);  // 2 atan2(triple product, den), triple product = -h 2A
      const double c1 = F[10], d1 = F[11], c2 = F[12], d2 = F[13];
      const double A[3] = {-(c1 * lam[1] + c2 * lam[2]), -(lam[0] + d1 * lam[1] + d2 * lam[2]), Om};
      add<FS>(part, h * h, A, D + 3ll * FS * id.x);
      if (t < nbf) {
        const double x = -(F[3] * a[0][0] + F[4] * a[0][1] + F[5] * a[0][2]);
        const double y = -(F[6] * a[0][0] + F[7] * a[0][1] + F[8] * a[0][2]);
        const double w0 = -y * lam[0], w1 = (c1 * (len0 - x) - d1 * y) * lam[1], w2 = -(c2 * x + d2 * y) * lam[2];
        const double dR0 = R[1] - R[0], dR1 = R[2] - R[1], dR2 = R[0] - R[2];
        const double z = c1 * d1 * dR1 + c2 * d2 * dR2, I = w0 + w1 + w2 + h * Om;
        const double Stt = I - (w1 * c1 * c1 + w2 * c2 * c2) - z;
        const double Smm = I - (w0 + w1 * d1 * d1 + w2 * d2 * d2) + z;
        const double Stm = -(w1 * c1 * d1 + w2 * c2 * d2) -
                           0.5 * (dR0 + (d1 * d1 - c1 * c1) * dR1 + (d2 * d2 - c2 * c2) * dR2);
        const double kt[3] = {x * A[0] + 0.5 * Stt, x * A[1] + 0.5 * Stm, x * Om - 0.5 * h * A[0]};
        const double km[3] = {y * A[0] + 0.5 * Stm, y * A[1] + 0.5 * Smm, y * Om - 0.5 * h * A[1]};
        const double* q = S + 9ll * FS * id.y;
        add<FS>(part, h, A, q);
        add<FS>(part, h, kt, q + 3 * FS);
        add<FS>(part, h, km, q + 6 * FS);
      }
    }
#pragma unroll
    for (int v = 0; v < FS; v++) acc[v] += part[v];
  }
  __syncthreads();
  double* red = pf;  // [sub][target][FS]
#pragma unroll
  for (int v = 0; v < FS; v++) red[tid * FS + v] = acc[v];
  __syncthreads();
  for (int t = tid; t < nt * FS; t += PF_THREADS) {
    const int ii = t / FS, v = t - ii * FS;
    if (b0 + v >= B) continue;
    double sum = 0.0;
    for (int k = 0; k < nsub; k++) sum += red[((k << lg) + ii) * FS + v];
    u_s[(int64_t)(i0 + ii) * B + b0 + v] += sum;
  }
}

template <int FS>
void launch_slice(Plan& P, const double* Ms, double* state, int B, int b0, double* u_s, cudaStream_t s) {
  double *D = state, *S = state + 3 * P.n_cl_f * FS;
  k_face_state<FS><<<nblk(P.n_cl_f * FS, 256), 256, 0, s>>>(P.n_cl_f, P.cl_ftet, P.cl_fidx, P.cl_frec, P.tets_s,
                                                            P.tet_grad, Ms, B, b0, D);
  DM_LAUNCH("k_face_state");
  k_face_affine<FS><<<(unsigned)P.n_clusters, 128, 0, s>>>(P.cl_cnt, P.cl_pos, P.cl_vnode, P.cl_frec, P.cl_fidx, Ms, B,
                                                           b0, S);
  DM_LAUNCH("k_face_affine");
  smem_opt_in((const void*)k_p2p_faces<FS>, PF_SMEM);
  k_p2p_faces<FS><<<(unsigned)P.n_pc_blk, PF_THREADS, PF_SMEM, s>>>(P.pc_blk, P.pc_off, P.pc_src, P.nodes_s, P.cl_cnt,
                                                                    P.cl_pos, P.cl_vnode, P.cl_edge, P.cl_elen,
                                                                    P.cl_frec, P.cl_fidx, D, S, B, b0, u_s);
  DM_LAUNCH("k_p2p_faces");
}

}  // namespace

size_t face_state_doubles(const Plan& P, int slice) { return (size_t)slice * (size_t)(3 * P.n_cl_f + 9 * P.n_cl_b); }

int launch_p2p_fp64(Plan& P, const double* Ms, double* state, int slice, int B, double* u_s, cudaStream_t s) {
  if (P.n_pc_blk == 0 || P.n_clusters == 0) return 0;
  int n = 0;
  for (int b0 = 0; b0 < B; n += 3) {
    int fs = 1;  // the smallest slice that takes what is left, within what the state buffer holds
    while (fs < B - b0 && fs < slice) fs *= 2;
    switch (fs) {
      case 1: launch_slice<1>(P, Ms, state, B, b0, u_s, s); break;
      case 2: launch_slice<2>(P, Ms, state, B, b0, u_s, s); break;
      case 4: launch_slice<4>(P, Ms, state, B, b0, u_s, s); break;
      case 8: launch_slice<8>(P, Ms, state, B, b0, u_s, s); break;
      default: launch_slice<16>(P, Ms, state, B, b0, u_s, s); break;
    }
    b0 += fs;
  }
  return n;
}

}  // namespace demag
