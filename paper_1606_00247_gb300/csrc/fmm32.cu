// fmm32.cu -- the mixed-precision evaluation driver, its input and output
// kernels and the FP32 gradient operator.
//
// The far field (far.cu) runs in FP32 on per-level scaled expansions.  The near
// field is the precomputed FP64 coefficient set W rounded to FP32 (near.cu), or
// the FP64 on-the-fly P2P when near_mode = 0.  u is accumulated in FP32 and the
// mass-lumped H is formed in FP32 by a sparse operator (below).
#include <algorithm>
#include <array>
#include <cmath>

#include "common.cuh"

namespace demag {

static inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

namespace {

// M (state, original node, component) -> Ms (sorted node, component, state):
// thread per (sorted node, state), the states of a node side by side, so the
// stores coalesce over the states; each thread reads the 24 contiguous bytes of
// its state's (node, x y z) row.  (A block of 128 threads per node leaves all but B
// of them idle: 72 -> 11 us for 126k nodes and two states.)
__global__ void __launch_bounds__(256) k_gather_M32(int64_t nn, int B, const int32_t* __restrict__ perm,
                                                    const double* __restrict__ M, float* Ms, double* Ms64) {
  const int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (it >= nn * B) return;
  const int64_t i = it / B;
  const int b = (int)(it - i * B);
  const double* src = M + ((int64_t)b * nn + perm[i]) * 3;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const double v = src[c];
    Ms[(i * 3 + c) * B + b] = (float)v;
    if (Ms64) Ms64[(i * 3 + c) * B + b] = v;
  }
}

// From GATHER_WIDE states on: block per (sorted node, 128 states), thread = state
// (no division per thread).  Against the kernel above, 36k nodes: 48 states 32 / 30 us,
// 64 to 160 states equal (37 us at 64), 256 states 110 / 113; 87k nodes, 256 states 309 /
// 399.
constexpr int GATHER_WIDE = 64;
__global__ void __launch_bounds__(128) k_gather_M32_wide(int64_t nn, int B, const int32_t* __restrict__ perm,
                                                         const double* __restrict__ M, float* Ms, double* Ms64) {
  const int64_t i = blockIdx.x;
  const int b = blockIdx.y * 128 + threadIdx.x;
  if (b >= B) return;
  const double* src = M + ((int64_t)b * nn + perm[i]) * 3;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const double v = src[c];
    Ms[(i * 3 + c) * B + b] = (float)v;
    if (Ms64) Ms64[(i * 3 + c) * B + b] = v;
  }
}

// u and the mass-lumped H of the mixed path, in the caller's layout: tiles of
// 32 original nodes x 32 states; reads coalesce over states, the transposed
// tile is written coalesced over nodes
__global__ void __launch_bounds__(256) k_out32(int64_t nn, int B, const int32_t* __restrict__ iperm,
                                               const int64_t* __restrict__ hoff, const int32_t* __restrict__ hcol,
                                               const float4* __restrict__ hw, const float* __restrict__ u32,
                                               double* u_out, double* H_out) {
  __shared__ float su[32][33];
  __shared__ float sh[32][97];
  const int64_t g0 = (int64_t)blockIdx.x * 32;
  const int b0 = blockIdx.y * 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int b = b0 + lane;
  for (int r = w; r < 32; r += 8) {
    const int64_t g = g0 + r;
    float uu = 0.f, hx = 0.f, hy = 0.f, hz = 0.f;
    if (g < nn && b < B) {
      const int64_t i = iperm[g];
      uu = u32[i * B + b];
      if (H_out)
        for (int64_t e = hoff[i], e1 = hoff[i + 1]; e < e1; e++) {
          const float4 wv = hw[e];
          const float uj = u32[(int64_t)hcol[e] * B + b];
          hx = fmaf(wv.x, uj, hx);
          hy = fmaf(wv.y, uj, hy);
          hz = fmaf(wv.z, uj, hz);
        }
    }
    su[lane][r] = uu;
    sh[lane][3 * r] = hx;
    sh[lane][3 * r + 1] = hy;
    sh[lane][3 * r + 2] = hz;
  }
  __syncthreads();
  for (int q = threadIdx.x; q < 32 * 32; q += blockDim.x) {
    const int bl = q >> 5, gl = q & 31;
    if (b0 + bl < B && g0 + gl < nn) u_out[(int64_t)(b0 + bl) * nn + g0 + gl] = (double)su[bl][gl];
  }
  if (H_out)
    for (int q = threadIdx.x; q < 32 * 96; q += blockDim.x) {
      const int bl = q / 96, rr = q - bl * 96;
      if (b0 + bl < B && g0 + rr / 3 < nn) H_out[((int64_t)(b0 + bl) * nn + g0) * 3 + rr] = (double)sh[bl][rr];
    }
}

// the same for a few states (OUT_SMALL_BATCH): thread per (state, original node),
// consecutive threads on consecutive nodes, so the stores of u and H coalesce.
// (The 32-state tiles above are mostly empty then: 64 -> 29 us for 126k
// nodes and two states.)
constexpr int OUT_SMALL_BATCH = 8;
__global__ void __launch_bounds__(256) k_out32_small(int64_t nn, int B, const int32_t* __restrict__ iperm,
                                                     const int64_t* __restrict__ hoff, const int32_t* __restrict__ hcol,
                                                     const float4* __restrict__ hw, const float* __restrict__ u32,
                                                     double* u_out, double* H_out) {
  const int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (it >= nn * B) return;
  const int b = (int)(it / nn);
  const int64_t i = iperm[it - (int64_t)b * nn];
  u_out[it] = (double)u32[i * B + b];
  if (!H_out) return;
  float hx = 0.f, hy = 0.f, hz = 0.f;
#pragma unroll 4
  for (int64_t e = hoff[i], e1 = hoff[i + 1]; e < e1; e++) {
    const float4 wv = hw[e];
    const float uj = u32[(int64_t)hcol[e] * B + b];
    hx = fmaf(wv.x, uj, hx);
    hy = fmaf(wv.y, uj, hy);
    hz = fmaf(wv.z, uj, hz);
  }
  H_out[3 * it] = (double)hx;
  H_out[3 * it + 1] = (double)hy;
  H_out[3 * it + 2] = (double)hz;
}

__global__ void k_u32_to_64(int64_t n, const float* __restrict__ a, double* b) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) b[i] = (double)a[i];
}

}  // namespace

// mass-lumped gradient (Sec. 4.1) as a sparse FP32 operator on u: row i holds,
// for every node j sharing a tet with i, -(1/V_i) sum_{t ni i, j} vol_t grad lambda_j^t
void build_gradient_operator(Plan& P) {
  cudaStream_t s = P.stream;
  const int64_t nn = P.nn, nt = P.nt;
  std::vector<int32_t> tets(4 * nt), nt_tet(4 * nt), perm(nn);
  std::vector<double> grad(12 * nt), vol(nt);
  std::vector<int64_t> nt_off(nn + 1);
  DM_CUDA(cudaMemcpyAsync(tets.data(), P.tets_s, sizeof(int32_t) * 4 * nt, cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(nt_tet.data(), P.nt_tet, sizeof(int32_t) * 4 * nt, cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(perm.data(), P.node_perm, sizeof(int32_t) * nn, cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(grad.data(), P.tet_grad, sizeof(double) * 12 * nt, cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(vol.data(), P.tet_vol, sizeof(double) * nt, cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaMemcpyAsync(nt_off.data(), P.nt_off, sizeof(int64_t) * (nn + 1), cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaStreamSynchronize(s));
  std::vector<int64_t> off(nn + 1, 0);
  std::vector<int32_t> col;
  std::vector<float4> w;
  std::vector<std::pair<int32_t, std::array<double, 3>>> row;
  for (int64_t i = 0; i < nn; i++) {
    row.clear();
    double V = 0;
    for (int64_t e = nt_off[i]; e < nt_off[i + 1]; e++) {
      const int64_t t = nt_tet[e];
      V += vol[t];
      for (int k = 0; k < 4; k++) {
        const int32_t j = tets[4 * t + k];
        auto it = std::find_if(row.begin(), row.end(), [&](const auto& x) { return x.first == j; });
        if (it == row.end()) {
          row.push_back({j, {0.0, 0.0, 0.0}});
          it = row.end() - 1;
        }
        for (int d = 0; d < 3; d++) it->second[d] += vol[t] * grad[12 * t + 3 * k + d];
      }
    }
    std::sort(row.begin(), row.end(), [](const auto& x, const auto& y) { return x.first < y.first; });
    if (V > 0)
      for (auto& x : row) {
        col.push_back(x.first);
        w.push_back(make_float4((float)(-x.second[0] / V), (float)(-x.second[1] / V), (float)(-x.second[2] / V), 0.f));
      }
    off[i + 1] = (int64_t)col.size();
  }
  std::vector<int32_t> iperm(nn);
  for (int64_t i = 0; i < nn; i++) iperm[perm[i]] = (int32_t)i;
  P.hg_off = dalloc<int64_t>(P, nn + 1);
  P.hg_col = dalloc<int32_t>(P, std::max<size_t>(col.size(), 1));
  P.hg_w = dalloc<float4>(P, std::max<size_t>(w.size(), 1));
  P.node_iperm = dalloc<int32_t>(P, nn);
  DM_CUDA(cudaMemcpyAsync(P.hg_off, off.data(), sizeof(int64_t) * (nn + 1), cudaMemcpyHostToDevice, s));
  if (!col.empty()) {
    DM_CUDA(cudaMemcpyAsync(P.hg_col, col.data(), sizeof(int32_t) * col.size(), cudaMemcpyHostToDevice, s));
    DM_CUDA(cudaMemcpyAsync(P.hg_w, w.data(), sizeof(float4) * w.size(), cudaMemcpyHostToDevice, s));
  }
  DM_CUDA(cudaMemcpyAsync(P.node_iperm, iperm.data(), sizeof(int32_t) * nn, cudaMemcpyHostToDevice, s));
  DM_CUDA(cudaStreamSynchronize(s));
}

void eval_mixed(Plan& P, const double* M, int B, double* u, double* H, cudaStream_t s) {
  eval_mixed_ws(P, workspace(P, B), M, B, u, H, s, true);
}

void eval_mixed_ws(Plan& P, Workspace& W, const double* M, int B, double* u, double* H, cudaStream_t s,
                   bool profile_ok) {
  const double* Md;
  double *ud, *Hd;
  const bool dev = eval_io_begin(P, W, M, B, u, H, &Md, &ud, &Hd, s);
  const bool otf = P.opt.near_mode == 0;
  const int nq = P.nq, nl = P.nl;
  StageClock clk(P, s, profile_ok);
  clk.begin(DEMAG_STAGE_GATHER);
  if (B >= GATHER_WIDE)
    k_gather_M32_wide<<<dim3((unsigned)P.nn, (unsigned)((B + 127) / 128)), 128, 0, s>>>(P.nn, B, P.node_perm, Md,
                                                                                        W.Ms32, otf ? W.Ms : nullptr);
  else
    k_gather_M32<<<nblk(P.nn * B, 256), 256, 0, s>>>(P.nn, B, P.node_perm, Md, W.Ms32, otf ? W.Ms : nullptr);
  DM_LAUNCH("k_gather_M32");
  clk.launched();
  clk.end();
  clk.begin(DEMAG_STAGE_P2M);
  DM_CUDA(cudaMemsetAsync(W.Q32, 0, sizeof(float) * P.ncells * nq * B, s));
  clk.launched(launch_p2m<float>(P, B, W.Ms32, W.Q32, s));
  clk.end();
  clk.begin(DEMAG_STAGE_M2M);
  clk.launched(launch_m2m<float>(P, B, W.Q32, s));
  clk.end();
  clk.begin(DEMAG_STAGE_M2L);
  DM_CUDA(cudaMemsetAsync(W.L32, 0, sizeof(float) * P.ncells * nl * B, s));
  const bool tc_prec = P.opt.precision == DEMAG_MIXED_TF32 || P.opt.precision == DEMAG_MIXED_BF16X3 ||
                       P.opt.precision == DEMAG_MIXED_BF16X6;
  if (P.h_m2l_targets.empty()) {
  } else if (tc_prec && B > m2l_table_batch(P) && launch_m2l_tc(P, B, W.Q32, W.QP, W.L32, W.err, s)) {
    clk.launched(2);
  } else if ((!tc_prec || P.opt.m2l_table_batch >= 0) && launch_m2l_tab<float>(P, B, W.Q32, W.L32, s)) {
    clk.launched();
  } else {
    launch_m2l_rows<float>(P, B, W.Q32, W.L32, s);
    clk.launched();
  }
  clk.end();
  clk.begin(DEMAG_STAGE_L2L);
  clk.launched(launch_l2l<float>(P, B, W.L32, s));
  clk.end();
  clk.begin(DEMAG_STAGE_L2P);
  clk.launched(launch_l2p<float>(P, B, W.L32, W.u32, s));
  clk.end();
  if (otf) {
    k_u32_to_64<<<nblk(P.nn * B, 256), 256, 0, s>>>(P.nn * B, W.u32, W.u_s);
    DM_LAUNCH("k_u32_to_64");
    near_field_fp64(P, W, B, clk, s);
  } else {
    clk.begin(DEMAG_STAGE_P2P);
    if (P.nf_W) {
      clk.launched(launch_near_tc(P, W.Ms32, W.MP, B, W.u32, W.err, s));
    } else if (!P.h_p2p_targets.empty()) {
      launch_near_apply32(P, W.Ms32, B, W.u32, W.err, s);
      clk.launched();
    }
    clk.end();
  }
  clk.begin(DEMAG_STAGE_H);
  if (otf) {
    launch_lumped_H_out(P, B, W.u_s, ud, Hd, s);  // FP64 near field: u in FP64
  } else if (B <= OUT_SMALL_BATCH) {
    k_out32_small<<<nblk(P.nn * B, 256), 256, 0, s>>>(P.nn, B, P.node_iperm, P.hg_off, P.hg_col, P.hg_w, W.u32, ud, Hd);
    DM_LAUNCH("k_out32_small");
  } else {
    k_out32<<<dim3((unsigned)((P.nn + 31) / 32), (unsigned)((B + 31) / 32)), 256, 0, s>>>(
        P.nn, B, P.node_iperm, P.hg_off, P.hg_col, P.hg_w, W.u32, ud, Hd);
    DM_LAUNCH("k_out32");
  }
  clk.launched();
  clk.end();
  clk.finish();
  eval_io_end(P, W, dev, B, u, H, s);
}

}  // namespace demag
