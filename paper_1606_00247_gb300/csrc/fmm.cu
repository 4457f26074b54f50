// fmm.cu -- the FP64 evaluation driver, the lumped H (Sec. 4.1), the workspace
// and the input and output layouts.  The far field is far.cu and m2l32.cu, the
// near field p2p.cu and near.cu.  All arrays keep the state index innermost:
// X[item][coefficient][state].
#include "common.cuh"

namespace demag {

static inline int nblk(int64_t n, int t) { return (int)((n + t - 1) / t > 0 ? (n + t - 1) / t : 1); }

// ---------------------------------------------------------------------------
// input / output layout
// ---------------------------------------------------------------------------
// Ms[(i*3+c)*B + b] = M[(b*nn + perm[i])*3 + c]
// thread per (sorted node, state), the states of a node side by side: stores coalesce over states
__global__ void __launch_bounds__(256) k_gather_M(int64_t nn, int B, const int32_t* __restrict__ perm,
                                                  const double* __restrict__ M, double* Ms) {
  const int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (it >= nn * B) return;
  const int64_t i = it / B;
  const int b = (int)(it - i * B);
  const double* src = M + ((int64_t)b * nn + perm[i]) * 3;
#pragma unroll
  for (int c = 0; c < 3; c++) Ms[(i * 3 + c) * B + b] = src[c];
}

// ---------------------------------------------------------------------------
// mass-lumped H (Sec. 4.1) and the output layout
//   H_i = -sum_{t ni i} |t| grad u_h|_t / sum_{t ni i} |t|
// Thread = (node, state, one of LH_LANES lanes over the node's tets): the states
// of a node are neighbours, so the loads of u coalesce; the lanes' sums are added
// by a fixed shuffle tree.  (One thread per node walked ~25 tets and all states in
// turn: 79 -> 70 us for 36k nodes and one state, 780 -> 120 us for 5k nodes
// and 16.)
// ---------------------------------------------------------------------------
constexpr int LH_LANES = 8;
__global__ void __launch_bounds__(256) k_lumped_H_out(int64_t nn, int B, const int32_t* __restrict__ perm,
                                                      const int64_t* __restrict__ nt_off,
                                                      const int32_t* __restrict__ nt_tet,
                                                      const int32_t* __restrict__ tets_s,
                                                      const double* __restrict__ grad, const double* __restrict__ vol,
                                                      const double* __restrict__ u_s, double* u_out, double* H_out) {
  // lane l of item (i, b): consecutive threads take consecutive states of one l, then the next l
  const int64_t it = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / 32;
  const int lane = threadIdx.x & 31, l = lane / (32 / LH_LANES);
  const int64_t item = it * (32 / LH_LANES) + lane % (32 / LH_LANES);
  const bool on = item < nn * B;
  const int64_t i = on ? item / B : 0;
  const int b = on ? (int)(item - i * B) : 0;
  const int64_t g = perm[i];
  if (on && l == 0) u_out[(int64_t)b * nn + g] = u_s[i * B + b];
  if (!H_out) return;
  double V = 0, h[3] = {0, 0, 0};
  if (on)
    for (int64_t e = nt_off[i] + l; e < nt_off[i + 1]; e += LH_LANES) {
      const int64_t t = nt_tet[e];
      const double* gr = grad + 12 * t;
      const double w = vol[t];
      double gu[3] = {0, 0, 0};
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const double uk = u_s[(int64_t)tets_s[4 * t + k] * B + b];
#pragma unroll
        for (int c = 0; c < 3; c++) gu[c] += uk * gr[3 * k + c];
      }
      V += w;
#pragma unroll
      for (int c = 0; c < 3; c++) h[c] += w * gu[c];
    }
#pragma unroll
  for (int o = 16; o >= 32 / LH_LANES; o >>= 1) {
    V += __shfl_xor_sync(0xffffffffu, V, o);
#pragma unroll
    for (int c = 0; c < 3; c++) h[c] += __shfl_xor_sync(0xffffffffu, h[c], o);
  }
  if (on && l == 0)
#pragma unroll
    for (int c = 0; c < 3; c++) H_out[((int64_t)b * nn + g) * 3 + c] = V > 0 ? -h[c] / V : 0.0;
}

// ---------------------------------------------------------------------------
// workspace and the FP64 driver
// ---------------------------------------------------------------------------
static void* ws_alloc(Workspace& W, size_t bytes) {
  void* p = nullptr;
  if (cudaMalloc(&p, bytes ? bytes : 16) != cudaSuccess) {
    cudaGetLastError();
    fail(DEMAG_ERR_OUT_OF_MEMORY, "workspace allocation failed");
  }
  W.ptrs.push_back(p);
  return p;
}

void destroy_workspace(Plan& P) {
  if (!P.ws) return;
  multi_forget_plan(&P);  // graphs recorded with this workspace
  for (void* p : P.ws->ptrs) cudaFree(p);
  delete P.ws;
  P.ws = nullptr;
}

// sized for the largest batch evaluated so far (grown, never shrunk), so a plan
// built for max_batch states holds only what its evaluations use
Workspace& workspace(Plan& P, int B) {
  const int need = B;
  if (P.ws && P.ws->B >= need) return *P.ws;
  destroy_workspace(P);
  Workspace* W = new Workspace();
  W->B = need;
  const size_t nn = P.nn, ncell = P.ncells;
  const bool mixed = P.opt.precision != DEMAG_FP64, otf = P.opt.near_mode == 0;
  if (!mixed || otf) W->Ms = (double*)ws_alloc(*W, sizeof(double) * nn * 3 * need);  // FP64 sorted M
  if (!mixed) {
    W->Q = (double*)ws_alloc(*W, sizeof(double) * ncell * P.nq * need);
    W->L = (double*)ws_alloc(*W, sizeof(double) * ncell * P.nl * need);
  } else {
    W->Ms32 = (float*)ws_alloc(*W, sizeof(float) * nn * 3 * need);
    W->Q32 = (float*)ws_alloc(*W, sizeof(float) * ncell * P.nq * need);
    W->L32 = (float*)ws_alloc(*W, sizeof(float) * ncell * P.nl * need);
    W->u32 = (float*)ws_alloc(*W, sizeof(float) * nn * need);
    const size_t qp = m2l_tc_pack_bytes(P, need);
    if (qp) W->QP = (unsigned char*)ws_alloc(*W, qp);
    const size_t mp = nf_mp_floats(P, need);
    if (mp) W->MP = (float*)ws_alloc(*W, sizeof(float) * mp);
  }
  if (!mixed || otf) W->u_s = (double*)ws_alloc(*W, sizeof(double) * nn * need);  // FP64 sorted u
  if (otf) {
    W->slice = p2p_slice(need);
    W->state = (double*)ws_alloc(*W, sizeof(double) * face_state_doubles(P, W->slice));
  }
  W->err = (int*)ws_alloc(*W, sizeof(int));  // staging for host M, u, H: at the first host-pointer call
  P.ws = W;
  return *W;
}

bool is_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

void eval_fp64(Plan& P, const double* M, int B, double* u, double* H, cudaStream_t s) {
  eval_fp64_ws(P, workspace(P, B), M, B, u, H, s, true);
}

void eval_fp64_ws(Plan& P, Workspace& W, const double* M, int B, double* u, double* H, cudaStream_t s,
                  bool profile_ok) {
  const double* Md;
  double *ud, *Hd;
  const bool dev = eval_io_begin(P, W, M, B, u, H, &Md, &ud, &Hd, s);
  StageClock clk(P, s, profile_ok);
  clk.begin(DEMAG_STAGE_GATHER);
  k_gather_M<<<nblk(P.nn * B, 256), 256, 0, s>>>(P.nn, B, P.node_perm, Md, W.Ms);
  DM_LAUNCH("k_gather_M");
  clk.launched();
  clk.end();
  // upward pass
  clk.begin(DEMAG_STAGE_P2M);
  DM_CUDA(cudaMemsetAsync(W.Q, 0, sizeof(double) * P.ncells * P.nq * B, s));
  clk.launched(launch_p2m<double>(P, B, W.Ms, W.Q, s));
  clk.end();
  clk.begin(DEMAG_STAGE_M2M);
  clk.launched(launch_m2m<double>(P, B, W.Q, s));
  clk.end();
  // M2L
  clk.begin(DEMAG_STAGE_M2L);
  DM_CUDA(cudaMemsetAsync(W.L, 0, sizeof(double) * P.ncells * P.nl * B, s));
  if (!P.h_m2l_targets.empty()) {
    if (!launch_m2l_tab<double>(P, B, W.Q, W.L, s)) launch_m2l_rows<double>(P, B, W.Q, W.L, s);
    clk.launched();
  }
  clk.end();
  // downward pass
  clk.begin(DEMAG_STAGE_L2L);
  clk.launched(launch_l2l<double>(P, B, W.L, s));
  clk.end();
  clk.begin(DEMAG_STAGE_L2P);
  clk.launched(launch_l2p<double>(P, B, W.L, W.u_s, s));
  clk.end();
  // near field
  near_field_fp64(P, W, B, clk, s);
  // lumped H and output layout
  clk.begin(DEMAG_STAGE_H);
  launch_lumped_H_out(P, B, W.u_s, ud, Hd, s);
  clk.launched();
  clk.end();
  clk.finish();
  eval_io_end(P, W, dev, B, u, H, s);
}

void near_field_fp64(Plan& P, Workspace& W, int B, StageClock& clk, cudaStream_t s) {
  if (P.opt.near_mode == 1) {
    clk.begin(DEMAG_STAGE_P2P);
    if (!P.h_p2p_targets.empty()) {
      launch_near_apply64(P, W.Ms, B, W.u_s, s);
      clk.launched();
    }
    clk.end();
    return;
  }
  clk.begin(DEMAG_STAGE_P2P);
  clk.launched(launch_p2p_fp64(P, W.Ms, W.state, W.slice, B, W.u_s, s));
  clk.end();
}

void launch_gather_M(Plan& P, const double* M, int B, double* Ms, cudaStream_t s) {
  k_gather_M<<<nblk(P.nn * B, 256), 256, 0, s>>>(P.nn, B, P.node_perm, M, Ms);
  DM_LAUNCH("k_gather_M");
}

void launch_lumped_H_out(Plan& P, int B, const double* u_s, double* u, double* H, cudaStream_t s) {
  k_lumped_H_out<<<nblk(P.nn * B * LH_LANES, 256), 256, 0, s>>>(P.nn, B, P.node_perm, P.nt_off, P.nt_tet, P.tets_s, P.tet_grad,
                                                 P.tet_vol, u_s, u, H);
  DM_LAUNCH("k_lumped_H_out");
}

// host/device pointer handling shared by the evaluation paths
bool eval_io_begin(Plan& P, Workspace& W, const double* M, int B, double* u, double* H, const double** Md, double** ud,
                   double** Hd, cudaStream_t s) {
  const bool dev = is_device_ptr(M);
  if (dev != is_device_ptr(u) || (H && dev != is_device_ptr(H)))
    fail(DEMAG_ERR_INVALID_ARG, "M, u and H must be all device or all host pointers");
  *Md = M;
  *ud = u;
  *Hd = H;
  if (!dev) {
    if (!W.M_dev) {
      const size_t nn = P.nn, need = W.B;
      W.M_dev = (double*)ws_alloc(W, sizeof(double) * nn * 3 * need);
      W.u_dev = (double*)ws_alloc(W, sizeof(double) * nn * need);
      W.H_dev = (double*)ws_alloc(W, sizeof(double) * nn * 3 * need);
    }
    DM_CUDA(cudaMemcpyAsync(W.M_dev, M, sizeof(double) * P.nn * 3 * B, cudaMemcpyHostToDevice, s));
    *Md = W.M_dev;
    *ud = W.u_dev;
    *Hd = H ? W.H_dev : nullptr;
  }
  DM_CUDA(cudaMemsetAsync(W.err, 0, sizeof(int), s));
  P.last_err = W.err;
  return dev;
}

void eval_io_end(Plan& P, Workspace& W, bool dev, int B, double* u, double* H, cudaStream_t s) {
  if (dev) return;
  DM_CUDA(cudaMemcpyAsync(u, W.u_dev, sizeof(double) * P.nn * B, cudaMemcpyDeviceToHost, s));
  if (H) DM_CUDA(cudaMemcpyAsync(H, W.H_dev, sizeof(double) * P.nn * 3 * B, cudaMemcpyDeviceToHost, s));
  int herr = 0;
  DM_CUDA(cudaMemcpyAsync(&herr, W.err, sizeof(int), cudaMemcpyDeviceToHost, s));
  DM_CUDA(cudaStreamSynchronize(s));
  if (herr) fail((demag_status)herr, "a bounded device wait expired in the near-field kernel");
}

}  // namespace demag
