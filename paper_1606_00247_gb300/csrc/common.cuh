// common.cuh -- internal declarations shared by the translation units of
// libdemag.so: the plan structure, error plumbing, multi-index helpers.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/demag.h"

namespace demag {

// ---------------------------------------------------------------------------
// errors
// ---------------------------------------------------------------------------
struct Error {
  demag_status status;
  std::string msg;
};
void set_last_error(const std::string& msg);
[[noreturn]] void fail(demag_status s, const std::string& msg);
void check_cuda(cudaError_t e, const char* what, const char* file, int line);
#define DM_CUDA(x) ::demag::check_cuda((x), #x, __FILE__, __LINE__)
#define DM_LAUNCH(what) ::demag::check_cuda(cudaGetLastError(), what, __FILE__, __LINE__)

// Octree constants (Sec. 3.1 reading): 21 bits per axis, cells split up to level 20.
constexpr int KEY_BITS = 21;
constexpr int MAX_LEVEL = 20;
constexpr int MAX_P = 12;
constexpr int MAX_NCOEF = (MAX_P + 1) * (MAX_P + 2) * (MAX_P + 3) / 6;  // 455
constexpr int NF_ROWS = 128;  // target nodes per tile of the tensor-core near field (MMA N <= 128)

__host__ __device__ inline int ncoef_of(int p) { return (p + 1) * (p + 2) * (p + 3) / 6; }

// one coefficient of an octree translation (far.cu)
template <class T>
struct TEnt {
  uint16_t k;  // M2M: class * nq + moment; L2L: local coefficient of the parent
  T c;
};

// one item of the table-driven M2L (m2l32.cu): TAB_TR rows m times TAB_TC moments n
constexpr int TAB_TR = 4, TAB_TC = 8;
struct TabItem {  // 80 bytes
  uint16_t idx[TAB_TR * TAB_TC];  // table position of b_{m+n} for row r, moment j (nc, a zero, where there is no term)
  uint8_t deg[TAB_TC];            // |n|
  int32_t chunk, pad;             // moments TAB_TC chunk ..
};

// Graded multi-index order: total degree t ascending; within t, n_x descending,
// then n_z ascending.  Index of (a,b,c):
//   t(t+1)(t+2)/6 + (b+c)(b+c+1)/2 + c,  t = a+b+c.
__host__ __device__ inline int mi_index(int a, int b, int c) {
  int t = a + b + c, j = b + c;
  return t * (t + 1) * (t + 2) / 6 + j * (j + 1) / 2 + c;
}
__host__ __device__ inline void mi_decode(int idx, int& a, int& b, int& c) {
  int t = 0;
  while ((t + 1) * (t + 2) * (t + 3) / 6 <= idx) t++;
  int r = idx - t * (t + 1) * (t + 2) / 6;
  int j = 0;
  while ((j + 1) * (j + 2) / 2 <= r) j++;
  c = r - j * (j + 1) / 2;
  b = j - c;
  a = t - j;
}

// ---------------------------------------------------------------------------
// Trace-free form of the expansions.  The derivatives b_k of 1/|x| and the
// local coefficients L_k are harmonic, sum_i X_{k+2e_i} = 0, so every X_k is
// fixed by the ones with k_x <= 1:
//   X_(a0+2q, b, c) = (-1)^q sum_{j<=q} C(q,j) X_(a0, b+2j, c+2(q-j)),  a0 in {0, 1}.
// Of the C(p+3, 3) coefficients of order p only (p+1)^2 are independent.  The
// moments enter through sum_n b_{n+m} Q_n alone, so they may be folded onto the
// same indices (the transposed relation, degree by degree: the truncation
// |n| + |m| <= p is untouched): 1,284 products per M2L pair at p = 8 instead
// of 2,838.  All moments have Q_0 = 0 (they are integrals of the gradient of
// y^n), so the rows |m| = p take no term and L has degree < p:
//   moments   nq = (p+1)^2 - 1 per cell, position h_index - 1
//   local     nl = p^2 per cell, position h_index.
// Order: degree t ascending from t^2; within it k_x = 0 by ascending k_z, then
// k_x = 1 by ascending k_z.
__host__ __device__ constexpr int nq_of(int p) { return (p + 1) * (p + 1) - 1; }
__host__ __device__ constexpr int nl_of(int p) { return p * p; }
__host__ __device__ constexpr int h_index(int a, int b, int c) {  // a in {0, 1}
  return (a + b + c) * (a + b + c) + (a ? a + b + c + 1 + c : c);
}
__host__ __device__ constexpr int h_degree(int idx) {
  int t = 0;
  while ((t + 1) * (t + 1) <= idx) t++;
  return t;
}
__host__ __device__ inline void h_decode(int idx, int& a, int& b, int& c) {
  const int t = h_degree(idx), r = idx - t * t;
  a = r > t;
  c = a ? r - t - 1 : r;
  b = t - a - c;
}
// sum over the full multi-indices n that fold onto (a, b, c) of weight * f(n)
template <class F>
__host__ __device__ inline double h_fold(int a, int b, int c, F&& f) {
  double v = 0.0;
  for (int i = 0; 2 * i <= b; i++) {
    int w = (i & 1) ? -1 : 1;  // (-1)^(i+l) C(i+l, i)
    for (int l = 0; 2 * l <= c; l++) {
      v += w * f(a + 2 * (i + l), b - 2 * i, c - 2 * l);
      w = -(w * (i + l + 1)) / (l + 1);  // exact
    }
  }
  return v;
}

// SB consecutive values, 16 bytes at a time where SB allows (then 16-byte aligned)
template <class T, int SB>
__device__ __forceinline__ void load_q(const T* q, T (&v)[SB]) {
  if constexpr (SB * sizeof(T) % 16 == 0) {
    constexpr int V = 16 / sizeof(T);
#pragma unroll
    for (int i = 0; i < SB / V; i++) {
      if constexpr (sizeof(T) == 4) {
        const float4 x = ((const float4*)q)[i];
        v[V * i] = x.x;
        v[V * i + 1] = x.y;
        v[V * i + 2] = x.z;
        v[V * i + 3] = x.w;
      } else {
        const double2 x = ((const double2*)q)[i];
        v[V * i] = x.x;
        v[V * i + 1] = x.y;
      }
    }
  } else if constexpr (SB == 2) {
    const float2 x = *(const float2*)q;
    v[0] = x.x;
    v[1] = x.y;
  } else {
#pragma unroll
    for (int i = 0; i < SB; i++) v[i] = q[i];
  }
}

// ---------------------------------------------------------------------------
// per-tet record used by the near field (sorted tet order, 66 doubles):
//   [0..11]  vertices v0..v3
//   [12..23] unit outward face normals n_F (face F opposite vertex F)
//   [24..59] unit outward in-plane edge normals m_{F,e}, edge e of face F
//   [60..65] edge lengths of the 6 edges (0,1),(0,2),(0,3),(1,2),(1,3),(2,3)
// Tets are stored positively oriented (vertices 2,3 swapped when needed) so the
// faces have the fixed counter-clockwise vertex orders below.
// ---------------------------------------------------------------------------
constexpr int TET_GEO = 66;
// integrated near field (p2p.cu): states per slice and target nodes per block (at
// most); tets per cluster, and the bounds of a cluster's vertices, edges and faces
constexpr int P2P_SLICE = 16, PF_G = 16;
constexpr int CL_TETS = 40;
constexpr int CL_V = 4 * CL_TETS, CL_E = 6 * CL_TETS, CL_F = 4 * CL_TETS;

// ---------------------------------------------------------------------------
// the plan
// ---------------------------------------------------------------------------
struct Plan;
struct Workspace;

struct DevBuf {
  void* ptr = nullptr;
  size_t bytes = 0;
};

struct Plan {
  int device = 0;
  int sms = 0;                    // streaming multiprocessors of the device
  cudaStream_t stream = nullptr;  // plan-build stream
  demag_options opt{};
  int p = 4, nc = 35, nc1 = 20;   // order, ncoef(p), ncoef(p-1)
  int nq = 24, nl = 16;           // trace-free moments and local coefficients per cell
  int64_t nn = 0, nt = 0;
  double lo[3] = {0, 0, 0}, side = 0, scale = 0;
  double plan_ms = 0;
  float tuned_leaf_ms = 0;  // leaf-size tuning: device time of one evaluation of max_batch states
  int tune_source = 0;      // 0: no tuning asked, 1: tuned by timing, 2: choices read from the tuner cache
  int tc_preset_nt = 0, tc_preset_kps = 0, tc_preset_budget = 0;  // M2L launch shape from the tuner cache

  // sorted geometry
  double* nodes_s = nullptr;      // nn x 3 (sorted node order)
  int32_t* tets_s = nullptr;      // nt x 4 sorted node ids, positively oriented
  int32_t* node_perm = nullptr;   // sorted -> original
  int32_t* tet_perm = nullptr;
  uint64_t* node_key = nullptr;   // original order
  uint64_t* tet_key = nullptr;
  double* tet_geo = nullptr;      // nt x TET_GEO
  double* tet_grad = nullptr;     // nt x 12 gradients of the barycentric coords
  double* tet_vol = nullptr;      // nt, |vol|
  double* node_vol = nullptr;     // nn, lumped nodal volume (original order), on first use
  double* node_vol_s = nullptr;   // nn, lumped nodal volume (sorted order), point-dipole sources

  // cells
  int64_t ncells = 0;
  int nlevels = 0;
  std::vector<int64_t> level_start;  // host, nlevels+1
  uint64_t* cell_prefix = nullptr;
  int32_t* cell_level = nullptr;
  int4* cell_range = nullptr;       // tet begin,end, node begin,end
  int32_t* cell_parent = nullptr;
  int32_t* cell_child0 = nullptr;
  int32_t* cell_nchild = nullptr;
  double* cell_centre = nullptr;    // ncells x 3
  double* cell_rsrc = nullptr;
  double* cell_rtgt = nullptr;
  int64_t nleaves = 0;

  // interaction lists (CSR by target cell)
  int64_t n_m2l = 0, n_p2p = 0, n_p2p_pairs = 0;
  int64_t* m2l_off = nullptr;
  int32_t* m2l_src = nullptr;
  int64_t* p2p_off = nullptr;
  int32_t* p2p_src = nullptr;
  // host copies used for launch shapes
  std::vector<int32_t> h_m2l_targets;  // cells with non-empty M2L lists
  std::vector<int32_t> h_p2p_targets;  // leaves with nodes and non-empty P2P lists
  int32_t* m2l_targets = nullptr;      // device copies of the two lists above
  int32_t* p2p_targets = nullptr;

  // targets
  int32_t* node_leaf = nullptr;     // sorted node -> leaf cell
  int32_t* node_leaves = nullptr;   // leaves holding nodes (their nodes are cell_range[c].z .. .w)
  int64_t n_node_leaves = 0;
  // source leaves: support nodes (unique nodes of the leaf's tets)
  int64_t n_sup = 0;
  int64_t* sup_off = nullptr;       // ncells + 1
  int32_t* sup_node = nullptr;      // n_sup sorted node ids
  int32_t* tet_col = nullptr;       // nt x 4: column of each vertex in its leaf's support
  std::vector<int32_t> h_src_leaves;// leaves holding tets
  int32_t* src_leaves = nullptr;
  double* Ghat = nullptr;           // n_sup x nc1 : int lambda_k y^m/m! over the leaf's tets at that node (plan time)

  // node -> incident tets (for lumped H)
  int64_t* nt_off = nullptr;        // nn + 1
  int32_t* nt_tet = nullptr;        // 4 nt, sorted tet ids

  // host copies of the shapes (plan time)
  std::vector<int4> h_range;
  std::vector<int64_t> h_p2p_off;
  std::vector<int32_t> h_p2p_src;

  // precomputed near field (near_mode = 1), per P2P target leaf ti:
  //   columns = unique source nodes of the tets of its P2P source leaves,
  //   W[w_off[ti] + (col * n_T + i) * 3 + c] = sum over those tets t ni col of
  //   int_t lambda_col(r') (r_i - r')_c / |r_i - r'|^3 dV'
  int64_t n_wcols = 0, n_wentries = 0;
  int64_t* w_coloff = nullptr;      // nT + 1
  int32_t* w_cols = nullptr;        // sorted node ids
  int64_t* w_off = nullptr;         // nT + 1, in units of doubles
  double* W64 = nullptr;
  int64_t* w_off32 = nullptr;       // nT + 1, in floats; W32 is [col][node][4]
  float* W32 = nullptr;

  // the same coefficients for the tensor-core near field (split-BF16
  // precisions, near_mode = 1; near_tc.cu): tiles of at most NF_ROWS target
  // nodes of consecutive P2P target leaves (leaves ordered by first node), the
  // union of their columns in groups of 16, W in split BF16 per k-step
  // (group, component) in the tensor-core K-major layout
  int64_t nf_ntiles = 0, nf_ncols = 0, nf_wbytes = 0;
  int64_t* nf_woff = nullptr;       // ntiles: byte offset of the tile in nf_W
  int64_t* nf_coff = nullptr;       // ntiles: first column of the tile in nf_cols
  int32_t* nf_ng = nullptr;         // ntiles: column groups of 16
  int32_t* nf_npad = nullptr;       // ntiles: rows padded to 16
  int32_t* nf_rownode = nullptr;    // ntiles x NF_ROWS: sorted node of each row, -1 = none
  int32_t* nf_cols = nullptr;       // sorted node of each column (groups padded with the last column)
  int32_t* nf_order = nullptr;      // ntiles: launch order, by decreasing column groups
  unsigned char* nf_W = nullptr;
  float* nf_S = nullptr;            // nn x 3: row sums S_i = sum_j W_ij of the coefficients (FP64 sums)

  // tensor-core M2L (TF32 / split BF16): one operator tile set per distinct
  // (level difference, lattice offset) and the operator index of every pair
  unsigned char* tc_ops = nullptr;
  int32_t* m2l_op = nullptr;        // n_m2l
  int64_t n_m2l_keys = 0;           // distinct translation keys (m2l_keys.cu)
  void* m2l_tab = nullptr;          // b_k(v) per key for the CUDA-core M2L (FP64 plans: doubles, else floats)
  TabItem* m2l_tab_items = nullptr; // its work items (per order)
  int m2l_tab_nitems = 0;
  int32_t* m2l_tab_opdl = nullptr;  // n_m2l: key index | (level difference & 255) << 24
  // M2L launch shape of max_batch states: targets per CTA, k-steps per slot, ring bytes; tuned: of every batch
  int tc_nt = 1, tc_kps = 0, tc_budget = 0;
  bool tc_tuned = false;
  int tc_ls = 0;                    // split BF16 limb scheme of the tensor-core M2L (m2l_tc.cu)
  int tc_prom_group = 0, tc_prom_rows = 16;  // accumulator promotion: sources per group (0 = off), rows
  int64_t* tc_g1_off = nullptr;     // one-target groups: list offsets in target order
  int64_t tc_n_g2 = 0;              // two-target groups (consecutive targets), union lists:
  int32_t* tc_g2_tgt = nullptr;     //   2 per group, -1 = none
  int64_t* tc_g2_off = nullptr;
  int32_t* tc_g2_src = nullptr;
  int32_t* tc_g2_op = nullptr;      //   2 per entry: each target's operator, -1 = not in its list

  // far-field operators (far.cu), in the arithmetic of the plan: FP64 plans hold
  // doubles, the others floats
  int g_stride = 0;                 // values per support node of the P2M operator: 3 nq, padded to 4
  void* far_G = nullptr;            // n_sup x g_stride: P2M operator, [moment q][component]
  void* far_h = nullptr;            // nn x nl: the L2P polynomials of every node
  // octree translations as coefficient lists (TEnt<T>, far.cu): M2M entry j of
  // row n at [j][n]; L2L entries of (row, parity class) q in [l2l_cls[q].x, .y)
  int m2m_width = 0;                // most entries of a row
  int32_t* m2m_cnt = nullptr;       // nq: entries of every row
  void* m2m_ent = nullptr;
  int l2l_nent = 0;
  int2* l2l_cls = nullptr;          // 8 nl
  void* l2l_ent = nullptr;
  int32_t* par_list = nullptr;      // cells with children, level by level
  std::vector<int64_t> par_start;   // host, nlevels + 1: parents of level l are par_list[par_start[l] ..]
  // FP32 mass-lumped gradient operator (mixed precision), rows by sorted node:
  //   H_i = sum_e w_e u_{col_e},  w_e = -(1/V_i) sum_{t ni i, col_e} vol_t grad lambda_{col_e}^t
  int64_t* hg_off = nullptr;        // nn + 1
  int32_t* hg_col = nullptr;
  float4* hg_w = nullptr;           // (x, y, z, 0)
  int32_t* node_iperm = nullptr;    // original -> sorted node

  // clusters of source tets of the integrated near field (near_mode 0; p2p.cu):
  // distinct vertices, edges and faces of at most 40 tets of one source leaf
  int64_t n_clusters = 0, n_cl_v = 0, n_cl_e = 0, n_cl_f = 0, n_cl_b = 0;
  int32_t* cl_off = nullptr;        // ncells + 1: clusters of every cell
  int4* cl_cnt = nullptr;           // vertices, edges, faces, boundary faces (which come first)
  int4* cl_pos = nullptr;           // first of each in the arrays below
  int32_t* cl_vnode = nullptr;      // sorted node
  uint32_t* cl_edge = nullptr;      // cluster vertices v0 | v1 << 16
  double* cl_elen = nullptr;
  double* cl_frec = nullptr;        // 16 doubles per face
  uint2* cl_fidx = nullptr;         // vertices (8 bits each), edges (9 bits each)
  int2* cl_ftet = nullptr;          // tets on the two sides, -1 = none
  int64_t n_pc = 0;
  int64_t* pc_off = nullptr;        // per P2P target: its source clusters
  int32_t* pc_src = nullptr;
  int64_t n_pc_blk = 0;
  int4* pc_blk = nullptr;           // the near field's blocks: P2P target, first sorted node, nodes, 0

  std::vector<DevBuf> bufs;
  int64_t device_bytes = 0;
  Workspace* ws = nullptr;
  int* last_err = nullptr;          // device error flag of the most recent evaluation (demag_eval_status)
  uint8_t* bnd_flag = nullptr;      // pointwise field: sorted nodes on a boundary face (on first use)
  double* field_buf = nullptr;      // pointwise field: [sorted node][3][state]
  int field_states = 0;
  int debug_flags = 0;              // demag_plan_debug: test hooks (bit 0: near-field stall, bit 1: planted audit entry)

  // per-stage timers (opt.profile) and launch counts
  double stage_ms[DEMAG_N_STAGES] = {};
  int64_t stage_launches[DEMAG_N_STAGES] = {};
  int64_t n_evals_profiled = 0;
  int64_t eval_launches = 0;
};

// Records CUDA events around the stages of one demag_eval when profiling is on
// and counts kernel launches always; each stage is also an NVTX range (host
// side, seen by profilers that attach to NVTX, free otherwise).
struct StageClock {
  Plan& P;
  cudaStream_t s;
  bool on;
  cudaEvent_t ev[2 * DEMAG_N_STAGES];
  int launches[DEMAG_N_STAGES] = {};
  bool used[DEMAG_N_STAGES] = {};
  int cur = -1;
  uint64_t range = 0;  // open NVTX range of the current stage (0: none)
  StageClock(Plan& P_, cudaStream_t s_, bool allow = true);
  ~StageClock();
  void begin(int stage);
  void end();
  void launched(int n = 1) { launches[cur] += n; }
  void finish();  // synchronises on the last event and accumulates
};

template <class T>
T* dalloc(Plan& P, size_t n) {
  void* p = nullptr;
  size_t bytes = n * sizeof(T);
  if (bytes == 0) bytes = 16;
  cudaError_t e = cudaMalloc(&p, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    fail(DEMAG_ERR_OUT_OF_MEMORY, "cudaMalloc of " + std::to_string(bytes) + " bytes failed");
  }
  P.bufs.push_back({p, bytes});
  P.device_bytes += (int64_t)bytes;
  return (T*)p;
}
void dfree_all(Plan& P);
void dfree(Plan& P, void* ptr);  // one plan buffer, before the plan is destroyed

// plan construction (plan.cu), FP64 evaluation and workspace (fmm.cu)
void build_plan(Plan& P, const double* nodes, const int32_t* tets);
// opt a kernel in to `bytes` of dynamic shared memory on the current device
// (set once per kernel, device and size; thread-safe)
void smem_opt_in(const void* func, size_t bytes);
// bounds audit of every index list of the plan (audit.cu); plant: also audit a
// copy of the M2L source list with one entry out of range (test hook)
void audit_plan(Plan& P, bool plant = false);
void eval_fp64(Plan& P, const double* M, int B, double* u, double* H, cudaStream_t s);
void destroy_workspace(Plan& P);
// pointwise field at the interior nodes (field.cu)
void eval_field(Plan& P, const double* M, int B, double* u, double* H, cudaStream_t s);

// evaluation workspace (one per plan, sized for max_batch states)
struct Workspace {
  int B = 0;
  int slice = 0;  // states per slice that `state` holds (integrated near field)
  double *Ms = nullptr, *Q = nullptr, *L = nullptr, *u_s = nullptr, *state = nullptr;
  float *Ms32 = nullptr, *Q32 = nullptr, *L32 = nullptr, *u32 = nullptr;
  unsigned char* QP = nullptr;  // moments in the tensor-core tile layout (TF32 / split BF16 M2L)
  float* MP = nullptr;          // tensor-core near field: M per 128-state block, [block][node][3][128]
  double *M_dev = nullptr, *u_dev = nullptr, *H_dev = nullptr;  // staging for host pointers
  int* err = nullptr;
  std::vector<void*> ptrs;
};
Workspace& workspace(Plan& P, int B);
// the two drivers on a given workspace (profile_ok = false: no CUDA events are created)
void eval_fp64_ws(Plan& P, Workspace& W, const double* M, int B, double* u, double* H, cudaStream_t s,
                  bool profile_ok);
void eval_mixed_ws(Plan& P, Workspace& W, const double* M, int B, double* u, double* H, cudaStream_t s,
                   bool profile_ok);
bool is_device_ptr(const void* p);
// shared FP64 stages (fmm.cu)
bool eval_io_begin(Plan& P, Workspace& W, const double* M, int B, double* u, double* H, const double** Md, double** ud,
                   double** Hd, cudaStream_t s);
void eval_io_end(Plan& P, Workspace& W, bool dev, int B, double* u, double* H, cudaStream_t s);
void near_field_fp64(Plan& P, Workspace& W, int B, StageClock& clk, cudaStream_t s);
void launch_gather_M(Plan& P, const double* M, int B, double* Ms, cudaStream_t s);
void launch_lumped_H_out(Plan& P, int B, const double* u_s, double* u, double* H, cudaStream_t s);

// precomputed near field (near.cu)
void build_near_field(Plan& P);
void launch_near_apply64(Plan& P, const double* Ms, int B, double* u_s, cudaStream_t s);
void launch_near_apply32(Plan& P, const float* Ms, int B, float* u_s, int* err, cudaStream_t s);
// tensor-core near field (near_tc.cu): used when the plan holds the tiles
bool near_tc_wanted(const Plan& P);
// MP: workspace of nf_mp_floats(P, B) floats for M in the layout of the kernel's bulk
// copies (small batches: for partial sums); returns the kernel launches
size_t nf_mp_floats(const Plan& P, int B);
int launch_near_tc(Plan& P, const float* Ms, float* MP, int B, float* u_s, int* err, cudaStream_t s);
struct M2lKeys {  // distinct translation keys (dl, lattice offset); the key of every pair is P.m2l_op
  bool ok = false;
  std::vector<int4> keys;
};
// the far field on trace-free expansions (far.cu): operators at plan time, then
// P2M, M2M, L2L and L2P in T = double (FP64 plans) or float; each returns its
// kernel launches
void build_far_operators(Plan& P);
template <class T>
int launch_p2m(Plan& P, int B, const T* Ms, T* Q, cudaStream_t s);
template <class T>
int launch_m2m(Plan& P, int B, T* Q, cudaStream_t s);
template <class T>
int launch_l2l(Plan& P, int B, T* L, cudaStream_t s);
template <class T>
int launch_l2p(Plan& P, int B, const T* L, T* u, cudaStream_t s);
// mixed precision: gradient operator and evaluation (fmm32.cu)
void build_gradient_operator(Plan& P);
void eval_mixed(Plan& P, const double* M, int B, double* u, double* H, cudaStream_t s);
// M2L on CUDA cores without a table (m2l32.cu)
template <class T>
void launch_m2l_rows(Plan& P, int B, const T* Q, T* L, cudaStream_t s);
// table-driven M2L on CUDA cores (m2l32.cu): derivative table per key at plan
// time; launch returns false when the plan has no table
void build_m2l_tab(Plan& P, const M2lKeys& K);
template <class T>
bool launch_m2l_tab(Plan& P, int B, const T* Q, T* L, cudaStream_t s);
// largest batch for which the tensor-core precisions run the table-driven FP32
// M2L instead of the tensor-core one (whose tiles hold 128 states)
inline int m2l_table_batch(const Plan& P) {
  return P.opt.m2l_table_batch < 0 ? 0 : (P.opt.m2l_table_batch == 0 ? 8 : P.opt.m2l_table_batch);
}
// several plans in one submission (multi.cu); cached graphs of a plan are
// dropped before the plan or its workspace goes away
void eval_multi(Plan* const* plans, int n, const double* const* M, const int* batch, double* const* u,
                double* const* H, cudaStream_t s);
void multi_forget_plan(const Plan* P);
// energy and LLG stepping (llg.cu); device pointers, user layout (B, N_n, 3)
const double* node_volumes(Plan& P);
void energy(Plan& P, const double* M, const double* H, int B, double* e, cudaStream_t s);
void llg_rk4(Plan& P, double* m, int B, double Ms, double alpha, const double* hext, double dt, int steps,
             cudaStream_t s);
// tensor-core M2L (m2l_tc.cu): operator table at plan time; bytes of the packed
// moments for B states (0 when the tensor-core M2L is off); packs Q into QP and
// runs the M2L (false: not available for this plan, use the CUDA-core M2L)
M2lKeys build_m2l_keys(Plan& P);      // m2l_keys.cu; also fills P.m2l_op and P.n_m2l_keys
void build_m2l_tc(Plan& P, const M2lKeys& K);
size_t m2l_tc_pack_bytes(const Plan& P, int B);
bool launch_m2l_tc(Plan& P, int B, const float* Q, unsigned char* QP, float* L, int* err, cudaStream_t s);

// near field (p2p.cu)
void build_tet_geometry(Plan& P);
// FP64 near field integrated at every evaluation (near_mode 0): clusters of
// source tets at plan time; the doubles of per-face state a slice of `slice`
// states takes; the launch (slices of at most `slice` states, a power of two;
// returns its kernel launches)
void build_clusters(Plan& P);
size_t face_state_doubles(const Plan& P, int slice);
inline int p2p_slice(int B) {
  int k = 1;
  while (k < B && k < P2P_SLICE) k *= 2;
  return k;
}
int launch_p2p_fp64(Plan& P, const double* Ms, double* state, int slice, int B, double* u_s, cudaStream_t s);

}  // namespace demag

// the opaque handle of the C ABI is the plan itself
struct demag_plan_s : demag::Plan {};
