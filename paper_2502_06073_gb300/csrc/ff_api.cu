// C ABI of libff: context, weights, workspace and the host-side order of the hot path
// (neighbour update -> per-chunk forward -> adjoint -> force gather -> FP64 energies).
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <algorithm>
#include <climits>
#include <atomic>
#include <mutex>
#include <cstdlib>
#include <string>
#include <vector>

#include "ff_internal.cuh"
#include "tp_gen.cuh"

// ----------------------------------------------------------------------------- launches
static std::atomic<long long> g_launches{0};
void ff_count_launch(int k) { g_launches.fetch_add(k, std::memory_order_relaxed); }

static thread_local std::string g_create_err;

// ----------------------------------------------------------------------------- device
const FfDevice* ff_device() {
  static PerDevice<FfDevice> devices;
  int dev = 0;
  const FfDevice* d = nullptr;
  if (cudaGetDevice(&dev) == cudaSuccess)
    d = devices.get(dev, [dev](FfDevice& v) {
      v.id = dev;
      return cudaDeviceGetAttribute(&v.n_sm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
             cudaDeviceGetAttribute(&v.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) ==
                 cudaSuccess;
    });
  if (!d) cudaGetLastError();
  return d;
}

// ----------------------------------------------------------------------------- profiling
namespace {
const char* kProfNames[PC_COUNT] = {"gemm_f32",   "gemm_bf16",  "env_tp_fwd",   "env_tp_bwd",
                                    "edge_features", "twobody_in", "edge_energy", "rowred_bwd",
                                    "edge_grad",  "force_gather", "neighbors",  "md",
                                    "misc"};
struct ProfState {
  std::mutex mu;
  bool on = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> pool;   // event pairs
  std::vector<std::pair<int, int>> pending;                 // (class, pair index)
  std::vector<int> free_idx;
  long long launches[PC_COUNT] = {0};
  double ms[PC_COUNT] = {0};
};
ProfState& prof() {
  static ProfState p;
  return p;
}
}  // namespace

ProfScope::ProfScope(int cls_, cudaStream_t s_) : cls(cls_), idx(-1), s(s_) {
  ProfState& p = prof();
  if (!p.on) return;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return;
  }
  std::lock_guard<std::mutex> g(p.mu);
  if (p.free_idx.empty()) {
    cudaEvent_t a, b;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    p.pool.push_back({a, b});
    p.free_idx.push_back((int)p.pool.size() - 1);
  }
  idx = p.free_idx.back();
  p.free_idx.pop_back();
  cudaEventRecord(p.pool[idx].first, s);
}

ProfScope::~ProfScope() {
  if (idx < 0) return;
  ProfState& p = prof();
  std::lock_guard<std::mutex> g(p.mu);
  cudaEventRecord(p.pool[idx].second, s);
  p.pending.push_back({cls, idx});
}

namespace {

// SplitMix64 (Steele, Lea & Flood 2014; constants of Vigna's reference splitmix64.c) used
// as a counter-based generator: out(s, n) = mix(s + n * gamma).
constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ULL;
inline uint64_t sm_mix(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
inline uint64_t sm_out(uint64_t s, uint64_t n) { return sm_mix(s + n * kGamma); }

// Weight k of tensor t: U(-sqrt3, sqrt3) (unit-variance uniform initialisation).
inline double init_weight(uint64_t seed, uint64_t t, uint64_t k) {
  const uint64_t key = sm_out(seed, t + 1);
  const uint64_t bits = sm_out(key, k + 1);
  const double u = (double)(bits >> 11) * (1.0 / 9007199254740992.0);
  return sqrt(3.0) * (2.0 * u - 1.0);
}

// Input/output kind of layer L of n_layers (the tensor-product kernels' template keys):
// output kind 2 for the last layer (0e only), 1 for the layer before it (natural-parity
// irreps only: no other output reaches a 0e output of the last layer), 0 otherwise; input
// kind 0 for the first layer, 3 (natural irreps from memory) for a last layer after it,
// else 1 after the first layer and 2 after later ones.
void layer_kinds(int L, int n_layers, int* ink, int* outk) {
  *outk = L == n_layers ? 2 : (L == n_layers - 1 ? 1 : 0);
  if (L == 1) *ink = 0;
  else if (L == n_layers) *ink = 3;
  else *ink = std::min(L - 1, 2);
}

const TPKindInfo* tp_kind(int lmax, int in_kind, int out_kind) {
  const int irr = in_kind == 3 ? 0 : in_kind;
  for (int i = 0; i < kNumTPKinds; ++i)
    if (kTPKinds[i].lmax == lmax && kTPKinds[i].in_kind == irr &&
        kTPKinds[i].out_kind == out_kind)
      return &kTPKinds[i];
  return nullptr;
}

struct Tensor {
  std::string name;
  int rows, cols;
  size_t off;   // offset in the FP64 parameter vector
};

}  // namespace

struct ff_ctx {
  ff_hparams hp{};
  uint64_t seed = 0;
  std::string err;
  // structure
  int D = 0, C = 0, lmax = 0, NL = 0, n2b = 0, nlat = 0, ns = 0, ldx = 0, ldw = 0, maxw = 0;
  int maxdim = 1;
  int cgroups = 1;     // channel groups of 32 in the tensor-product kernels (C > 32)
  int layer_np[FF_MAX_LAYERS + 1] = {0}, layer_dout[FF_MAX_LAYERS + 1] = {0};
  int layer_din[FF_MAX_LAYERS + 1] = {0};
  int layer_ink[FF_MAX_LAYERS + 1] = {0}, layer_outk[FF_MAX_LAYERS + 1] = {0};
  std::vector<Tensor> tensors;
  std::vector<double> params;
  // device weights
  float* wbuf = nullptr;
  float* W2b[4] = {nullptr}; float* W2bT[4] = {nullptr};
  float* Wenv[FF_MAX_LAYERS + 1] = {nullptr}; float* WenvT[FF_MAX_LAYERS + 1] = {nullptr};
  float* theta[FF_MAX_LAYERS + 1] = {nullptr};
  float* Wlat[FF_MAX_LAYERS + 1][4] = {{nullptr}}; float* WlatT[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  float* w_eff = nullptr;
  // bf16 weight copies for the tensor-core path: W [in][out] (adjoint operand) and
  // W^T [out][in] (forward operand)
  __nv_bfloat16* wbuf_b = nullptr;
  __nv_bfloat16* W2b_b[4] = {nullptr}; __nv_bfloat16* W2bT_b[4] = {nullptr};
  __nv_bfloat16* Wenv_b[FF_MAX_LAYERS + 1] = {nullptr};
  __nv_bfloat16* Bcat_b[FF_MAX_LAYERS + 1] = {nullptr};
  int bcat_k1p = 0, bcat_ld = 0;
  __nv_bfloat16* WenvT_b[FF_MAX_LAYERS + 1] = {nullptr};
  __nv_bfloat16* Wlat_b[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  __nv_bfloat16* WlatT_b[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  // FP32 path on the tensor cores: three bf16 slices of every dense weight matrix, laid out
  // as the W^T [out][in] (forward) and W [in][out] (adjoint) operands; of the first latent
  // matrix's adjoint operand Wlat_s[L][0] holds the scalar rows D.., Bcat_s the others,
  // concatenated with the env weights as in Bcat_b
  __nv_bfloat16* wbuf_s = nullptr;
  __nv_bfloat16* W2b_s[4] = {nullptr}; __nv_bfloat16* W2bT_s[4] = {nullptr};
  __nv_bfloat16* Bcat_s[FF_MAX_LAYERS + 1] = {nullptr};
  __nv_bfloat16* WenvT_s[FF_MAX_LAYERS + 1] = {nullptr};
  __nv_bfloat16* Wlat_s[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  __nv_bfloat16* WlatT_s[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  bool gemm_fail = false;
  // system
  int n = 0, n_sys = 0, pbc[3] = {0, 0, 0};
  int n_alloc = 0;            // atoms that the per-atom buffers are sized for
  double box[3] = {0, 0, 0};
  bool bound = false, allpairs = false, built = false;
  // the stream of the last call, and whether calls have used others since the device was last
  // waited for (ff_neighbors)
  cudaStream_t last_stream = nullptr;
  bool used = false, mixed = false;
  NbrGrid grid{};
  float rl2 = 0.f, rc2 = 0.f;
  int vmax = 0;
  int ncells = 0;
  std::vector<int> sys_ptr_h;
  // elements of the buffers that a rebind keeps when they fit (dalloc_keep)
  size_t cap_sys_ptr = 0, cap_esys = 0, cap_ccount = 0, cap_cstart = 0, cap_cfill = 0;
  size_t cap_vlj = 0, cap_vls = 0;
  int* Z = nullptr; int* sys_ptr = nullptr; int* sys_of = nullptr;
  double* L_d = nullptr; float* Lf_d = nullptr;
  int* vl_j = nullptr; int* vl_s = nullptr; int* vl_cnt = nullptr;
  int* cell_of = nullptr; int4* img = nullptr; float4* xf = nullptr;
  int* cell_count = nullptr; int* cell_start = nullptr; int* cell_fill = nullptr;
  int* cell_atoms = nullptr;
  double* xref = nullptr;
  bool xref_set = false;      // xref holds positions of the bound system
  // row_ptr belongs to the standing list; a list update scans into row_ptr_new, and the two are
  // exchanged once the update is known to have succeeded
  int* cnt = nullptr; int* row_ptr = nullptr; int* row_ptr_new = nullptr;
  int* col = nullptr; int* shift = nullptr; int* src = nullptr; int* rev = nullptr;
  long long ecap = 0, E = 0;
  bool listed = false;        // row_ptr .. rev and E are the model list of the bound system
  std::vector<int> row_ptr_h;   // [0] and [n] always; all of it when row_ptr_full
  bool row_ptr_full = false;
  int* scan_tmp = nullptr;
  int* flags = nullptr;       // [0] error bits, [1] displacement flag, [2] edges counted
  int* flags_h = nullptr;     // pinned mirror
  float4* g = nullptr;
  float* E_atom = nullptr;
  float* F_int = nullptr;
  double* esys_tmp = nullptr;
  // workspace (per chunk of edges)
  long long wcap = 0;
  int acap = 0;
  void* wsp = nullptr;
  size_t wsp_bytes = 0;
  float* ef = nullptr; int* zz = nullptr;
  float* fenv = nullptr;   // the cutoff envelope per edge, dense (one float per edge)
  float* z2b[4] = {nullptr}; float* h2b[4] = {nullptr};
  // pre-activations of the tensor-core path, kept in bf16 for the adjoint's SiLU'
  __nv_bfloat16* z2bb[4] = {nullptr};
  __nv_bfloat16* zlatb[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  float* X[FF_MAX_LAYERS + 1] = {nullptr};
  float* zlat[FF_MAX_LAYERS + 1][4] = {{nullptr}}; float* hlat[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  float* Wv[FF_MAX_LAYERS + 1] = {nullptr};
  // env weights of the tensor-core path: the env projection's bf16 output
  __nv_bfloat16* Wvb[FF_MAX_LAYERS + 1] = {nullptr};
  float* V[FF_MAX_LAYERS + 1] = {nullptr};
  float* Gam[FF_MAX_LAYERS + 1] = {nullptr};
  float* GX[2] = {nullptr}; float* GZ[2] = {nullptr}; float* gV[2] = {nullptr};
  float* GW = nullptr; float* gY = nullptr; float* gf = nullptr;
  // bf16 GEMM operands of the tensor-core path
  __nv_bfloat16* h2bb[4] = {nullptr};
  __nv_bfloat16* hlatb[FF_MAX_LAYERS + 1][4] = {{nullptr}};
  __nv_bfloat16* Xb[FF_MAX_LAYERS + 1] = {nullptr};
  __nv_bfloat16* GZb[2] = {nullptr};
  __nv_bfloat16* GWb = nullptr;
  // fused readout (last latent GEMM + edge-energy head; BF16 path: D <= 256): dE_e/dz of the
  // last latent layer, per-edge energies and the envelope-gradient seed, as sums per 128-column
  // slice: E_edge[slice][wcap] and the first slots of gfp (the one-tile GEMM: whole rows,
  // E_edge[0] and gfL)
  bool head = false;
  __nv_bfloat16* GZL = nullptr;
  float* GZLf = nullptr;
  float* E_edge = nullptr; float* gfL = nullptr;
  // envelope-gradient partials written by the fused RES + SiLU-adjoint GEMMs: one slot per
  // (fused launch, 128-column slice), wcap floats each
  float* gfp = nullptr; int gfp_slots = 0;
  // FF_TEST_STALL_ONCE set at creation: the next tensor-core GEMM launch withholds a
  // completion signal so that a bounded device wait runs out (tests of the timeout path)
  bool test_stall_pending = false;
  // state of the last evaluation
  bool state_valid = false;
  int state_chunks = 0;
  std::vector<int> state_starts;   // chunk plan of the last evaluation
  // frozen-list CUDA-graph mode
  long long list_gen = 0;          // incremented by every Verlet-list build
  bool list_fixed = false;         // the model list is the whole Verlet list (rc + skin)
  long long fixed_gen = -1;
  std::vector<int> fixed_starts;
  bool graph_md = false;
  cudaStream_t gstream = nullptr;
  cudaEvent_t ev_a = nullptr, ev_b = nullptr;
  cudaGraphExec_t gexec = nullptr;
  const void* gkey[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
  long long gkey_gen = -1;
  // edge gradients g of the last force evaluation (for the virial)
  const double* g_pos = nullptr;
  double* vir_part = nullptr;
  double* nh_buf = nullptr;     // NVT scratch: kinetic energy and scale factor per system
  // tensor-core GEMM tile configuration (set by ff_autotune)
  int tune_slice = 128, tune_stages = 0;   // the autotuner's pick for 12,288-atom water
  const double* state_pos = nullptr;
  const double* md_force_pos = nullptr;
  long long md_force_gen = -1;
  long long eval_gen = 0;
};

namespace {

int set_err(ff_ctx* c, int code, const std::string& msg) {
  if (c) c->err = msg; else g_create_err = msg;
  return code;
}

#define FF_CK(ctx, call)                                                                   \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess)                                                                 \
      return set_err(ctx, FF_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

#define FF_TRY(expr)          \
  do {                        \
    int r_ = (expr);          \
    if (r_ != FF_OK) return r_; \
  } while (0)

template <typename T>
int dalloc(ff_ctx* c, T** p, size_t count) {
  if (*p) { cudaFree(*p); *p = nullptr; }
  if (count == 0) count = 1;
  cudaError_t e = cudaMalloc((void**)p, count * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
    return set_err(c, FF_ERR_OOM,
                   std::string("cudaMalloc of ") + std::to_string(count * sizeof(T)) +
                                      " bytes failed: " + cudaGetErrorString(e));
  }
  return FF_OK;
}

// dalloc for a buffer whose capacity is remembered: kept while it fits and is at most four
// times what is asked for (a free and an allocation cost more than a small system's whole
// neighbour build), given back and allocated anew otherwise.
template <typename T>
int dalloc_keep(ff_ctx* c, T** p, size_t* cap, size_t count) {
  if (*p && count <= *cap && *cap <= 4 * count + 4096) return FF_OK;
  *cap = 0;
  const int r = dalloc(c, p, count);
  if (r == FF_OK) *cap = count;
  return r;
}

template <typename T>
void dfree(T*& p) {
  if (p) cudaFree((void*)p);
  p = nullptr;
}

bool width_ok(int w) { return w >= 16 && w <= 512 && w % 16 == 0; }

int validate(const ff_hparams& hp, std::string& why) {
  if (!(hp.rc > 0.f) || !(hp.skin >= 0.f)) { why = "rc must be > 0 and skin >= 0"; return 0; }
  if (hp.n_basis < 1 || hp.n_basis > 10) { why = "n_basis must be in 1..10"; return 0; }
  if (hp.poly_p < 2) { why = "poly_p must be >= 2"; return 0; }
  if (hp.lmax < 1 || hp.lmax > 2) { why = "lmax must be 1 or 2"; return 0; }
  if (hp.parity != 1) { why = "only parity = 1 (full O(3)) is supported"; return 0; }
  if (hp.n_layers < 1 || hp.n_layers > FF_MAX_LAYERS) {
    why = "n_layers must be in 1..4";
    return 0;
  }
  if (hp.channels != 16 && hp.channels != 32 && hp.channels != 64 && hp.channels != 128) {
    why = "channels must be 16, 32, 64 or 128"; return 0;
  }
  if (hp.n_two_body < 1 || hp.n_two_body > 4) { why = "n_two_body must be in 1..4"; return 0; }
  if (hp.n_latent < 1 || hp.n_latent > 4) { why = "n_latent must be in 1..4"; return 0; }
  if (hp.n_edge_eng < 0 || hp.n_edge_eng > 2) { why = "n_edge_eng must be in 0..2"; return 0; }
  for (int k = 0; k < hp.n_two_body; ++k)
    if (!width_ok(hp.two_body[k])) {
      why = "two_body widths must be multiples of 16 in 16..512";
      return 0;
    }
  for (int k = 0; k < hp.n_latent; ++k)
    if (!width_ok(hp.latent[k])) {
      why = "latent widths must be multiples of 16 in 16..512";
      return 0;
    }
  for (int k = 0; k < hp.n_edge_eng; ++k)
    if (hp.edge_eng[k] < 1) { why = "edge_eng widths must be positive"; return 0; }
  if (hp.latent[hp.n_latent - 1] != hp.two_body[hp.n_two_body - 1]) {
    why = "the last latent width must equal the last two-body width"; return 0;
  }
  if (!(hp.avg_num_neighbors > 0.f)) { why = "avg_num_neighbors must be > 0"; return 0; }
  if (hp.precision != 0 && hp.precision != 1) { why = "precision must be 0 or 1"; return 0; }
  return 1;
}

void build_structure(ff_ctx* c) {
  const ff_hparams& hp = c->hp;
  c->C = hp.channels;
  c->lmax = hp.lmax;
  c->NL = hp.n_layers;
  c->n2b = hp.n_two_body;
  c->nlat = hp.n_latent;
  c->D = hp.two_body[hp.n_two_body - 1];
  c->ns = hp.lmax + 1;
  c->ldx = c->D + c->ns * c->C;
  c->ldw = (hp.lmax + 1) * c->C;
  c->cgroups = c->C > 32 ? c->C / 32 : 1;
  c->head = hp.precision == 0 || c->D <= 256;   // (the last latent width is D)
  c->maxw = c->ldx;
  for (int k = 0; k < hp.n_two_body; ++k) c->maxw = std::max(c->maxw, hp.two_body[k]);
  for (int k = 0; k < hp.n_latent; ++k) c->maxw = std::max(c->maxw, hp.latent[k]);
  c->maxdim = 1;
  for (int L = 1; L <= c->NL; ++L) {
    layer_kinds(L, c->NL, &c->layer_ink[L], &c->layer_outk[L]);
    const TPKindInfo* k = tp_kind(c->lmax, c->layer_ink[L], c->layer_outk[L]);
    c->layer_np[L] = k->n_paths;
    c->layer_din[L] = k->dim_in;
    c->layer_dout[L] = k->dim_out;
    c->maxdim = std::max(c->maxdim, std::max(k->dim_in, k->dim_out));
  }
  // tensor list (the documented order fixes the tensor ids of the generator)
  c->tensors.clear();
  size_t off = 0;
  auto add = [&](const std::string& name, int r, int co) {
    c->tensors.push_back({name, r, co, off});
    off += (size_t)r * co;
  };
  int fan = 2 * FF_N_SPECIES + hp.n_basis;
  for (int k = 0; k < hp.n_two_body; ++k) {
    add("W2b." + std::to_string(k), fan, hp.two_body[k]);
    fan = hp.two_body[k];
  }
  for (int L = 1; L <= c->NL; ++L) {
    add("Wenv." + std::to_string(L), c->D, c->ldw);
    if (L < c->NL) add("theta." + std::to_string(L), c->layer_np[L], c->C);
    fan = c->ldx;
    for (int k = 0; k < hp.n_latent; ++k) {
      add("Wlat." + std::to_string(L) + "." + std::to_string(k), fan, hp.latent[k]);
      fan = hp.latent[k];
    }
  }
  fan = c->D;
  for (int k = 0; k <= hp.n_edge_eng; ++k) {
    const int w = k < hp.n_edge_eng ? hp.edge_eng[k] : 1;
    add("We." + std::to_string(k), fan, w);
    fan = w;
  }
  c->params.assign(off, 0.0);
  for (size_t t = 0; t < c->tensors.size(); ++t) {
    const Tensor& T = c->tensors[t];
    const size_t n = (size_t)T.rows * T.cols;
    for (size_t k = 0; k < n; ++k) c->params[T.off + k] = init_weight(c->seed, t, k);
  }
}

const Tensor* find_tensor(const ff_ctx* c, const std::string& name) {
  for (const Tensor& t : c->tensors)
    if (t.name == name) return &t;
  return nullptr;
}

int upload_weights(ff_ctx* c) {
  // forward copies [in][out] and transposed copies [out][in] of every matrix, FP32
  std::vector<float> host;
  std::vector<std::pair<float**, size_t>> fix;
  auto put = [&](float** dst, const Tensor* t, bool transpose) {
    const size_t base = host.size();
    const size_t n = (size_t)t->rows * t->cols;
    host.resize(base + ((n + 3) / 4) * 4, 0.f);
    for (int r = 0; r < t->rows; ++r)
      for (int q = 0; q < t->cols; ++q) {
        const double v = c->params[t->off + (size_t)r * t->cols + q];
        if (!transpose) host[base + (size_t)r * t->cols + q] = (float)v;
        else host[base + (size_t)q * t->rows + r] = (float)v;
      }
    fix.push_back({dst, base});
  };
  for (int k = 0; k < c->n2b; ++k) {
    const Tensor* t = find_tensor(c, "W2b." + std::to_string(k));
    put(&c->W2b[k], t, false);
    put(&c->W2bT[k], t, true);
  }
  for (int L = 1; L <= c->NL; ++L) {
    const Tensor* t = find_tensor(c, "Wenv." + std::to_string(L));
    put(&c->Wenv[L], t, false);
    put(&c->WenvT[L], t, true);
    // path weights transposed to [channel][path] (each thread reads its own row) and
    // multiplied by 1/sqrt(paths into the output irrep) in FP32, the product the tensor
    // product applies to every edge
    if (L < c->NL) {
      const size_t base = host.size();
      put(&c->theta[L], find_tensor(c, "theta." + std::to_string(L)), true);
      const TPKindInfo* k = tp_kind(c->lmax, c->layer_ink[L], c->layer_outk[L]);
      const float* sc = kTPPathScale[k - kTPKinds];
      for (int ch = 0; ch < c->C; ++ch)
        for (int q = 0; q < k->n_paths; ++q) {
          float& t = host[base + (size_t)ch * k->n_paths + q];
          t = t * sc[q];
        }
    }
    for (int k = 0; k < c->nlat; ++k) {
      const Tensor* tl = find_tensor(c, "Wlat." + std::to_string(L) + "." + std::to_string(k));
      put(&c->Wlat[L][k], tl, false);
      put(&c->WlatT[L][k], tl, true);
    }
  }
  // the linear edge-energy MLP folds into one vector: w_eff = We0 We1 ... / sqrt(fans)
  std::vector<double> u(1, 1.0);
  for (int k = c->hp.n_edge_eng; k >= 0; --k) {
    const Tensor* t = find_tensor(c, "We." + std::to_string(k));
    std::vector<double> un(t->rows, 0.0);
    for (int r = 0; r < t->rows; ++r) {
      double s = 0.0;
      for (int q = 0; q < t->cols; ++q) s += c->params[t->off + (size_t)r * t->cols + q] * u[q];
      un[r] = s / sqrt((double)t->rows);
    }
    u.swap(un);
  }
  {
    const size_t base = host.size();
    host.resize(base + ((u.size() + 3) / 4) * 4, 0.f);
    for (size_t d = 0; d < u.size(); ++d) host[base + d] = (float)u[d];
    fix.push_back({&c->w_eff, base});
  }
  FF_TRY(dalloc(c, &c->wbuf, host.size()));
  FF_CK(c, cudaMemcpy(c->wbuf, host.data(), host.size() * sizeof(float), cudaMemcpyHostToDevice));
  for (auto& f : fix) *f.first = c->wbuf + f.second;
  if (c->hp.precision == 0) {
    // bf16 slices of the dense weights for the FP32 GEMM on the tensor cores
    struct Src { __nv_bfloat16** dst; const float* w1; const float* w2; int n, k1, k2; };
    std::vector<Src> src;
    auto add = [&](__nv_bfloat16** dst, const float* w, int rows, int cols) {
      src.push_back({dst, w, nullptr, rows, cols, 0});
    };
    auto both = [&](__nv_bfloat16** w_s, __nv_bfloat16** wt_s, const float* w, const float* wt,
                    int rows, int cols) {
      add(w_s, w, rows, cols);
      add(wt_s, wt, cols, rows);
    };
    const ff_hparams& hp = c->hp;
    for (int k = 1; k < c->n2b; ++k)
      both(&c->W2b_s[k], &c->W2bT_s[k], c->W2b[k], c->W2bT[k], hp.two_body[k - 1], hp.two_body[k]);
    for (int L = 1; L <= c->NL; ++L) {
      const int lat0 = hp.latent[0];
      add(&c->WenvT_s[L], c->WenvT[L], c->ldw, c->D);
      add(&c->WlatT_s[L][0], c->WlatT[L][0], lat0, c->ldx);
      add(&c->Wlat_s[L][0], c->Wlat[L][0] + (size_t)c->D * lat0, c->ldx - c->D, lat0);
      // [Wlat[:D] | (a_env / a_lat) Wenv], a_lat = ldx^-1/2, a_env = D^-1/2 the fan-in scales
      src.push_back({&c->Bcat_s[L], c->Wlat[L][0], c->Wenv[L], c->D, lat0, c->ldw});
      for (int k = 1; k < c->nlat; ++k)
        both(&c->Wlat_s[L][k], &c->WlatT_s[L][k], c->Wlat[L][k], c->WlatT[L][k],
             hp.latent[k - 1], hp.latent[k]);
    }
    std::vector<size_t> off;
    size_t total = 0;
    for (const Src& t : src) {
      off.push_back(total);
      total += ((size_t)3 * t.n * split_ld(t.k1, t.k2) + 127) / 128 * 128;
    }
    FF_TRY(dalloc(c, &c->wbuf_s, total));
    const double ratio = sqrt((double)c->ldx) / sqrt((double)c->D);
    for (size_t i = 0; i < src.size(); ++i) {
      const Src& t = src[i];
      *t.dst = c->wbuf_s + off[i];
      launch_split_weights(t.w1, t.n, t.k1, t.w2, t.k2, ratio, *t.dst, nullptr);
    }
    FF_CK(c, cudaGetLastError());
    FF_CK(c, cudaStreamSynchronize(nullptr));
  }
  if (c->hp.precision != 1) return FF_OK;
  // bf16 copies (rounded once from the FP64 draws) for the tensor-core GEMMs
  std::vector<__nv_bfloat16> hb;
  std::vector<std::pair<__nv_bfloat16**, size_t>> fixb;
  auto putb = [&](__nv_bfloat16** dst, const Tensor* t, bool transpose) {
    const size_t base = hb.size();
    const size_t n = (size_t)t->rows * t->cols;
    hb.resize(base + ((n + 127) / 128) * 128, __float2bfloat16_rn(0.f));
    for (int r = 0; r < t->rows; ++r)
      for (int q = 0; q < t->cols; ++q) {
        const float v = (float)c->params[t->off + (size_t)r * t->cols + q];
        if (!transpose) hb[base + (size_t)r * t->cols + q] = __float2bfloat16_rn(v);
        else hb[base + (size_t)q * t->rows + r] = __float2bfloat16_rn(v);
      }
    fixb.push_back({dst, base});
  };
  for (int k = 0; k < c->n2b; ++k) {
    const Tensor* t = find_tensor(c, "W2b." + std::to_string(k));
    if (k > 0) {
      putb(&c->W2b_b[k], t, false);
      putb(&c->W2bT_b[k], t, true);
    }
  }
  for (int L = 1; L <= c->NL; ++L) {
    const Tensor* t = find_tensor(c, "Wenv." + std::to_string(L));
    putb(&c->Wenv_b[L], t, false);
    putb(&c->WenvT_b[L], t, true);
    for (int k = 0; k < c->nlat; ++k) {
      const Tensor* tl = find_tensor(c, "Wlat." + std::to_string(L) + "." + std::to_string(k));
      putb(&c->Wlat_b[L][k], tl, false);
      putb(&c->WlatT_b[L][k], tl, true);
    }
  }
  // adjoint of the latent input and the env weights in one GEMM over [GZ | GW]: per layer
  // Bcat [D][K1p + K2p] = [Wlat[:D] | 0 | (a_env / a_lat) Wenv | 0] with a_lat = ldx^-1/2,
  // a_env = D^-1/2 (the two fan-in scales), K parts padded to multiples of 64
  c->bcat_k1p = (c->hp.latent[0] + 63) / 64 * 64;
  c->bcat_ld = c->bcat_k1p + (c->ldw + 63) / 64 * 64;
  for (int L = 1; L <= c->NL; ++L) {
    const Tensor* tl = find_tensor(c, "Wlat." + std::to_string(L) + ".0");   // [ldx][latent0]
    const Tensor* te = find_tensor(c, "Wenv." + std::to_string(L));          // [D][ldw]
    const double ratio = sqrt((double)c->ldx) / sqrt((double)c->D);
    const size_t base = hb.size();
    const size_t n = (size_t)c->D * c->bcat_ld;
    hb.resize(base + ((n + 127) / 128) * 128, __float2bfloat16_rn(0.f));
    for (int r = 0; r < c->D; ++r) {
      __nv_bfloat16* row = hb.data() + base + (size_t)r * c->bcat_ld;
      for (int q = 0; q < tl->cols; ++q)
        row[q] = __float2bfloat16_rn((float)c->params[tl->off + (size_t)r * tl->cols + q]);
      for (int q = 0; q < te->cols; ++q)
        row[c->bcat_k1p + q] =
            __float2bfloat16_rn((float)(ratio * c->params[te->off + (size_t)r * te->cols + q]));
    }
    fixb.push_back({&c->Bcat_b[L], base});
  }
  FF_TRY(dalloc(c, &c->wbuf_b, hb.size()));
  FF_CK(c, cudaMemcpy(c->wbuf_b, hb.data(), hb.size() * sizeof(__nv_bfloat16),
                      cudaMemcpyHostToDevice));
  for (auto& f : fixb) *f.first = c->wbuf_b + f.second;
  return FF_OK;
}

void free_workspace(ff_ctx* c) {
  if (c->wsp) cudaFree(c->wsp);
  c->wsp = nullptr;
  c->wsp_bytes = 0;
  c->wcap = 0;
  c->acap = 0;
}

// Harmonic-gradient slices per edge: one per (layer, channel group) for the fan-out of the
// environment adjoint, plus one per channel group for the layer-1 term of V^0 = w (x) Y.
int gy_slices(const ff_ctx* c) { return (c->NL + 1) * c->cgroups; }

// Every per-chunk buffer for `ecap` edges and `acap` atoms: (pointer, bytes).
using Plan = std::vector<std::pair<void**, size_t>>;
Plan workspace_plan(ff_ctx* c, long long ecap, long long acap) {
  const ff_hparams& hp = c->hp;
  Plan plan;
  const bool tc = hp.precision == 1;
  const int nsl = (c->D + 127) / 128;
  auto f32 = [&](float** p, long long count) { plan.push_back({(void**)p, (size_t)count * 4}); };
  auto b16 = [&](__nv_bfloat16** p, long long count) {
    plan.push_back({(void**)p, (size_t)count * 2});
  };
  f32(&c->ef, ecap * FF_EF_STRIDE);
  plan.push_back({(void**)&c->zz, (size_t)ecap * 8});
  f32(&c->fenv, ecap);
  for (int k = 0; k < c->n2b; ++k) {
    if (tc) b16(&c->z2bb[k], ecap * hp.two_body[k]);
    else f32(&c->z2b[k], ecap * hp.two_body[k]);
    if (k < c->n2b - 1) {
      if (tc) b16(&c->h2bb[k], ecap * hp.two_body[k]);
      else f32(&c->h2b[k], ecap * hp.two_body[k]);
    }
  }
  // the tensor-core path keeps the residual stream in bf16 (its GEMM operand); x^N is stored,
  // in FP32, only when the readout is not fused
  for (int L = 0; L <= c->NL; ++L) {
    if (L == c->NL ? !c->head : !tc) f32(&c->X[L], ecap * c->ldx);
    if (tc) b16(&c->Xb[L], ecap * c->ldx);
  }
  for (int L = 1; L <= c->NL; ++L) {
    for (int k = 0; k < c->nlat; ++k) {
      if (!(c->head && L == c->NL && k == c->nlat - 1)) {   // (the fused readout keeps none)
        if (tc) b16(&c->zlatb[L][k], ecap * hp.latent[k]);
        else f32(&c->zlat[L][k], ecap * hp.latent[k]);
      }
      if (k < c->nlat - 1) {
        if (tc) b16(&c->hlatb[L][k], ecap * hp.latent[k]);
        else f32(&c->hlat[L][k], ecap * hp.latent[k]);
      }
    }
    if (tc) b16(&c->Wvb[L], ecap * c->ldw);
    else f32(&c->Wv[L], ecap * c->ldw);
    if (L < c->NL) f32(&c->V[L], ecap * (long long)c->layer_dout[L] * c->C);
    f32(&c->Gam[L], acap * 9 * c->C);
  }
  for (int b = 0; b < 2; ++b) {
    f32(&c->GX[b], ecap * c->ldx);
    f32(&c->GZ[b], ecap * c->maxw);
    f32(&c->gV[b], ecap * (long long)c->maxdim * c->C);
  }
  f32(&c->GW, ecap * c->ldw);
  f32(&c->gY, ecap * 9 * gy_slices(c));
  if (tc) {
    f32(&c->gf, ecap);
    b16(&c->GZb[0], ecap * c->maxw);
    b16(&c->GZb[1], ecap * c->maxw);
    b16(&c->GWb, ecap * c->ldw);
  }
  if (c->head) {
    if (tc) b16(&c->GZL, ecap * c->D);
    else f32(&c->GZLf, ecap * c->D);
    f32(&c->E_edge, ecap * nsl);
    if (tc) f32(&c->gfL, ecap);
  }
  c->gfp_slots = (c->NL + 1) * nsl;
  f32(&c->gfp, ecap * c->gfp_slots);
  return plan;
}

// Carve every per-chunk buffer from one allocation sized for `ecap` edges / `acap` atoms.
int ensure_workspace(ff_ctx* c, long long ecap, int acap, long long budget_edges) {
  if (ecap <= c->wcap && acap <= c->acap) return FF_OK;
  // grow with headroom (edge counts drift from step to step in MD, and every regrowth is
  // a free + malloc of the whole workspace), but never beyond the budget
  ecap = std::max(std::min(ecap + ecap / 8 + 4096, std::max(budget_edges / 8 * 9, ecap)), c->wcap);
  acap = std::max(acap + acap / 16 + 64, c->acap);
  free_workspace(c);
  const Plan plan = workspace_plan(c, ecap, acap);
  size_t total = 0;
  for (auto& p : plan) total += (p.second + 255) & ~(size_t)255;
  void* base = nullptr;
  cudaError_t e = cudaMalloc(&base, total);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return set_err(c, FF_ERR_OOM, "workspace allocation of " + std::to_string(total) +
                                      " bytes failed: " + cudaGetErrorString(e));
  }
  c->wsp = base;
  c->wsp_bytes = total;
  size_t off = 0;
  for (auto& p : plan) {
    *p.first = (char*)base + off;
    off += (p.second + 255) & ~(size_t)255;
  }
  c->wcap = ecap;
  c->acap = acap;
  return FF_OK;
}

size_t bytes_per_edge(ff_ctx* c) {
  size_t b = 0;
  for (auto& p : workspace_plan(c, 1, 0)) b += p.second;
  return b;
}

// Edges per chunk: 120 GB (or FF_WORKSPACE_MB) of workspace with its headroom, at most 60 % of
// the device memory that is free or already held by this context's workspace.  Independent of the
// current capacity, so the plan cannot feed back into the allocation.
long long chunk_edge_budget(ff_ctx* c) {
  size_t budget = (size_t)120 << 30;
  if (const char* s = getenv("FF_WORKSPACE_MB")) budget = (size_t)atoll(s) << 20;
  size_t fr = 0, tot = 0;
  if (cudaMemGetInfo(&fr, &tot) == cudaSuccess)
    budget = std::min(budget, (size_t)((fr + c->wsp_bytes) * 0.6));
  else
    cudaGetLastError();
  long long e = (long long)(budget / bytes_per_edge(c)) / 9 * 8;
  return std::max(e, 4096LL);
}

int read_flags(ff_ctx* c, cudaStream_t s) {
  FF_CK(c, cudaMemcpyAsync(c->flags_h, c->flags, 3 * sizeof(int), cudaMemcpyDeviceToHost, s));
  FF_CK(c, cudaStreamSynchronize(s));
  const int e = c->flags_h[0];
  if (e) {
    FF_CK(c, cudaMemsetAsync(c->flags, 0, sizeof(int), s));
    const char* what = nullptr;
    // a list that must grow is rebuilt, which would lose the timeout of work enqueued earlier
    const int st = ff_flags_status(e & FF_FLAG_TIMEOUT ? e & ~FF_FLAG_CAPACITY : e, &what);
    if (st != FF_OK) return set_err(c, st, what);
  }
  return FF_OK;
}

void setup_grid(ff_ctx* c) {
  const float rl = c->hp.rc + c->hp.skin;
  c->rl2 = rl * rl;
  c->rc2 = c->hp.rc * c->hp.rc;
  const double cw_min = (double)rl * (1.0 + 1e-6) + 1e-4;
  long long total = 1;
  for (int k = 0; k < 3; ++k) {
    c->grid.pbc[k] = c->pbc[k];
    c->grid.L[k] = c->box[k];
    c->grid.Lf[k] = (float)c->box[k];
    int nc = (int)floor(c->box[k] / cw_min);
    nc = std::max(1, std::min(nc, 1024));
    c->grid.ncell[k] = nc;
    const double cw = c->box[k] / nc;
    c->grid.reach[k] = c->pbc[k] ? std::max(1, (int)ceil(cw_min / cw)) : 1;
    total *= nc;
  }
  // keep the cell grid below 8M cells (coarser cells only cost extra candidate checks)
  while (total > (8LL << 20)) {
    int kmax = 0;
    for (int k = 1; k < 3; ++k)
      if (c->grid.ncell[k] > c->grid.ncell[kmax]) kmax = k;
    total /= c->grid.ncell[kmax];
    c->grid.ncell[kmax] = std::max(1, c->grid.ncell[kmax] / 2);
    total *= c->grid.ncell[kmax];
    const double cw = c->box[kmax] / c->grid.ncell[kmax];
    c->grid.reach[kmax] = c->pbc[kmax] ? std::max(1, (int)ceil(cw_min / cw)) : 1;
  }
  c->ncells = (int)total;
}

// Enqueue the Verlet list at rc + skin.  A non-finite coordinate sets its error bit; its atom is
// in no cell and in no pair.
void enqueue_build(ff_ctx* c, const double* pos, cudaStream_t s) {
  launch_check_pos(pos, c->n, c->flags, s);
  if (c->allpairs) {
    launch_pos_to_f32(pos, c->n, c->xf, s);
    launch_verlet_allpairs(c->n, c->sys_of, c->sys_ptr, c->xf, c->rl2, c->vmax, c->vl_j, c->vl_s,
                           c->vl_cnt, c->flags, s);
    return;
  }
  cudaMemsetAsync(c->cell_count, 0, (size_t)c->ncells * sizeof(int), s);
  launch_bin_atoms(pos, c->n, c->grid, c->cell_of, c->img, c->xf, c->cell_count, s);
  launch_scan_i32(c->cell_count, c->cell_start, c->ncells, c->scan_tmp, nullptr, s);
  cudaMemsetAsync(c->cell_fill, 0, (size_t)c->ncells * sizeof(int), s);
  launch_cell_scatter(c->cell_of, c->n, c->cell_start, c->cell_fill, c->cell_atoms, s);
  launch_verlet_cells(c->n, c->grid, c->cell_of, c->img, c->xf, c->cell_start, c->cell_atoms,
                      c->rl2, c->vmax, c->vl_j, c->vl_s, c->vl_cnt, c->flags, s);
}

// Grow the per-atom capacity to the largest count of the list just built.
int grow_verlet(ff_ctx* c) {
  std::vector<int> cnt(c->n);
  FF_CK(c, cudaMemcpy(cnt.data(), c->vl_cnt, (size_t)c->n * sizeof(int), cudaMemcpyDeviceToHost));
  const int mx = *std::max_element(cnt.begin(), cnt.end());
  if (mx > FF_MAX_NEIGHBORS)
    return set_err(c, FF_ERR_CAPACITY, "an atom has " + std::to_string(mx) +
                                           " neighbours within rc + skin (limit " +
                                           std::to_string(FF_MAX_NEIGHBORS) + ")");
  c->vmax = std::min(FF_MAX_NEIGHBORS, ((mx * 5 / 4) + 31) / 32 * 32);
  c->bound = false;   // (until both buffers are there)
  FF_TRY(dalloc_keep(c, &c->vl_j, &c->cap_vlj, (size_t)c->n * c->vmax));
  FF_TRY(dalloc_keep(c, &c->vl_s, &c->cap_vls, (size_t)c->n * c->vmax));
  c->bound = true;
  return FF_OK;
}

int built_ok(ff_ctx* c, const double* pos, cudaStream_t s) {
  if (pos != c->xref)
    FF_CK(c, cudaMemcpyAsync(c->xref, pos, (size_t)c->n * 3 * sizeof(double),
                             cudaMemcpyDeviceToDevice, s));
  c->xref_set = true;
  c->built = true;
  c->list_gen++;
  return FF_OK;
}

int build_verlet(ff_ctx* c, const double* pos, cudaStream_t s) {
  c->built = false;
  for (int attempt = 0; attempt < 3; ++attempt) {
    enqueue_build(c, pos, s);
    FF_CK(c, cudaGetLastError());
    const int r = read_flags(c, s);
    if (r == FF_OK) return built_ok(c, pos, s);
    if (r != FF_ERR_CAPACITY) return r;
    FF_TRY(grow_verlet(c));
  }
  return set_err(c, FF_ERR_CAPACITY, "neighbour capacity could not be established");
}

// Edges per atom at distance below the cutoff, their CSR offsets (row_ptr_new) and their number
// (flags[2]).  Nothing of the standing list is written.
void enqueue_count(ff_ctx* c, const double* pos, cudaStream_t s, float r2cut, bool have_xf) {
  if (!have_xf) launch_pos_to_f32(pos, c->n, c->xf, s);
  launch_filter(0, c->n, c->xf, c->Lf_d, r2cut, c->vmax, c->vl_j, c->vl_s, c->vl_cnt, c->cnt,
                nullptr, nullptr, nullptr, nullptr, s);
  launch_scan_i32(c->cnt, c->row_ptr_new, c->n, c->scan_tmp, c->flags + 2, s);
}

// The counts read back without an error (c->flags_h[2] edges) become the model list, and what
// was computed on the one before is given up.  The host keeps all CSR offsets only when the list
// may need several chunks (fill_row_ptr).
int take_list(ff_ctx* c, cudaStream_t s, float r2cut) {
  if ((long long)c->n * c->vmax > INT32_MAX) {
    // the int32 CSR offsets wrap beyond 2^31 - 1 edges: count the edges in 64 bits first
    std::vector<int> cnt_h(c->n);
    FF_CK(c, cudaMemcpy(cnt_h.data(), c->cnt, (size_t)c->n * sizeof(int),
                        cudaMemcpyDeviceToHost));
    long long tot = 0;
    for (const int v : cnt_h) tot += v;
    if (tot > INT32_MAX)
      return set_err(c, FF_ERR_CAPACITY, "the model list has " + std::to_string(tot) +
                                             " edges (limit 2^31 - 1)");
  }
  std::swap(c->row_ptr, c->row_ptr_new);
  c->state_valid = false;
  c->g_pos = nullptr;
  c->list_fixed = false;
  c->listed = false;
  const long long E = c->flags_h[2];
  if (E > c->ecap) {
    const long long cap = std::max(E + E / 8 + 1024, 2 * c->ecap);
    c->ecap = 0;   // (until every buffer is there)
    FF_TRY(dalloc(c, &c->col, cap));
    FF_TRY(dalloc(c, &c->shift, cap));
    FF_TRY(dalloc(c, &c->src, cap));
    FF_TRY(dalloc(c, &c->rev, cap));
    FF_TRY(dalloc(c, &c->g, cap));
    c->ecap = cap;
  }
  c->E = E;
  c->listed = true;
  c->row_ptr_full = false;
  c->row_ptr_h.resize(c->n + 1);
  c->row_ptr_h[0] = 0;
  c->row_ptr_h[c->n] = (int)E;
  launch_filter(1, c->n, c->xf, c->Lf_d, r2cut, c->vmax, c->vl_j, c->vl_s, c->vl_cnt, c->cnt,
                c->row_ptr, c->col, c->shift, c->src, s);
  launch_rev_index(c->E, c->row_ptr, c->col, c->shift, c->src, c->rev, c->flags, s);
  FF_CK(c, cudaGetLastError());
  return FF_OK;
}

// The model list at `r2cut` for positions `pos`, from the standing Verlet list or (build) from
// a new one.  One read-back and wait in the usual case: the error word, the displacement flag
// and the edge count together.  check_disp: also rebuild when an atom has moved more than
// skin/2; the count made on the old list is then thrown away.  An update that fails leaves the
// standing model list and the state computed on it as they were (a Verlet list that it had
// begun to rebuild is built anew by the next update).
int make_list(ff_ctx* c, const double* pos, cudaStream_t s, float r2cut, bool build,
              bool check_disp) {
  if (check_disp && !build) {
    const double lim = 0.5 * (double)c->hp.skin;
    launch_disp_check(pos, c->xref, c->n, lim * lim, c->flags + 1, s);
  }
  for (int attempt = 0; attempt < 4; ++attempt) {
    if (build) {
      c->built = false;
      enqueue_build(c, pos, s);
    }
    enqueue_count(c, pos, s, r2cut, build);
    FF_CK(c, cudaGetLastError());
    const int r = read_flags(c, s);
    if (build && r == FF_ERR_CAPACITY) {
      FF_TRY(grow_verlet(c));
      continue;
    }
    if (r != FF_OK) return r;
    if (!build && check_disp && c->flags_h[1]) {
      FF_CK(c, cudaMemsetAsync(c->flags + 1, 0, sizeof(int), s));
      build = true;
      continue;
    }
    if (build) FF_TRY(built_ok(c, pos, s));
    return take_list(c, s, r2cut);
  }
  return set_err(c, FF_ERR_CAPACITY, "neighbour capacity could not be established");
}

int update_neighbors(ff_ctx* c, const double* pos, cudaStream_t s) {
  return make_list(c, pos, s, c->rc2, !c->built || c->hp.skin <= 0.f, true);
}

// every CSR offset on the host
int fill_row_ptr(ff_ctx* c, cudaStream_t s) {
  if (c->row_ptr_full) return FF_OK;
  FF_CK(c, cudaMemcpyAsync(c->row_ptr_h.data(), c->row_ptr, (size_t)(c->n + 1) * sizeof(int),
                           cudaMemcpyDeviceToHost, s));
  FF_CK(c, cudaStreamSynchronize(s));
  c->row_ptr_full = true;
  return FF_OK;
}

// chunks of consecutive centre atoms with at most `cap` edges each
void plan_chunks(const ff_ctx* c, long long cap, std::vector<int>& starts) {
  starts.clear();
  int a = 0;
  starts.push_back(0);
  if (c->E <= cap) {   // one chunk (the host may not have the offsets in between)
    starts.push_back(c->n);
    return;
  }
  while (a < c->n) {
    int b = a + 1;
    // binary search the last atom boundary within the capacity
    int lo = a + 1, hi = c->n;
    while (lo <= hi) {
      const int mid = (lo + hi) / 2;
      if ((long long)c->row_ptr_h[mid] - c->row_ptr_h[a] <= cap) { b = mid; lo = mid + 1; }
      else hi = mid - 1;
    }
    a = b;
    starts.push_back(a);
  }
}

// C = alpha A B with the precision of the context: FP32 (A32; Wt_s = bf16 slices of W^T
// [N][K]) or BF16 (Ab, Wt_b = W^T [N][K]).
void mlp_gemm(ff_ctx* c, int mode, long long M, int N, int K, const float* A32,
              const __nv_bfloat16* Ab, int lda, const __nv_bfloat16* Wt_s,
              const __nv_bfloat16* Wt_b, const EpiParams& ep, cudaStream_t s) {
  EpiParams e2 = ep;
  if (c->test_stall_pending) {
    e2.test_stall = 1;
    c->test_stall_pending = false;
  }
  if (c->hp.precision == 0) {
    if (!launch_gemm_f32(mode, (int)M, N, K, A32, lda, Wt_s, K, e2, c->flags, s))
      c->gemm_fail = true;
    return;
  }
  if (!launch_gemm_bf16(mode, (int)M, N, K, Ab, lda, Wt_b, K, e2, c->flags, s, c->tune_slice,
                        c->tune_stages))
    c->gemm_fail = true;
}

// Whether all GEMMs are the persistent ones, with row sums per 128-column slice in gfp.
bool slice_sums(const ff_ctx* c) {
  return c->hp.precision == 0 || (c->tune_stages == 0 && c->tune_slice == 128);
}

void forward_chunk(ff_ctx* c, const double* pos, int a0, int a1, float* E_atom, cudaStream_t s) {
  const ff_hparams& hp = c->hp;
  const bool tc = hp.precision == 1;
  const int e0 = c->row_ptr_h[a0];
  const long long Ec = (long long)c->row_ptr_h[a1] - e0;
  const int* rp = c->row_ptr + a0;
  const int na = a1 - a0;
  launch_edge_features(Ec, c->src + e0, c->col + e0, c->shift + e0, pos, c->L_d, 0, c->Z, hp.rc,
                       hp.n_basis, hp.poly_p, c->lmax, c->ef, c->zz, c->fenv, s);
  const float* fptr = c->fenv;   // read with stride 1 by the GEMM epilogues
  // two-body latent MLP
  const int w0 = hp.two_body[0];
  const float a0f = (float)(1.0 / sqrt((double)(2 * FF_N_SPECIES + hp.n_basis)));
  if (c->n2b == 1) {
    launch_twobody_in(Ec, w0, hp.n_basis, c->ef, c->zz, c->W2b[0], a0f, c->z2b[0], c->z2bb[0],
                      tc ? nullptr : c->X[0], c->ldx, tc ? c->Xb[0] : nullptr, c->ldx, 1, s);
  } else {
    launch_twobody_in(Ec, w0, hp.n_basis, c->ef, c->zz, c->W2b[0], a0f, c->z2b[0], c->z2bb[0],
                      tc ? nullptr : c->h2b[0], w0, tc ? c->h2bb[0] : nullptr, w0, 0, s);
    for (int k = 1; k < c->n2b; ++k) {
      const int win = hp.two_body[k - 1], wout = hp.two_body[k];
      const bool last = k == c->n2b - 1;
      EpiParams ep{};
      ep.alpha = (float)(1.0 / sqrt((double)win));
      ep.pre = c->z2b[k]; ep.preb = c->z2bb[k]; ep.ldp = wout;
      if (last) {
        ep.f = fptr; ep.ldf = 1;
        if (tc) { ep.outb = c->Xb[0]; ep.ldob = c->ldx; }
        else { ep.out = c->X[0]; ep.ldo = c->ldx; }
      } else if (tc) {
        ep.outb = c->h2bb[k]; ep.ldob = wout;
      } else {
        ep.out = c->h2b[k]; ep.ldo = wout;
      }
      mlp_gemm(c, last ? EPI_SILU_F : EPI_SILU, Ec, wout, win, c->h2b[k - 1], c->h2bb[k - 1], win,
               c->W2bT_s[k], c->W2bT_b[k], ep, s);
    }
  }
  const float inv_sqrt_nu = (float)(1.0 / sqrt((double)hp.avg_num_neighbors));
  for (int L = 1; L <= c->NL; ++L) {
    EpiParams ep{};
    ep.alpha = (float)(1.0 / sqrt((double)c->D));
    if (tc) { ep.outb = c->Wvb[L]; ep.ldob = c->ldw; }
    else { ep.out = c->Wv[L]; ep.ldo = c->ldw; }
    mlp_gemm(c, EPI_STORE, Ec, c->ldw, c->D, c->X[L - 1], c->Xb[L - 1], c->ldx,
             c->WenvT_s[L], c->WenvT_b[L], ep, s);
    const int last = L == c->NL ? 1 : 0;
    launch_env_tp_fwd(c->lmax, c->layer_ink[L], c->layer_outk[L], c->C, na, rp, e0, c->ef,
                      tc ? (const void*)c->Wvb[L] : (const void*)c->Wv[L], tc ? 1 : 0, c->ldw, L >= 2 ? c->V[L - 1] : nullptr,
                      last ? nullptr : c->theta[L], tc ? nullptr : c->X[L - 1],
                      tc ? c->Xb[L - 1] : nullptr,
                      c->ldx, c->D, last ? nullptr : c->V[L], c->Gam[L], inv_sqrt_nu, s);
    const float* A32 = c->X[L - 1];
    const __nv_bfloat16* Ab = c->Xb[L - 1];
    int fan = c->ldx, lda = c->ldx;
    for (int k = 0; k < c->nlat; ++k) {
      const int wout = hp.latent[k];
      const bool lastk = k == c->nlat - 1;
      EpiParams el{};
      el.alpha = (float)(1.0 / sqrt((double)fan));
      el.pre = c->zlat[L][k]; el.preb = c->zlatb[L][k]; el.ldp = wout;
      if (lastk && c->head && L == c->NL) {
        // last latent layer + edge-energy head in one epilogue: per-edge energies, the
        // envelope-gradient seed and dE/dz of this layer; x^N itself is never stored
        el.pre = nullptr; el.preb = nullptr;
        el.resb = c->Xb[L - 1]; el.res = c->X[L - 1]; el.ldr = c->ldx;
        el.f = fptr; el.ldf = 1;
        el.beta = (float)(1.0 / sqrt(2.0));
        el.wv = c->w_eff;
        el.outb = c->GZL; el.ldob = c->D;
        el.out = c->GZLf; el.ldo = c->D;
        // the envelope-gradient seed: slots of 128 columns, or, where the adjoint takes it from
        // one array, that array.  The readout of D <= 128 with tiles (256, 0) is the persistent
        // kernel too; its only slot is then the array.
        el.eout = c->E_edge; el.gfo = c->gfL;
        el.gfp = slice_sums(c) ? c->gfp : c->gfL; el.gfp_ld = c->wcap;
        mlp_gemm(c, EPI_HEAD, Ec, wout, fan, A32, Ab, lda, c->WlatT_s[L][k],
                 c->WlatT_b[L][k], el, s);
        break;
      }
      if (lastk) {
        el.out = c->X[L]; el.ldo = c->ldx;   // null in the tensor-core path but for x^N
        el.f = fptr; el.ldf = 1;
        el.beta = (float)(1.0 / sqrt(2.0));
        el.ldr = c->ldx;
        if (tc) {
          el.resb = c->Xb[L - 1];
          el.outb = c->Xb[L]; el.ldob = c->ldx;
        } else {
          el.res = c->X[L - 1];
        }
      } else if (tc) {
        el.outb = c->hlatb[L][k]; el.ldob = wout;
      } else {
        el.out = c->hlat[L][k]; el.ldo = wout;
      }
      mlp_gemm(c, lastk ? EPI_SILU_RES : EPI_SILU, Ec, wout, fan, A32, Ab, lda,
               c->WlatT_s[L][k], c->WlatT_b[L][k], el, s);
      A32 = c->hlat[L][k];
      Ab = c->hlatb[L][k];
      fan = lda = wout;
    }
  }
  if (c->head)
    launch_energy_sum(na, rp, e0, c->E_edge, slice_sums(c) ? (c->D + 127) / 128 : 1, c->wcap,
                      E_atom + a0, s);
  else launch_energy(na, rp, e0, c->X[c->NL], c->ldx, c->D, c->w_eff, E_atom + a0, s);
}

void backward_chunk(ff_ctx* c, int a0, int a1, const double* seed, cudaStream_t s) {
  const ff_hparams& hp = c->hp;
  const bool tc = hp.precision == 1;
  const int e0 = c->row_ptr_h[a0];
  const long long Ec = (long long)c->row_ptr_h[a1] - e0;
  if (Ec <= 0) return;
  const int* rp = c->row_ptr + a0;
  const int na = a1 - a0;
  const float* gx = c->w_eff;
  int ldgx = 0;
  int cur = 0, gvb = 0;
  const float inv_sqrt_nu = (float)(1.0 / sqrt((double)hp.avg_num_neighbors));
  const float r2 = (float)(1.0 / sqrt(2.0));
  // with the persistent GEMMs, each layer's dE/dx GEMM also applies the SiLU adjoint of the
  // layer below (its row reduction): dE/dz out, envelope-gradient partials per 128-column
  // slice into their own slots (summed in order by the geometric adjoint); BF16 path: when
  // that dE/dz is bf16, i.e. not below a two-body MLP of a single layer
  const int kb = c->n2b - 1, kl = c->nlat - 1;
  const bool rr_fuse = slice_sums(c);
  const int nsl = (c->D + 127) / 128;
  int n_gfp = c->head && rr_fuse ? nsl : 0;   // the first slots came from the readout
  // the envelope gradient outside the slots, where a row reduction adds to it (BF16 path: above
  // an unfused readout or a two-body MLP of one layer, or with the one-tile GEMMs)
  const float* gf = nullptr;
  if (tc && !(c->head && rr_fuse && kb >= 1)) {
    if (c->head && !rr_fuse)
      cudaMemcpyAsync(c->gf, c->gfL, (size_t)Ec * sizeof(float), cudaMemcpyDeviceToDevice, s);
    else
      cudaMemsetAsync(c->gf, 0, (size_t)Ec * sizeof(float), s);
    gf = c->gf;
  }
  bool rr_done = false;   // dE/dz of the next layer down was produced by the last GEMM
  int zb0 = 0;            // which of the ping-pong dE/dz buffers holds this layer's
  for (int L = c->NL; L >= 1; --L) {
    // dE/dz of this layer came from the readout or from the previous layer's GEMM
    const bool from_head = c->head && L == c->NL;
    const bool fused = from_head || rr_done;
    rr_done = false;
    if (!fused) {   // BF16 path only
      zb0 = 0;
      launch_rowred_bwd(Ec, hp.latent[kl], gx, ldgx, c->zlatb[L][kl], hp.latent[kl], c->ef, r2,
                        nullptr, hp.latent[kl], c->GZb[0], c->gf, s);
    }
    int gzb = from_head ? 0 : zb0;
    const __nv_bfloat16* gzA = from_head ? c->GZL : c->GZb[gzb];
    const float* gzF = from_head ? c->GZLf : c->GZ[gzb];
    for (int k = kl; k >= 1; --k) {
      EpiParams ep{};
      ep.alpha = (float)(1.0 / sqrt((double)hp.latent[k - 1]));
      if (tc) { ep.outb = c->GZb[gzb ^ 1]; ep.ldob = hp.latent[k - 1]; }
      else { ep.out = c->GZ[gzb ^ 1]; ep.ldo = hp.latent[k - 1]; }
      ep.z = c->zlat[L][k - 1]; ep.zb = c->zlatb[L][k - 1]; ep.ldz = hp.latent[k - 1];
      mlp_gemm(c, EPI_DSILU, Ec, hp.latent[k - 1], hp.latent[k], gzF, gzA, hp.latent[k],
               c->Wlat_s[L][k], c->Wlat_b[L][k], ep, s);
      gzb ^= 1;
      gzA = c->GZb[gzb];
      gzF = c->GZ[gzb];
    }
    {
      // gradients of the tensor-product scalars only (GX columns D..): the TP adjoint needs
      // them; the first D columns come after it, together with the env-weight term
      EpiParams ep{};
      ep.alpha = (float)(1.0 / sqrt((double)c->ldx));
      ep.out = c->GX[cur] + c->D; ep.ldo = c->ldx;
      mlp_gemm(c, EPI_STORE, Ec, c->ldx - c->D, hp.latent[0], gzF, gzA, hp.latent[0],
               c->Wlat_s[L][0], tc ? c->Wlat_b[L][0] + (size_t)c->D * hp.latent[0] : nullptr, ep,
               s);
    }
    const int last = L == c->NL ? 1 : 0;
    launch_env_tp_bwd(c->lmax, c->layer_ink[L], c->layer_outk[L], c->C, na, rp, e0, c->ef,
                      tc ? (const void*)c->Wvb[L] : (const void*)c->Wv[L], tc ? 1 : 0, c->ldw,
                      L >= 2 ? c->V[L - 1] : nullptr, last ? nullptr : c->theta[L], c->GX[cur],
                      c->ldx, c->D, last ? nullptr : c->gV[gvb],
                      L >= 2 ? c->gV[gvb ^ 1] : nullptr, c->GW, tc ? c->GWb : nullptr,
                      c->gY + (size_t)c->NL * c->cgroups * 9,
                      c->gY + (size_t)(L - 1) * c->cgroups * 9, 9 * gy_slices(c), c->Gam[L],
                      inv_sqrt_nu, s);
    // dE/dx^(L-1) = a_lat GZ Wlat[:D]^T + a_env GW Wenv^T + gx / sqrt(2): one GEMM over the
    // concatenated K of [GZ | GW] (the env part of Bcat carries a_env / a_lat)
    EpiParams ep{};
    ep.alpha = (float)(1.0 / sqrt((double)c->ldx));
    ep.out = c->GX[cur]; ep.ldo = c->ldx;
    ep.res = gx; ep.ldr = ldgx; ep.beta = r2; ep.split = c->D;
    // the layer below: latent layer L-1 (scale 1/sqrt2) or the two-body MLP (scale 1)
    const bool below_2b = L == 1;
    int mode = EPI_RES;
    if (rr_fuse && !(tc && below_2b && kb < 1)) {
      mode = EPI_RES_DS;
      ep.zs = below_2b ? c->z2bb[kb] : c->zlatb[L - 1][kl];
      ep.z = below_2b ? c->z2b[kb] : c->zlat[L - 1][kl];
      ep.ldzs = ep.ldz = c->D;
      // below the first layer nothing reads dE/dx itself, only the dE/dz of this epilogue
      // (1 KB per edge of writes at D = 256)
      if (below_2b) ep.out = nullptr;
      ep.alpha2 = below_2b ? 1.f : r2;
      zb0 = gzb ^ 1;   // not this GEMM's own operand
      ep.gzo = c->GZb[zb0]; ep.ldgzo = c->D;
      ep.pre = c->GZ[zb0]; ep.ldp = c->D;
      ep.f = c->fenv; ep.ldf = 1;
      ep.gfp = c->gfp + (size_t)n_gfp * c->wcap; ep.gfp_ld = c->wcap;
      n_gfp += nsl;
      rr_done = true;
    }
    const bool ok =
        tc ? launch_gemm_bf16(mode, (int)Ec, c->D, hp.latent[0], gzA, hp.latent[0], c->Bcat_b[L],
                              c->bcat_ld, ep, c->flags, s, c->tune_slice, c->tune_stages, c->GWb,
                              c->ldw, c->ldw)
           : launch_gemm_f32(mode, (int)Ec, c->D, hp.latent[0], gzF, hp.latent[0], c->Bcat_s[L],
                             split_ld(hp.latent[0], c->ldw), ep, c->flags, s, c->GW, c->ldw, c->ldw);
    if (!ok) c->gemm_fail = true;
    gx = c->GX[cur];
    ldgx = c->ldx;
    cur ^= 1;
    gvb ^= 1;
  }
  // two-body MLP: x^0 = f * silu(z_last); the last gradient (dE/dz_0) stays FP32
  const bool b16_first = kb >= 1;
  if (!rr_done)   // BF16 path only
    launch_rowred_bwd(Ec, hp.two_body[kb], gx, ldgx, c->z2bb[kb], hp.two_body[kb], c->ef, 1.f,
                      b16_first ? nullptr : c->GZ[0], hp.two_body[kb],
                      b16_first ? c->GZb[0] : nullptr, c->gf, s);
  int gzb = rr_done ? zb0 : 0;
  for (int k = kb; k >= 1; --k) {
    EpiParams ep{};
    ep.alpha = (float)(1.0 / sqrt((double)hp.two_body[k - 1]));
    if (tc && k > 1) { ep.outb = c->GZb[gzb ^ 1]; ep.ldob = hp.two_body[k - 1]; }
    else { ep.out = c->GZ[gzb ^ 1]; ep.ldo = hp.two_body[k - 1]; }
    ep.z = c->z2b[k - 1]; ep.zb = c->z2bb[k - 1]; ep.ldz = hp.two_body[k - 1];
    mlp_gemm(c, EPI_DSILU, Ec, hp.two_body[k - 1], hp.two_body[k], c->GZ[gzb], c->GZb[gzb],
             hp.two_body[k], c->W2b_s[k], c->W2b_b[k], ep, s);
    gzb ^= 1;
  }
  const int w0 = hp.two_body[0];
  const float a0f = (float)(1.0 / sqrt((double)(2 * FF_N_SPECIES + hp.n_basis)));
  launch_edge_grad(Ec, w0, hp.n_basis, hp.rc, hp.poly_p, c->lmax, c->ef, c->GZ[gzb], w0,
                   c->W2b[0] + (size_t)2 * FF_N_SPECIES * w0, a0f, gf, c->gfp, n_gfp,
                   c->wcap, c->gY, gy_slices(c), c->src + e0, c->sys_of, seed, c->g + e0, s);
}

// chunk plan for the current model list, workspace sized for it
int plan_and_reserve(ff_ctx* c, std::vector<int>& starts, cudaStream_t s) {
  // a list that fits the workspace at hand is one chunk (asking the driver for the free memory
  // takes longer than several kernels of a small system)
  if (c->E <= c->wcap && c->n <= c->acap && !getenv("FF_WORKSPACE_MB")) {
    starts = {0, c->n};
    return FF_OK;
  }
  const long long budget = chunk_edge_budget(c);
  long long cap = budget;
  if (c->E > budget) {
    FF_TRY(fill_row_ptr(c, s));
    // as few chunks as the budget allows, of equal size (an atom has at most FF_MAX_NEIGHBORS
    // edges, so this capacity gives no more of them): 10.4 million edges in chunks of the whole
    // budget and a rest allocate more than they use, and a new system's first pass takes 89.4 ms
    // instead of 83.5 (a pass among others 82.2, now 81.8)
    const long long k = (c->E + budget - 1) / budget;
    cap = std::min(budget, c->E / k + FF_MAX_NEIGHBORS + 1);
  }
  plan_chunks(c, cap, starts);
  long long maxc = 0;
  int maxa = 0;
  for (size_t k = 0; k + 1 < starts.size(); ++k) {
    maxc = std::max(maxc, (long long)c->row_ptr_h[starts[k + 1]] - c->row_ptr_h[starts[k]]);
    maxa = std::max(maxa, starts[k + 1] - starts[k]);
  }
  return ensure_workspace(c, std::max(maxc, 1LL), std::max(maxa, 1), budget);
}

// The model on the current list: per-chunk forward (+ adjoint), system energies, force
// gather.  Enqueues work only (no synchronisation, no allocation), so it can be captured.
int run_model(ff_ctx* c, const double* pos, double* E_sys, float* E_atom, float* F,
              const double* seed, bool forces, const std::vector<int>& starts, cudaStream_t s) {
  float* Ea = E_atom ? E_atom : c->E_atom;
  for (size_t k = 0; k + 1 < starts.size(); ++k) {
    forward_chunk(c, pos, starts[k], starts[k + 1], Ea, s);
    if (forces) backward_chunk(c, starts[k], starts[k + 1], seed, s);
  }
  if (E_atom && E_atom != c->E_atom)
    FF_CK(c, cudaMemcpyAsync(c->E_atom, E_atom, (size_t)c->n * sizeof(float),
                             cudaMemcpyDeviceToDevice, s));
  if (E_sys) launch_esys(Ea, c->sys_ptr, c->n_sys, E_sys, s);
  if (forces) launch_force_gather(c->n, c->row_ptr, c->rev, c->g, F, s);
  FF_CK(c, cudaGetLastError());
  if (c->gemm_fail) {
    c->gemm_fail = false;
    return set_err(c, FF_ERR_CUDA, "tensor-core GEMM launch could not be set up");
  }
  return FF_OK;
}

// check_err: read the device error word back before returning (an MD loop instead reads
// it with each step's displacement check and once after its last step).
int evaluate(ff_ctx* c, const double* pos, double* E_sys, float* E_atom, float* F,
             const double* seed, bool forces, cudaStream_t s, bool check_err = true) {
  FF_TRY(update_neighbors(c, pos, s));
  std::vector<int> starts;
  FF_TRY(plan_and_reserve(c, starts, s));
  FF_TRY(run_model(c, pos, E_sys, E_atom, F, seed, forces, starts, s));
  // the error word of this evaluation (a tensor-core pipeline timeout) is reported by it
  if (check_err) FF_TRY(read_flags(c, s));
  c->g_pos = (forces && !seed) ? pos : nullptr;
  c->state_valid = true;
  c->state_chunks = (int)starts.size() - 1;
  c->state_starts = starts;
  c->state_pos = pos;
  c->eval_gen++;
  return FF_OK;
}

void graph_reset(ff_ctx* c) {
  if (c->gexec) cudaGraphExecDestroy(c->gexec);
  c->gexec = nullptr;
  c->gkey_gen = -1;
}

// The whole Verlet list (rc + skin, as built at the reference positions) becomes the model
// list: edges beyond rc contribute exactly zero (the envelope and its derivative vanish),
// so it stays valid while every atom is within skin/2 of its reference position (`pos`, when the
// bound system has had no list yet).
int prepare_fixed(ff_ctx* c, const double* pos, cudaStream_t s) {
  FF_TRY(make_list(c, c->xref_set ? c->xref : pos, s, c->rl2, !c->built, false));
  FF_TRY(plan_and_reserve(c, c->fixed_starts, s));
  c->list_fixed = true;
  c->fixed_gen = c->list_gen;
  graph_reset(c);
  return FF_OK;
}

// E (+ F) on the frozen list through a CUDA graph: captured at the first call for a set of
// pointers and list generation, replayed afterwards on an internal stream ordered after
// (and before) the caller's stream.
int graph_eval(ff_ctx* c, const double* pos, double* E_sys, float* E_atom, float* F,
               cudaStream_t s) {
  if (!c->list_fixed || c->fixed_gen != c->list_gen) FF_TRY(prepare_fixed(c, pos, s));
  if (!c->gstream) {
    FF_CK(c, cudaStreamCreateWithFlags(&c->gstream, cudaStreamNonBlocking));
    FF_CK(c, cudaEventCreateWithFlags(&c->ev_a, cudaEventDisableTiming));
    FF_CK(c, cudaEventCreateWithFlags(&c->ev_b, cudaEventDisableTiming));
  }
  const bool forces = F != nullptr;
  const void* key[5] = {pos, E_sys, E_atom, F, (const void*)(uintptr_t)forces};
  bool same = c->gexec && c->gkey_gen == c->fixed_gen;
  for (int k = 0; k < 5 && same; ++k) same = key[k] == c->gkey[k];
  FF_CK(c, cudaEventRecord(c->ev_a, s));
  FF_CK(c, cudaStreamWaitEvent(c->gstream, c->ev_a, 0));
  if (same) {
    FF_CK(c, cudaGraphLaunch(c->gexec, c->gstream));
  } else {
    graph_reset(c);
    // this call's result comes from a plain run; the capture that follows records the
    // same kernel sequence for the next calls (the capture does not execute anything)
    FF_TRY(run_model(c, pos, E_sys, E_atom, F, nullptr, forces, c->fixed_starts, c->gstream));
    cudaGraph_t g = nullptr;
    FF_CK(c, cudaStreamBeginCapture(c->gstream, cudaStreamCaptureModeThreadLocal));
    const int r = run_model(c, pos, E_sys, E_atom, F, nullptr, forces, c->fixed_starts,
                            c->gstream);
    const cudaError_t ec = cudaStreamEndCapture(c->gstream, &g);
    if (r != FF_OK) {
      if (g) cudaGraphDestroy(g);
      return r;
    }
    if (ec != cudaSuccess || !g)
      return set_err(c, FF_ERR_CUDA,
                     std::string("graph capture failed: ") + cudaGetErrorString(ec));
    const cudaError_t ei = cudaGraphInstantiate(&c->gexec, g, 0);
    cudaGraphDestroy(g);
    if (ei != cudaSuccess) {
      c->gexec = nullptr;
      return set_err(c, FF_ERR_CUDA, std::string("graph instantiation failed: ") +
                                         cudaGetErrorString(ei));
    }
    for (int k = 0; k < 5; ++k) c->gkey[k] = key[k];
    c->gkey_gen = c->fixed_gen;
  }
  FF_CK(c, cudaEventRecord(c->ev_b, c->gstream));
  FF_CK(c, cudaStreamWaitEvent(s, c->ev_b, 0));
  c->g_pos = forces ? pos : nullptr;
  c->state_valid = false;       // the adjoint entry point needs a plain evaluation
  c->eval_gen++;
  return FF_OK;
}

// Waits for a stream at the end of its scope, unless done is set by then.
struct WaitUnless {
  cudaStream_t s;
  bool done = false;
  ~WaitUnless() {
    if (!done) cudaStreamSynchronize(s);
  }
};

// Rebuild the Verlet list when an atom moved more than skin/2 from its reference.
int check_rebuild(ff_ctx* c, const double* x, cudaStream_t s) {
  const double lim = 0.5 * (double)c->hp.skin;
  launch_disp_check(x, c->xref, c->n, lim * lim, c->flags + 1, s);
  // one read of both words: the displacement flag and the error word of the graph replays
  // enqueued before it (a tensor-core pipeline timeout)
  FF_TRY(read_flags(c, s));
  if (c->flags_h[1] || !c->built) {
    FF_CK(c, cudaMemsetAsync(c->flags + 1, 0, sizeof(int), s));
    FF_TRY(build_verlet(c, x, s));
  }
  return FF_OK;
}

// The stream of a call.
cudaStream_t on_stream(ff_ctx* c, void* stream) {
  const cudaStream_t s = (cudaStream_t)stream;
  if (c->used && s != c->last_stream) c->mixed = true;
  c->used = true;
  c->last_stream = s;
  return s;
}

}  // namespace

// ============================================================================= C ABI
extern "C" {

int ff_create(ff_ctx** out, const ff_hparams* hp, uint64_t seed) {
  if (!out || !hp) return set_err(nullptr, FF_ERR_ARG, "null argument");
  *out = nullptr;
  std::string why;
  if (!validate(*hp, why)) return set_err(nullptr, FF_ERR_ARG, why);
  if (!gemm_bf16_available())
    return set_err(nullptr, FF_ERR_ARG, "tensor-core path unavailable (no tensor-map encoder)");
  ff_ctx* c = new ff_ctx();
  c->hp = *hp;
  c->seed = seed;
  c->test_stall_pending = getenv("FF_TEST_STALL_ONCE") != nullptr;
  build_structure(c);
  int r = upload_weights(c);
  if (r == FF_OK) r = dalloc(c, &c->flags, 4);
  if (r == FF_OK) {
    if (cudaMallocHost((void**)&c->flags_h, 4 * sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      r = set_err(c, FF_ERR_OOM, "pinned host allocation failed");
    }
  }
  if (r == FF_OK && cudaMemset(c->flags, 0, 4 * sizeof(int)) != cudaSuccess)
    r = set_err(c, FF_ERR_CUDA, "cudaMemset failed");
  if (r == FF_OK) r = dalloc(c, &c->scan_tmp, 3 * FF_SCAN_BLOCK + 4);
  if (r == FF_OK) r = dalloc(c, &c->L_d, 3);
  if (r == FF_OK) r = dalloc(c, &c->Lf_d, 3);
  if (r != FF_OK) {
    g_create_err = c->err;
    ff_destroy(c);
    return r;
  }
  *out = c;
  return FF_OK;
}

void ff_destroy(ff_ctx* c) {
  if (!c) return;
  cudaDeviceSynchronize();
  graph_reset(c);
  if (c->gstream) cudaStreamDestroy(c->gstream);
  if (c->ev_a) cudaEventDestroy(c->ev_a);
  if (c->ev_b) cudaEventDestroy(c->ev_b);
  free_workspace(c);
  dfree(c->wbuf); dfree(c->wbuf_b); dfree(c->wbuf_s); dfree(c->Z); dfree(c->sys_ptr); dfree(c->sys_of);
  dfree(c->L_d); dfree(c->Lf_d);
  dfree(c->vl_j); dfree(c->vl_s); dfree(c->vl_cnt); dfree(c->cell_of); dfree(c->img); dfree(c->xf);
  dfree(c->cell_count); dfree(c->cell_start); dfree(c->cell_fill); dfree(c->cell_atoms);
  dfree(c->xref); dfree(c->cnt); dfree(c->row_ptr); dfree(c->row_ptr_new);
  dfree(c->col); dfree(c->shift); dfree(c->src);
  dfree(c->rev); dfree(c->scan_tmp); dfree(c->flags); dfree(c->g); dfree(c->E_atom);
  dfree(c->F_int); dfree(c->esys_tmp); dfree(c->vir_part); dfree(c->nh_buf);
  if (c->flags_h) cudaFreeHost(c->flags_h);
  delete c;
}

int ff_neighbors(ff_ctx* c, const double* pos, const int32_t* Z, int n_atoms, const double box[3],
                 const int pbc[3], const int32_t* sys_ptr, int n_sys, void* stream) {
  if (!c) return FF_ERR_ARG;
  cudaStream_t s = on_stream(c, stream);
  if (!pos || !Z || !box || !pbc || n_atoms < 1 || n_atoms > (16 << 20))
    return set_err(c, FF_ERR_ARG, "pos, Z, box, pbc must be given and 1 <= n_atoms <= 16M");
  if (n_sys < 1) n_sys = 1;
  std::vector<int> sp;
  if (sys_ptr) sp.assign(sys_ptr, sys_ptr + n_sys + 1);
  else { sp = {0, n_atoms}; n_sys = 1; }
  if (sp.front() != 0 || sp.back() != n_atoms)
    return set_err(c, FF_ERR_ARG, "sys_ptr must start at 0 and end at n_atoms");
  for (int k = 0; k < n_sys; ++k)
    if (sp[k + 1] < sp[k]) return set_err(c, FF_ERR_ARG, "sys_ptr must be non-decreasing");
  for (int k = 0; k < 3; ++k) {
    if (!(box[k] > 0.0)) return set_err(c, FF_ERR_ARG, "box lengths must be positive");
    if (pbc[k] != 0 && pbc[k] != 1) return set_err(c, FF_ERR_ARG, "pbc entries must be 0 or 1");
  }
  const bool any_pbc = pbc[0] || pbc[1] || pbc[2];
  if (n_sys > 1 && any_pbc)
    return set_err(c, FF_ERR_ARG, "several systems need a fully non-periodic box");
  // The host arrays that this call copies to the device (box is the caller's).  A copy from
  // pageable memory may still be reading them when cudaMemcpyAsync returns: they outlive the
  // wait of make_list, and a return that does not get there waits itself.
  std::vector<int> sof;
  const float Lf[3] = {(float)box[0], (float)box[1], (float)box[2]};
  WaitUnless copied{s};
  // Replays and other work of earlier calls on another stream may still be reading the buffers
  // that this call writes: allocating them anew waited for the device, keeping them does not.
  if (c->mixed) {
    FF_CK(c, cudaDeviceSynchronize());
    c->mixed = false;
  }
  // the system bound so far is given up here; only a new one that is in place can be evaluated
  c->bound = false;
  c->listed = false;
  c->xref_set = false;
  c->built = false;
  c->state_valid = false;
  c->g_pos = nullptr;
  c->md_force_pos = nullptr;
  c->list_fixed = false;
  c->n = n_atoms;
  c->n_sys = n_sys;
  c->sys_ptr_h = sp;
  for (int k = 0; k < 3; ++k) { c->box[k] = box[k]; c->pbc[k] = pbc[k]; }
  c->allpairs = n_sys > 1;
  setup_grid(c);
  const float rl = c->hp.rc + c->hp.skin;
  if (n_atoms != c->n_alloc) {
    c->n_alloc = 0;   // (until every buffer is there)
    FF_TRY(dalloc(c, &c->Z, n_atoms));
    FF_TRY(dalloc(c, &c->sys_of, n_atoms));
    FF_TRY(dalloc(c, &c->vl_cnt, n_atoms));
    FF_TRY(dalloc(c, &c->cell_of, n_atoms));
    FF_TRY(dalloc(c, &c->img, n_atoms));
    FF_TRY(dalloc(c, &c->xf, n_atoms));
    FF_TRY(dalloc(c, &c->cell_atoms, n_atoms));
    FF_TRY(dalloc(c, &c->xref, (size_t)n_atoms * 3));
    FF_TRY(dalloc(c, &c->cnt, n_atoms));
    FF_TRY(dalloc(c, &c->row_ptr, n_atoms + 1));
    FF_TRY(dalloc(c, &c->row_ptr_new, n_atoms + 1));
    FF_TRY(dalloc(c, &c->E_atom, n_atoms));
    FF_TRY(dalloc(c, &c->F_int, (size_t)n_atoms * 3));
    c->n_alloc = n_atoms;
  }
  FF_TRY(dalloc_keep(c, &c->sys_ptr, &c->cap_sys_ptr, n_sys + 1));
  FF_TRY(dalloc_keep(c, &c->esys_tmp, &c->cap_esys, n_sys));
  FF_TRY(dalloc_keep(c, &c->cell_count, &c->cap_ccount, c->ncells));
  FF_TRY(dalloc_keep(c, &c->cell_start, &c->cap_cstart, c->ncells + 1));
  FF_TRY(dalloc_keep(c, &c->cell_fill, &c->cap_cfill, c->ncells));
  // initial per-atom capacity from the density (grown on overflow)
  int vm;
  if (c->allpairs) {
    int mx = 1;
    for (int k = 0; k < n_sys; ++k) mx = std::max(mx, sp[k + 1] - sp[k]);
    vm = mx;
  } else {
    const double vol = box[0] * box[1] * box[2];
    const double est = 4.0 / 3.0 * M_PI * (double)rl * rl * rl * n_atoms / vol;
    vm = (int)(1.5 * est) + 32;
  }
  vm = std::min(FF_MAX_NEIGHBORS, std::max(32, (vm + 31) / 32 * 32));
  c->vmax = vm;
  FF_TRY(dalloc_keep(c, &c->vl_j, &c->cap_vlj, (size_t)n_atoms * vm));
  FF_TRY(dalloc_keep(c, &c->vl_s, &c->cap_vls, (size_t)n_atoms * vm));
  FF_CK(c, cudaMemcpyAsync(c->Z, Z, (size_t)n_atoms * sizeof(int), cudaMemcpyDeviceToDevice, s));
  if (n_sys == 1) {
    FF_CK(c, cudaMemsetAsync(c->sys_of, 0, (size_t)n_atoms * sizeof(int), s));
  } else {
    sof.resize(n_atoms);
    for (int k = 0; k < n_sys; ++k)
      for (int i = sp[k]; i < sp[k + 1]; ++i) sof[i] = k;
    FF_CK(c, cudaMemcpyAsync(c->sys_of, sof.data(), (size_t)n_atoms * sizeof(int),
                             cudaMemcpyHostToDevice, s));
  }
  FF_CK(c, cudaMemcpyAsync(c->sys_ptr, sp.data(), (size_t)(n_sys + 1) * sizeof(int),
                           cudaMemcpyHostToDevice, s));
  FF_CK(c, cudaMemcpyAsync(c->L_d, box, 3 * sizeof(double), cudaMemcpyHostToDevice, s));
  FF_CK(c, cudaMemcpyAsync(c->Lf_d, Lf, 3 * sizeof(float), cudaMemcpyHostToDevice, s));
  launch_check_species(c->Z, n_atoms, c->flags, s);
  const int r = make_list(c, pos, s, c->rc2, true, false);
  // a list that cannot be built at these positions leaves a system that can be evaluated at others
  c->bound = r != FF_ERR_SPECIES && r != FF_ERR_OOM && r != FF_ERR_CUDA;
  copied.done = r == FF_OK;
  return r;
}

int ff_energy_forces(ff_ctx* c, const double* pos, double* E_sys, float* E_atom, float* F,
                     void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!c->bound) return set_err(c, FF_ERR_STATE, "ff_neighbors must be called first");
  if (!pos) return set_err(c, FF_ERR_ARG, "pos is null");
  c->md_force_pos = nullptr;
  return evaluate(c, pos, E_sys, E_atom, F, nullptr, F != nullptr, on_stream(c, stream));
}

int ff_forces(ff_ctx* c, const double* grad_E, float* F, void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!c->state_valid || !c->state_pos)
    return set_err(c, FF_ERR_STATE, "ff_forces needs a preceding ff_energy_forces");
  if (!F) return set_err(c, FF_ERR_ARG, "F is null");
  cudaStream_t s = on_stream(c, stream);
  if (c->state_chunks == 1) {
    backward_chunk(c, 0, c->n, grad_E, s);
  } else {
    const std::vector<int>& starts = c->state_starts;   // the plan the workspace was sized for
    for (size_t k = 0; k + 1 < starts.size(); ++k) {
      forward_chunk(c, c->state_pos, starts[k], starts[k + 1], c->E_atom, s);
      backward_chunk(c, starts[k], starts[k + 1], grad_E, s);
    }
  }
  launch_force_gather(c->n, c->row_ptr, c->rev, c->g, F, s);
  FF_CK(c, cudaGetLastError());
  if (c->gemm_fail) {
    c->gemm_fail = false;
    return set_err(c, FF_ERR_CUDA, "tensor-core GEMM launch could not be set up");
  }
  FF_TRY(read_flags(c, s));
  c->g_pos = grad_E ? nullptr : c->state_pos;
  return FF_OK;
}

int ff_virial(ff_ctx* c, double* W, void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!W) return set_err(c, FF_ERR_ARG, "W is null");
  if (!c->g_pos)
    return set_err(c, FF_ERR_STATE, "ff_virial needs a preceding force evaluation (unit seed)");
  FF_TRY(dalloc(c, &c->vir_part, (size_t)c->n_sys * 32 * 9));
  launch_virial(c->sys_ptr, c->n_sys, c->row_ptr, c->src, c->col, c->shift, c->g_pos, c->L_d,
                c->g, c->vir_part, W, on_stream(c, stream));
  FF_CK(c, cudaGetLastError());
  return FF_OK;
}

int ff_md_step(ff_ctx* c, double* x, double* v, const double* mass, int n_steps, double dt_fs,
               double* E_pot, double* E_kin, void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!c->bound) return set_err(c, FF_ERR_STATE, "ff_neighbors must be called first");
  if (!x || !v || !mass || n_steps < 0) return set_err(c, FF_ERR_ARG, "bad md arguments");
  cudaStream_t s = on_stream(c, stream);
  if (c->graph_md) {
    // frozen Verlet list + graph replay; the list is rebuilt (and the graph recaptured)
    // when an atom has moved more than skin/2
    if (!(c->md_force_pos == x && c->md_force_gen == c->eval_gen)) {
      FF_TRY(check_rebuild(c, x, s));
      FF_TRY(graph_eval(c, x, nullptr, nullptr, c->F_int, s));
    }
    for (int it = 0; it < n_steps; ++it) {
      launch_kick(c->n, v, c->F_int, mass, 0.5 * dt_fs, s);
      launch_drift(c->n, x, v, dt_fs, s);
      FF_TRY(check_rebuild(c, x, s));
      FF_TRY(graph_eval(c, x, E_pot ? c->esys_tmp : nullptr, nullptr, c->F_int, s));
      if (E_pot)
        FF_CK(c, cudaMemcpyAsync(E_pot + (size_t)it * c->n_sys, c->esys_tmp,
                                 (size_t)c->n_sys * sizeof(double), cudaMemcpyDeviceToDevice, s));
      launch_kick(c->n, v, c->F_int, mass, 0.5 * dt_fs, s);
      if (E_kin) launch_kinetic(v, mass, c->sys_ptr, c->n_sys, E_kin + (size_t)it * c->n_sys, s);
    }
    FF_CK(c, cudaGetLastError());
    FF_TRY(read_flags(c, s));   // the last replay (earlier ones: the next step's check)
    c->md_force_pos = x;
    c->md_force_gen = c->eval_gen;
    return FF_OK;
  }
  if (!(c->md_force_pos == x && c->md_force_gen == c->eval_gen))
    FF_TRY(evaluate(c, x, nullptr, nullptr, c->F_int, nullptr, true, s));
  for (int it = 0; it < n_steps; ++it) {
    launch_kick(c->n, v, c->F_int, mass, 0.5 * dt_fs, s);
    launch_drift(c->n, x, v, dt_fs, s);
    FF_TRY(evaluate(c, x, E_pot ? E_pot + (size_t)it * c->n_sys : nullptr, nullptr, c->F_int,
                    nullptr, true, s, false));
    launch_kick(c->n, v, c->F_int, mass, 0.5 * dt_fs, s);
    if (E_kin) launch_kinetic(v, mass, c->sys_ptr, c->n_sys, E_kin + (size_t)it * c->n_sys, s);
  }
  FF_CK(c, cudaGetLastError());
  FF_TRY(read_flags(c, s));   // the last step's evaluation (earlier ones: the next step's check)
  c->md_force_pos = x;
  c->md_force_gen = c->eval_gen;
  return FF_OK;
}

int ff_energy_forces_graph(ff_ctx* c, const double* pos, double* E_sys, float* E_atom,
                           float* F, void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!c->bound) return set_err(c, FF_ERR_STATE, "ff_neighbors must be called first");
  if (!pos) return set_err(c, FF_ERR_ARG, "pos is null");
  c->md_force_pos = nullptr;
  return graph_eval(c, pos, E_sys, E_atom, F, on_stream(c, stream));
}

int ff_autotune(ff_ctx* c, const double* pos, int* slice, int* stages, double* ms_best,
                void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!c->bound) return set_err(c, FF_ERR_STATE, "ff_neighbors must be called first");
  if (!pos) return set_err(c, FF_ERR_ARG, "pos is null");
  cudaStream_t s = on_stream(c, stream);
  if (c->hp.precision == 1) {
    // stages 0 = the launcher's default (2 stages for 256-column slices; the persistent
    // kernel for narrower ones), 1..4 = the non-persistent kernel with that ring depth
    static const int cand[][2] = {{256, 0}, {256, 3}, {256, 4}, {128, 0},
                                  {128, 1}, {128, 2}, {128, 3}};
    constexpr int ncand = (int)(sizeof(cand) / sizeof(cand[0]));
    cudaEvent_t e0, e1;
    FF_CK(c, cudaEventCreate(&e0));
    FF_CK(c, cudaEventCreate(&e1));
    float best = 1e30f;
    int bi = 0;
    for (int k = 0; k < ncand; ++k) {
      c->tune_slice = cand[k][0];
      c->tune_stages = cand[k][1];
      FF_TRY(evaluate(c, pos, nullptr, nullptr, c->F_int, nullptr, true, s));   // warm-up
      float tot = 0.f;
      for (int r = 0; r < 3; ++r) {
        // neighbour work and host synchronisation stay outside the timed region
        FF_TRY(update_neighbors(c, pos, s));
        std::vector<int> starts;
        FF_TRY(plan_and_reserve(c, starts, s));
        FF_CK(c, cudaEventRecord(e0, s));
        FF_TRY(run_model(c, pos, nullptr, nullptr, c->F_int, nullptr, true, starts, s));
        FF_CK(c, cudaEventRecord(e1, s));
        FF_CK(c, cudaEventSynchronize(e1));
        float ms = 0.f;
        FF_CK(c, cudaEventElapsedTime(&ms, e0, e1));
        tot += ms;
      }
      if (tot < best) { best = tot; bi = k; }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->tune_slice = cand[bi][0];
    c->tune_stages = cand[bi][1];
    if (ms_best) *ms_best = best / 3.0;
    graph_reset(c);
  }
  if (slice) *slice = c->tune_slice;
  if (stages) *stages = c->tune_stages;
  c->state_valid = false;
  c->md_force_pos = nullptr;
  return FF_OK;
}

int ff_set_tiles(ff_ctx* c, int slice, int stages) {
  if (!c) return FF_ERR_ARG;
  if ((slice != 128 && slice != 256) || stages < 0 || stages > 4)
    return set_err(c, FF_ERR_ARG, "slice must be 128 or 256 and stages 0..4");
  c->tune_slice = slice;
  c->tune_stages = stages;
  graph_reset(c);
  c->state_valid = false;
  c->md_force_pos = nullptr;
  return FF_OK;
}

int ff_set_graph(ff_ctx* c, int enable) {
  if (!c) return FF_ERR_ARG;
  c->graph_md = enable != 0;
  c->md_force_pos = nullptr;
  return FF_OK;
}

int ff_md_nvt(ff_ctx* c, double* x, double* v, const double* mass, int n_steps, double dt_fs,
              double T_K, double tau_fs, double* thermo, double* E_pot, double* E_kin,
              double* H, void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!c->bound) return set_err(c, FF_ERR_STATE, "ff_neighbors must be called first");
  if (!x || !v || !mass || !thermo || n_steps < 0 || !(T_K > 0.0) || !(tau_fs > 0.0))
    return set_err(c, FF_ERR_ARG, "bad NVT arguments");
  cudaStream_t s = on_stream(c, stream);
  const double kT = 8.617333262e-5 * T_K;
  FF_TRY(dalloc(c, &c->nh_buf, (size_t)c->n_sys * 2));
  double* ke = c->nh_buf;
  double* scale = c->nh_buf + c->n_sys;
  if (!(c->md_force_pos == x && c->md_force_gen == c->eval_gen))
    FF_TRY(evaluate(c, x, nullptr, nullptr, c->F_int, nullptr, true, s));
  for (int it = 0; it < n_steps; ++it) {
    launch_nh_half(c->n, c->n_sys, c->sys_ptr, c->sys_of, v, mass, ke, scale, thermo, dt_fs, kT,
                   tau_fs, s);
    launch_kick(c->n, v, c->F_int, mass, 0.5 * dt_fs, s);
    launch_drift(c->n, x, v, dt_fs, s);
    FF_TRY(evaluate(c, x, c->esys_tmp, nullptr, c->F_int, nullptr, true, s, false));
    launch_kick(c->n, v, c->F_int, mass, 0.5 * dt_fs, s);
    launch_nh_half(c->n, c->n_sys, c->sys_ptr, c->sys_of, v, mass, ke, scale, thermo, dt_fs, kT,
                   tau_fs, s);
    launch_kinetic(v, mass, c->sys_ptr, c->n_sys, ke, s);
    const size_t o = (size_t)it * c->n_sys;
    if (E_pot)
      FF_CK(c, cudaMemcpyAsync(E_pot + o, c->esys_tmp, c->n_sys * sizeof(double),
                               cudaMemcpyDeviceToDevice, s));
    if (E_kin)
      FF_CK(c, cudaMemcpyAsync(E_kin + o, ke, c->n_sys * sizeof(double),
                               cudaMemcpyDeviceToDevice, s));
    if (H) launch_nh_energy(c->n_sys, c->sys_ptr, c->esys_tmp, ke, thermo, kT, tau_fs, H + o, s);
  }
  FF_CK(c, cudaGetLastError());
  FF_TRY(read_flags(c, s));   // the last step's evaluation (earlier ones: the next step's check)
  c->md_force_pos = x;
  c->md_force_gen = c->eval_gen;
  return FF_OK;
}

int ff_export_params(ff_ctx* c, double* host_buf, size_t cap, size_t* needed) {
  if (!c) return FF_ERR_ARG;
  if (needed) *needed = c->params.size();
  if (!host_buf) return FF_OK;
  if (cap < c->params.size()) return set_err(c, FF_ERR_ARG, "buffer too small");
  memcpy(host_buf, c->params.data(), c->params.size() * sizeof(double));
  return FF_OK;
}

int ff_get_edges(ff_ctx* c, int64_t* n_edges, int32_t* row_ptr, int32_t* col, int32_t* shift,
                 int32_t* rev, size_t cap, void* stream) {
  if (!c) return FF_ERR_ARG;
  if (!c->bound || !c->listed) return set_err(c, FF_ERR_STATE, "no edge list");
  cudaStream_t s = on_stream(c, stream);
  if (n_edges) *n_edges = c->E;
  if (!row_ptr && !col && !shift && !rev) return FF_OK;
  if (cap < (size_t)c->E) return set_err(c, FF_ERR_ARG, "buffer too small");
  if (row_ptr)
    FF_CK(c, cudaMemcpyAsync(row_ptr, c->row_ptr, (size_t)(c->n + 1) * sizeof(int),
                             cudaMemcpyDeviceToHost, s));
  if (col)
    FF_CK(c, cudaMemcpyAsync(col, c->col, (size_t)c->E * sizeof(int), cudaMemcpyDeviceToHost, s));
  if (rev)
    FF_CK(c, cudaMemcpyAsync(rev, c->rev, (size_t)c->E * sizeof(int), cudaMemcpyDeviceToHost, s));
  std::vector<int> packed;
  if (shift) {
    packed.resize(c->E);
    FF_CK(c, cudaMemcpyAsync(packed.data(), c->shift, (size_t)c->E * sizeof(int),
                             cudaMemcpyDeviceToHost, s));
  }
  FF_CK(c, cudaStreamSynchronize(s));
  if (shift)
    for (long long e = 0; e < c->E; ++e)
      ff_unpack_shift(packed[e], shift[3 * e], shift[3 * e + 1], shift[3 * e + 2]);
  return FF_OK;
}

int64_t ff_kernel_launches(const ff_ctx* /*c*/) { return g_launches.load(); }

int ff_profile_enable(int on) {
  ProfState& p = prof();
  std::lock_guard<std::mutex> g(p.mu);
  p.on = on != 0;
  return FF_OK;
}

int ff_profile_read(int64_t* launches, double* ms, int cap, int* n_classes) {
  if (n_classes) *n_classes = PC_COUNT;
  if (cap < PC_COUNT || !launches || !ms) return FF_ERR_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return FF_ERR_CUDA;
  ProfState& p = prof();
  std::lock_guard<std::mutex> g(p.mu);
  for (auto& pr : p.pending) {
    float t = 0.f;
    if (cudaEventElapsedTime(&t, p.pool[pr.second].first, p.pool[pr.second].second) ==
        cudaSuccess) {
      p.ms[pr.first] += t;
      p.launches[pr.first] += 1;
    } else {
      cudaGetLastError();
    }
    p.free_idx.push_back(pr.second);
  }
  p.pending.clear();
  for (int k = 0; k < PC_COUNT; ++k) {
    launches[k] = p.launches[k];
    ms[k] = p.ms[k];
    p.launches[k] = 0;
    p.ms[k] = 0.0;
  }
  return FF_OK;
}

const char* ff_profile_class(int k) { return (k >= 0 && k < PC_COUNT) ? kProfNames[k] : ""; }

const char* ff_last_error(const ff_ctx* c) {
  if (!c) return g_create_err.c_str();
  return c->err.c_str();
}

}  // extern "C"
