// Multi-layer kernel reduction (Sec. 3.1, the sum of RBF layers):
//   out_i = sum_l var_l sum_j exp(-|x_i - y_j|^2 / (2 l_l^2)) v_{l,j}
// over ONE set of query and source points (the paper's image-plane GP uses
// several layers on the same ray-traced points). It runs on the culled chunk
// sweep (cull.cuh, kCullLay): the squared distance of a pair is formed once
// and shared by the layers, each layer costs one scale, one exp2 and one
// accumulation per right-hand side, and a chunk evaluates only the layers
// whose kernel value there is not 0. Grid sources are read as points.
//
// The sweep over all pairs that served this before was bound by its 3
// exponentials per pair (0.82 of the exp2 rate); of the 2.6e9 pairs of a
// 160k-point image against 128 x 128 sources 10 % are within reach of the
// widest layer and 0.4 % of the narrowest (length scales 1 : 0.447 : 0.2).
// 3 layers x 4 right-hand sides at that size: 1.83 ms before, 0.16 ms now (whole
// calls; 1 right-hand side 0.97 and 0.12 ms). Where every layer reaches every
// source (length scales of the field's own size) the chunk bookkeeping is pure
// cost: 1.07 (4 right-hand sides) to 1.18 times the earlier sweep.
#include <math.h>

#include <algorithm>

#include "cull.cuh"
#include "host.cuh"

namespace lr {

constexpr int kLyMaxRhs = 4;

struct LyPlan {
  int64_t n, m;
  bool q_raytrace, q_grid, self, s_grid;
  CullPlan cull;
  size_t off_q, off_cull, bytes;
};

static lr_status plan_layers(const lr_points* q, const lr_points* s, int32_t L, int32_t nrhs, bool have_beta_out,
                             LyPlan* P) {
  lr_status st = validate_points(q, "gp_kernel_matvec_layers(query)", false);
  if (st != LR_OK) return st;
  if (s) {
    if ((st = validate_points(s, "gp_kernel_matvec_layers(source)", false)) != LR_OK) return st;
    LR_REQUIRE(!has_lens(s), "gp_kernel_matvec_layers: sources must not be ray-traced (use a self-kernel)");
  }
  LR_REQUIRE(L >= 1 && L <= kMaxLayers, "gp_kernel_matvec_layers: n_layers = %d outside [1, %d]", L, kMaxLayers);
  LR_REQUIRE(nrhs >= 1 && nrhs <= kLyMaxRhs, "gp_kernel_matvec_layers: nrhs = %d outside [1, %d]", nrhs, kLyMaxRhs);
  LyPlan p{};
  p.n = q->n;
  p.self = s == nullptr;
  p.m = p.self ? q->n : s->n;
  p.q_raytrace = has_lens(q);
  p.q_grid = !p.q_raytrace && q->xy == nullptr;
  p.s_grid = !p.self && s->xy == nullptr;
  size_t off = 0;
  p.off_q = off;
  if ((p.q_raytrace || p.q_grid) && !have_beta_out) off += align256(8 * (size_t)p.n);
  p.off_cull = off;
  const lr_grid* layout = query_layout(q);
  if (p.n > 0 && p.m > 0) {
    st = plan_cull(kCullLay, nrhs, p.n, layout, p.m, p.self ? layout : query_layout(s), &p.cull, L);
    if (st != LR_OK) return st;
    off += p.cull.bytes;
  }
  p.bytes = off;
  *P = p;
  return LR_OK;
}

}  // namespace lr

using namespace lr;

extern "C" lr_status lr_matvec_layers_workspace_size(const lr_points* query, const lr_points* source, int32_t n_layers,
                                                     int32_t nrhs, size_t* bytes) {
  LR_REQUIRE(bytes != nullptr, "lr_matvec_layers_workspace_size: bytes is NULL");
  LyPlan P;
  lr_status st = plan_layers(query, source, n_layers, nrhs, false, &P);
  if (st != LR_OK) return st;
  *bytes = P.bytes;
  return LR_OK;
}

extern "C" lr_status gp_kernel_matvec_layers(const lr_points* query, const lr_points* source, int32_t n_layers,
                                             const float* lengthscales, const float* variances, const float* v,
                                             int32_t nrhs, float* out, float* beta_out, void* workspace,
                                             size_t workspace_bytes, lr_stream stream) {
  LyPlan P;
  lr_status st = plan_layers(query, source, n_layers, nrhs, beta_out != nullptr, &P);
  if (st != LR_OK) return st;
  LR_REQUIRE(lengthscales != nullptr && variances != nullptr, "gp_kernel_matvec_layers: NULL hyperparameters");
  for (int l = 0; l < n_layers; ++l) {
    LR_REQUIRE(isfinite(lengthscales[l]) && lengthscales[l] > 0.f, "gp_kernel_matvec_layers: lengthscale %d <= 0", l);
    LR_REQUIRE(isfinite(variances[l]), "gp_kernel_matvec_layers: variance %d not finite", l);
  }
  LR_REQUIRE(out != nullptr || P.n == 0, "gp_kernel_matvec_layers: out is NULL");
  LR_REQUIRE(v != nullptr || P.m == 0, "gp_kernel_matvec_layers: v is NULL");
  LR_REQUIRE(workspace_bytes >= P.bytes, "gp_kernel_matvec_layers: workspace of %zu bytes, %zu needed",
             workspace_bytes, P.bytes);
  LR_REQUIRE(P.bytes == 0 || workspace != nullptr, "gp_kernel_matvec_layers: workspace is NULL");
  LR_REQUIRE(((uintptr_t)workspace & 255u) == 0 && ((uintptr_t)beta_out & 7u) == 0,
             "gp_kernel_matvec_layers: misaligned workspace or beta_out");
  cudaStream_t s = as_cuda(stream);
  if (P.n == 0) return LR_OK;
  if (P.m == 0) {
    LR_CHECK_CUDA(cudaMemsetAsync(out, 0, 4 * (size_t)P.n * (size_t)nrhs, s));
    return LR_OK;
  }
  char* ws = static_cast<char*>(workspace);
  const float2* xq = reinterpret_cast<const float2*>(query->xy);
  if (P.q_raytrace || P.q_grid) {
    float2* qb = beta_out ? reinterpret_cast<float2*>(beta_out) : reinterpret_cast<float2*>(ws + P.off_q);
    st = P.q_raytrace ? launch_raytrace(query, qb, nullptr, s) : launch_grid_points(query->grid, qb, s);
    if (st != LR_OK) return st;
    xq = qb;
  }
  const float2* ys = P.self ? xq : reinterpret_cast<const float2*>(P.s_grid ? nullptr : source->xy);
  // the layers in descending length scale
  int32_t order[kMaxLayers];
  for (int l = 0; l < n_layers; ++l) order[l] = l;
  std::stable_sort(order, order + n_layers, [&](int a, int b) { return lengthscales[a] > lengthscales[b]; });
  CullArgs A{};
  float var[kMaxLayers];
  for (int k = 0; k < n_layers; ++k) {
    const double ll = (double)lengthscales[order[k]], c = 1.4426950408889634 / (2.0 * ll * ll);
    A.lay_c[k] = (float)c;
    A.lay_sc[k] = (float)sqrt(c);
    var[k] = variances[order[k]];
  }
  char* cws = ws + P.off_cull;
  if ((st = launch_cull_prep_layers(P.cull, ys, P.s_grid ? &source->grid : nullptr, v, order, var, cws, s)) != LR_OK) return st;
  A.x = xq;
  A.n = P.n;
  A.sc = A.lay_sc[0];
  A.nrhs = nrhs;
  A.out = out;
  return launch_cull_sweep(P.cull, A, cws, -1, s);
}
