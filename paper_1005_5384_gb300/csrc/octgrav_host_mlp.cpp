// octgrav_host_mlp.cpp -- C ABI of the learned opening criterion: the network
// handed to a tree (BF16 weights), training samples and labels from the walk,
// the gradient and the training loop (Sec. 2.2's opening test replaced by a
// network, with the plain test as fallback).
#include "octgrav_host.h"
#include "octgrav_mlp.h"

using namespace ogh;

extern "C" {

// ---- learned opening criterion

static uint16_t to_bf16(float f) {  // round to nearest even
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7f800000u) == 0x7f800000u) return static_cast<uint16_t>(u >> 16);
  u += 0x7fffu + ((u >> 16) & 1u);
  return static_cast<uint16_t>(u >> 16);
}
static uint32_t pack2(float lo, float hi) { return to_bf16(lo) | (static_cast<uint32_t>(to_bf16(hi)) << 16); }

int octgrav_set_criterion(octgrav_tree* t, const float* record, double tau, double theta_lo, double theta_hi,
                          double theta_fb) {
  if (!t) return fail(OCTGRAV_ERR_ARG, "tree is NULL");
  if (!record) {
    if (!t->learned) return OCTGRAV_OK;
    t->learned = false;
    return ogh::rebuild_items(t);  // plain-criterion items (item_split)
  }
  if (!(theta_lo >= 0 && theta_hi >= theta_lo && theta_fb >= 0) || !std::isfinite(tau) || !std::isfinite(theta_hi))
    return fail(OCTGRAV_ERR_ARG, "need 0 <= theta_lo <= theta_hi, theta_fb >= 0 and a finite tau");
  const float* mu = record;
  const float* sg = record + 12;
  const float* xmin = record + 24;
  const float* xmax = record + 36;
  const float* w = record + 48;
  const float* W1 = w;
  const float* b1 = W1 + og::MLP_NH * og::MLP_NF;
  const float* W2 = b1 + og::MLP_NH;
  const float* b2 = W2 + og::MLP_NH * og::MLP_NH;
  const float* w3 = b2 + og::MLP_NH;
  og::MlpDevice D;
  std::memset(&D, 0, sizeof D);
  auto w1 = [&](int u, int k) { return k < og::MLP_NF ? W1[u * og::MLP_NF + k] : 0.f; };
  for (int j = 0; j < 8; ++j)
    for (int L = 0; L < 32; ++L) {  // B fragment of W1^T: rows k = 2(L%4)+{0,1}, +8; column u = 8j + L/4
      const int u = 8 * j + L / 4, k = 2 * (L % 4);
      D.w1f[j][L] = make_uint2(pack2(w1(u, k), w1(u, k + 1)), pack2(w1(u, k + 8), w1(u, k + 9)));
    }
  for (int kk = 0; kk < 4; ++kk)
    for (int j = 0; j < 8; ++j)
      for (int L = 0; L < 32; ++L) {
        const int u = 8 * j + L / 4, k = 16 * kk + 2 * (L % 4);
        const float* r = W2 + u * og::MLP_NH;
        D.w2f[kk][j][L] = make_uint2(pack2(r[k], r[k + 1]), pack2(r[k + 8], r[k + 9]));
      }
  for (int j = 0; j < og::MLP_NH; ++j) {
    D.b1[j] = b1[j];
    D.b2[j] = b2[j];
    D.w3[j] = w3[j];
  }
  for (int i = 0; i < 16; ++i) {
    const bool v = i < og::MLP_NF;
    D.mu[i] = v ? mu[i] : 0.f;
    D.isig[i] = v ? 1.f / sg[i] : 0.f;
    D.xmin[i] = v ? xmin[i] : 0.f;
    D.xmax[i] = v ? xmax[i] : 0.f;
  }
  D.b3 = w3[og::MLP_NH];
  D.tau = static_cast<float>(tau);
  int rc = t->dev->mlp.reserve(sizeof D);
  if (rc) return rc;
  CUDA_TRY(cudaMemcpy(t->dev->mlp.p, &D, sizeof D, cudaMemcpyHostToDevice));
  CUDA_TRY(cudaGetDevice(&t->mlp_device));
  const bool was = t->learned;
  t->learned = true;
  t->theta_lo = static_cast<float>(theta_lo);
  t->theta_hi = static_cast<float>(theta_hi);
  t->theta_fb = static_cast<float>(theta_fb);
  return was ? OCTGRAV_OK : ogh::rebuild_items(t);  // learned-criterion items (item_split)
}

// Host copy of the walk's FP32 opening test (same operations, no contraction).
static bool open_f32_host(const float4& g, const float4& b0, const float4& b1, float theta2, float* d2out) {
  const float h = g.w;
  const float gmin[3] = {b0.x, b0.y, b0.z}, gmax[3] = {b1.x, b1.y, b1.z}, c[3] = {g.x, g.y, g.z};
  float d[3];
  for (int k = 0; k < 3; ++k) {
    const float below = gmin[k] - (c[k] + h), above = (c[k] - h) - gmax[k];
    const float tt = below > above ? below : above;
    d[k] = tt > 0.f ? tt : 0.f;
  }
  const float d2 = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2];
  if (d2out) *d2out = d2;
  return 4.0f * (h * h) >= theta2 * d2;
}

int octgrav_mlp_samples(octgrav_tree* t, const int64_t* groups, int64_t n_groups, double theta_walk, double eps,
                        float* features, float* labels, int64_t* pairs, int64_t cap, int64_t* n_out, void* stream) {
  if (!t || !groups || n_groups < 0 || !n_out) return fail(OCTGRAV_ERR_ARG, "bad argument");
  int rc = check_params(eps, theta_walk, 1.0);
  if (rc) return rc;
  if ((rc = host_images(t))) return rc;
  const int64_t ngr = static_cast<int64_t>(t->group_cell.size());
  const float th2 = static_cast<float>(theta_walk * theta_walk);
  std::vector<int32_t> s_item, s_cell;
  std::vector<int64_t> s_group;
  int max_count = 1;
  for (int64_t q = 0; q < n_groups; ++q) {
    const int64_t g = groups[q];
    if (g < 0 || g >= ngr) return fail(OCTGRAV_ERR_ARG, "group index %lld out of range", (long long)g);
    const int item = t->group_item[g];
    const int4 it = t->items[item];
    const float4 b0 = t->ibox[4 * item], b1 = t->ibox[4 * item + 1];
    max_count = std::max<int>(max_count, static_cast<int>(t->pcount[t->group_cell[g]]));
    std::vector<int32_t> stack;
    if (t->link[it.x].y > 0) stack.push_back(it.x);
    while (!stack.empty()) {
      const int node = stack.back();
      stack.pop_back();
      const int2 lk = t->link[node];
      for (int c = lk.x; c < lk.x + lk.y; ++c) {
        float d2 = 0.f;
        const bool op = open_f32_host(t->geo[c], b0, b1, th2, &d2);
        if (t->geo[c].w > 0.f && d2 > 0.f) {
          s_item.push_back(item);
          s_cell.push_back(c);
          s_group.push_back(g);
        }
        if (op && t->link[c].y > 0) stack.push_back(c);
      }
    }
  }
  const int64_t ns = static_cast<int64_t>(s_item.size());
  *n_out = ns;
  if (!features || !labels || cap <= 0 || ns == 0) return OCTGRAV_OK;
  const int64_t nw = std::min(ns, cap);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (!t->uploaded || t->sysp_dirty) {
    if ((rc = upload(t, st))) return rc;
  }
  // reference accelerations: the same walk at theta = 0.3 with the plain test
  const bool learned = t->learned;
  t->learned = false;
  if ((rc = t->dev->out.reserve(sizeof(float4) * t->n))) { t->learned = learned; return rc; }
  rc = launch(t, eps, 0.3, 1.0, static_cast<float4*>(t->dev->out.p), st);
  t->learned = learned;
  if (rc) return rc;
  if ((rc = read_status(t, st))) return rc;
  // per-cell (first, count) and FP64 moments
  const int64_t nc = t->n_cells;
  std::vector<int2> fc(nc);
  for (int64_t c = 0; c < nc; ++c) fc[c] = make_int2(t->cfirst[c], static_cast<int>(t->pcount[c]));
  DevBuf b_item, b_cell, b_fc, b_com, b_M, b_S, b_feat, b_lab;
  if ((rc = b_item.reserve(4 * nw)) || (rc = b_cell.reserve(4 * nw)) || (rc = b_fc.reserve(8 * nc)) ||
      (rc = b_com.reserve(24 * nc)) || (rc = b_M.reserve(8 * nc)) || (rc = b_S.reserve(48 * nc)) ||
      (rc = b_feat.reserve(4 * og::MLP_NF * nw)) || (rc = b_lab.reserve(8 * nw)))
    return rc;
  CUDA_TRY(cudaMemcpyAsync(b_item.p, s_item.data(), 4 * nw, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(b_cell.p, s_cell.data(), 4 * nw, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(b_fc.p, fc.data(), 8 * nc, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(b_com.p, t->com.data(), 24 * nc, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(b_M.p, t->M.data(), 8 * nc, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(b_S.p, t->S.data(), 48 * nc, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemsetAsync(b_lab.p, 0, 8 * nw, st));
  og::MlpSampleArgs a{};
  a.n = static_cast<int>(nw);
  a.chunks = (max_count + 31) / 32;
  a.item = static_cast<const int*>(b_item.p);
  a.cell = static_cast<const int*>(b_cell.p);
  a.items = static_cast<const int4*>(t->dev->items.p);
  a.ibox = static_cast<const float4*>(t->dev->ibox.p);
  a.geo = static_cast<const float4*>(t->dev->geo.p);
  a.mp = static_cast<const float4*>(t->dev->mp.p);
  a.parts = static_cast<const float4*>(t->dev->parts.p);
  a.link_first_count = static_cast<const int2*>(b_fc.p);
  a.com64 = static_cast<const double*>(b_com.p);
  a.M64 = static_cast<const double*>(b_M.p);
  a.S64 = static_cast<const double*>(b_S.p);
  a.aref = static_cast<const float4*>(t->dev->out.p);
  a.eps2 = eps * eps;
  a.n_group = t->n_group;
  a.feat = static_cast<float*>(b_feat.p);
  a.label64 = static_cast<double*>(b_lab.p);
  cudaError_t e = og::mlp_sample_features(a, st);
  if (e == cudaSuccess) e = og::mlp_sample_labels(a, st);
  if (e != cudaSuccess) return fail(OCTGRAV_ERR_CUDA, "sample kernels failed: %s", cudaGetErrorString(e));
  std::vector<double> lab(nw);
  CUDA_TRY(cudaMemcpyAsync(features, b_feat.p, 4 * og::MLP_NF * nw, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpyAsync(lab.data(), b_lab.p, 8 * nw, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  for (int64_t k = 0; k < nw; ++k) {
    labels[k] = static_cast<float>(lab[k]);
    if (pairs) {
      pairs[2 * k] = s_group[k];
      pairs[2 * k + 1] = s_cell[k];
    }
  }
  return OCTGRAV_OK;
}

static double splitmix_uniform(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  return static_cast<double>(z >> 11) * (1.0 / 9007199254740992.0);
}

}  // extern "C"

namespace {

constexpr int kTrainSteps = 512;  // training steps of one launch

// Bytes of an array of floats in a call's scratch.
size_t room(size_t floats) { return Scratch::room(4 * floats); }

}  // namespace

extern "C" {

int octgrav_mlp_grad(const float* params, const float* x, const float* target, int64_t n, float* grad, float* loss,
                     void* stream) {
  if (!params || !x || !target || n < 1 || n > (1 << 30) || !grad) return fail(OCTGRAV_ERR_ARG, "bad argument");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int B = static_cast<int>(n);
  const size_t nx = static_cast<size_t>(og::MLP_NF) * B, np = og::MLP_PART * static_cast<size_t>(og::mlp_blocks(B));
  Scratch S(st);
  int rc = S.reserve(2 * room(og::MLP_NPARAM) + room(nx) + room(B) + room(np) +
                     room(1));
  if (rc) return rc;
  float *w = S.take<float>(og::MLP_NPARAM), *g = S.take<float>(og::MLP_NPARAM), *dx = S.take<float>(nx), *dt = S.take<float>(B), *part = S.take<float>(np),
        *dl = S.take<float>(1);
  CUDA_TRY(cudaMemcpyAsync(w, params, 4 * og::MLP_NPARAM, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(dx, x, 4 * nx, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(dt, target, 4 * n, cudaMemcpyHostToDevice, st));
  cudaError_t e = og::mlp_gradient(w, dx, dt, B, part, g, dl, st);
  if (e != cudaSuccess) return fail(OCTGRAV_ERR_CUDA, "gradient kernel failed: %s", cudaGetErrorString(e));
  float l = 0;
  CUDA_TRY(cudaMemcpyAsync(grad, g, 4 * og::MLP_NPARAM, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpyAsync(&l, dl, 4, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  S.waited = true;
  if (loss) *loss = l;
  return OCTGRAV_OK;
}

int octgrav_mlp_train(const float* features, const float* labels, int64_t n, int steps, int batch, double lr,
                      uint64_t seed, float* record, float* final_loss, void* stream) {
  if (!features || !labels || !record || n < 2 || n > (1 << 30) || steps < 1 || batch < 1 || !(lr > 0))
    return fail(OCTGRAV_ERR_ARG, "bad argument");
  const int F = og::MLP_NF;
  // He-uniform initialisation from a counter-based generator
  std::vector<float> w(og::MLP_NPARAM, 0.f);
  uint64_t rs = seed;
  const int NH = og::MLP_NH;
  for (int k = 0; k < NH * F; ++k) w[k] = static_cast<float>((2 * splitmix_uniform(rs) - 1) * std::sqrt(6.0 / F));
  float* W2 = w.data() + NH * F + NH;
  for (int k = 0; k < NH * NH; ++k) W2[k] = static_cast<float>((2 * splitmix_uniform(rs) - 1) * std::sqrt(6.0 / NH));
  float* w3 = W2 + NH * NH + NH;
  for (int k = 0; k < NH; ++k) w3[k] = static_cast<float>((2 * splitmix_uniform(rs) - 1) * std::sqrt(3.0 / NH));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int B = static_cast<int>(std::min<int64_t>(batch, n));
  const size_t np = og::MLP_PART * static_cast<size_t>(og::mlp_blocks(B));
  const size_t nx = static_cast<size_t>(F) * n;
  Scratch S(st);
  int rc = S.reserve(3 * room(og::MLP_NPARAM) + room(nx) + 2 * room(n) +
                     room(np) + room(og::MLP_STD_FLOATS) + room(4 * F) +
                     room(2 * kTrainSteps) + room(2) + room(1));
  if (rc) return rc;
  float *dw = S.take<float>(og::MLP_NPARAM), *dm = S.take<float>(og::MLP_NPARAM), *dv = S.take<float>(og::MLP_NPARAM), *dx = S.take<float>(nx),
        *dlab = S.take<float>(n), *dy = S.take<float>(n), *part = S.take<float>(np), *dstd = S.take<float>(og::MLP_STD_FLOATS), *drec = S.take<float>(4 * F),
        *dcoef = S.take<float>(2 * kTrainSteps), *dbar = S.take<float>(2), *dl = S.take<float>(1);
  CUDA_TRY(cudaMemcpyAsync(dx, features, 4 * nx, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(dlab, labels, 4 * n, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemcpyAsync(dw, w.data(), 4 * og::MLP_NPARAM, cudaMemcpyHostToDevice, st));
  CUDA_TRY(cudaMemsetAsync(dm, 0, 2 * room(og::MLP_NPARAM), st));  // dm and dv follow each other
  {  // targets: log10 of the error label; inputs standardised per feature
    const cudaError_t e = og::mlp_standardise(dx, dlab, n, dstd, dy, drec, st);
    if (e != cudaSuccess) return fail(OCTGRAV_ERR_CUDA, "standardisation failed: %s", cudaGetErrorString(e));
  }
  // a launch for every 512 steps (a few milliseconds)
  std::vector<float2> coef(kTrainSteps);
  for (int k0 = 1; k0 <= steps; k0 += kTrainSteps) {
    const int nk = std::min(kTrainSteps, steps - k0 + 1);
    for (int k = 0; k < nk; ++k)
      coef[k] = make_float2(1.f / (1.f - powf(0.9f, static_cast<float>(k0 + k))),
                            1.f / (1.f - powf(0.999f, static_cast<float>(k0 + k))));
    CUDA_TRY(cudaMemcpyAsync(dcoef, coef.data(), sizeof(float2) * nk, cudaMemcpyHostToDevice, st));
    const cudaError_t e = og::mlp_train_steps(dw, dm, dv, dx, dy, static_cast<int>(n), B, k0, nk, seed,
                                              static_cast<float>(lr), reinterpret_cast<const float2*>(dcoef), part, dl,
                                              reinterpret_cast<int*>(dbar), st);
    if (e != cudaSuccess) return fail(OCTGRAV_ERR_CUDA, "training kernel failed: %s", cudaGetErrorString(e));
    int stuck = 0;
    CUDA_TRY(cudaMemcpyAsync(&stuck, reinterpret_cast<int*>(dbar) + 1, 4, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    if (stuck) return fail(OCTGRAV_ERR_TIMEOUT, "a training step's barrier timed out");
  }
  float l = 0, stats[4 * og::MLP_NF];
  CUDA_TRY(cudaMemcpyAsync(stats, drec, sizeof stats, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpyAsync(w.data(), dw, 4 * og::MLP_NPARAM, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpyAsync(&l, dl, 4, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  S.waited = true;
  // The range limits are the training extremes widened by kRangeMargin standard
  // deviations: an input equal to an extreme is in range however it is
  // rounded (several inputs take discrete values -- counts, cell sizes -- that
  // sit exactly on an extreme, and an FP32 and an FP64 evaluation of them
  // differ in the last bits).
  constexpr float kRangeMargin = 1e-3f;
  for (int i = 0; i < F; ++i) {
    record[i] = stats[i];
    record[12 + i] = stats[12 + i];
    record[24 + i] = stats[24 + i] - kRangeMargin;
    record[36 + i] = stats[36 + i] + kRangeMargin;
  }
  std::memcpy(record + 48, w.data(), 4 * og::MLP_NPARAM);
  if (final_loss) *final_loss = l;
  return OCTGRAV_OK;
}

}  // extern "C"
