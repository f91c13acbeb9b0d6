// sv_f32.cu -- the refinement network in FP32 on the CUDA cores, batched over the pairs of a
// call (conv_f32.cu, wgrad_f32.cu): packed weights, inference, the training forward (FP32, or
// the tensor-core form's with its saved activations converted) and the backward.
#include <algorithm>
#include <cstring>
#include <vector>

#include "sv_ctx.cuh"

namespace sv {

template <typename T>
cudaError_t launch_up4_bwd(const T* gU, const T* gx0, int W, int H, int w, int h, T* gc, cudaStream_t st);

namespace {

// Bytes of activations one group of pairs may hold: pairs beyond it run as further groups on
// the same workspace.  Where an allocation of a group fails, smaller groups are tried, down to one pair.
// A 1242 x 375 pair of the 32/64/128 net needs 134 MB; 2 GiB hold 15, more than fill the GPU.
constexpr size_t kGroupBytes = size_t(2) << 30;

// Pairs of a group: the largest z extent of a launch's grid.
constexpr int kGroupPairs = 65535;

// Bytes of weight-gradient slots a launch may use.  A slot is a copy of the layer's weights and a pair has
// up to 304 of them: 142 MB a 1242 x 375 pair for dec1 of the 32/64/128 net.  1 GiB holds 7, whose 1680
// chains fill the GPU several times over.
constexpr size_t kSlotBytes = size_t(1) << 30;

constexpr size_t pad32(size_t v) { return (v + 31) / 32 * 32; }

}  // namespace

// Plans the FP32 layers and their packed weights: FP32 contexts when they are created, BF16 contexts
// (which only train in FP32) at their first training call.
sv_status Ctx::f32_plan(cudaStream_t st) {
  auto src = [&](int l) { return F32Src{net.w_off(l), net.ks(l), net.cout(l), net.cin(l)}; };
  std::vector<F32PackDesc> descs;
  size_t total = 0;
  auto add = [&](F32Layer& l, int kind, int layer) { l = f32_plan_layer(kind, false, src(layer), descs, total); };
  auto add_grad = [&](int kind, int layer) { f32_g[layer] = f32_plan_layer(kind, true, src(layer), descs, total); };
  if (t1) {
    t1_plan_layers(t1_l, descs, total);
  } else {
    add(f32_l[L_ENC2], FK_S2, L_ENC2);
    add(f32_l[L_ENC3], FK_S2, L_ENC3);
    add(f32_l[L_MU], FK_P1, L_MU);
    add(f32_l[L_LV], FK_P1, L_LV);
    for (int l : {L_DEC1, L_DEC2, L_DEC3}) {
      if (cfg.precision == SV_FP32) {  // (a BF16 context decodes on the tensor cores)
        add(f32_l[l], FK_UP2, l);
        f32_t[l] = f32_l[l];  // the nine unsummed taps, also the summed form's edge weights
        f32_t[l].kind = FK_UP2X;
        f32_t[l].w[0] = f32_l[l].wb;
      }
      add_grad(FK_DUP2, l);
    }
    add_grad(FK_P1, L_MU);
    add_grad(FK_P1, L_LV);
    add_grad(FK_DS2, L_ENC3);
    add_grad(FK_DS2, L_ENC2);
  }
  size_t max_count = 0;
  for (auto& d : descs) max_count = std::max(max_count, d.count);
  sv_status s;
  if ((s = cuda(f32_w.ensure(total * sizeof(float)), "alloc packed FP32 weights"))) return s;
  if ((s = cuda(f32_descs.ensure(descs.size() * sizeof(F32PackDesc)), "alloc pack table"))) return s;
  if ((s = cuda(cudaMemcpyAsync(f32_descs.p, descs.data(), descs.size() * sizeof(F32PackDesc), cudaMemcpyHostToDevice,
                                st),
                "upload pack table")))
    return s;
  // The count says that the plan is there (f32_pack, the first training call): set once it is.
  f32_n_descs = (int)descs.size();
  f32_max_count = max_count;
  return SV_OK;
}

sv_status Ctx::f32_pack(cudaStream_t st) {
  if (f32_n_descs == 0) return SV_OK;
  LaunchScope ls(*this, "pack_f32", st);
  return cuda(launch_f32_pack((const F32PackDesc*)f32_descs.p, f32_n_descs, f32_max_count, (const float*)w32.p,
                              (float*)f32_w.p, st),
              "pack FP32 weights");
}

namespace {
// Job tables of one call, uploaded together.
struct Tables {
  std::vector<unsigned char> host;
  template <typename J>
  size_t put(const std::vector<J>& v) {
    const size_t o = (host.size() + 255) / 256 * 256, b = v.size() * sizeof(J);
    host.resize(o + b);
    if (b) memcpy(host.data() + o, v.data(), b);
    return o;
  }
};
}  // namespace

// Forward pass of pairs [0, n) whose tensors `t` are placed: the layers of the small network in
// order, one launch a layer.
sv_status Ctx::f32_forward(const sv_pair* pairs, int n, const F32Tensors* t, const int16_t* const* coarse_i,
                           const float* const* coarse_f, const float* const* eps, float* const* Y, cudaStream_t st) {
  const bool train = eps != nullptr;
  std::vector<F32Img> img(n);
  std::vector<F32Job> job[L_COUNT];
  std::vector<F32Lat> lat(train ? n : 0);
  int mH[4] = {0, 0, 0, 0}, mW[4] = {0, 0, 0, 0};
  size_t max_lat = 0;
  for (int i = 0; i < n; ++i) {
    const sv_pair& p = pairs[i];
    const Levels lv(p.height, p.width);
    for (int k = 0; k < 4; ++k) {
      mH[k] = std::max(mH[k], lv.H[k]);
      mW[k] = std::max(mW[k], lv.W[k]);
    }
    F32Img& m = img[i];
    m = F32Img{};
    m.L = p.left; m.pitch = p.pitch; m.W = p.width; m.H = p.height; m.w = p.width / 4; m.h = p.height / 4;
    m.coarse_i = coarse_i ? coarse_i[i] : nullptr;
    m.coarse_f = coarse_f ? coarse_f[i] : nullptr;
    m.e1 = t[i].e1; m.d3 = t[i].d3; m.Y = Y[i]; m.W1 = lv.W[1]; m.H1 = lv.H[1];
    auto J = [&](int l, const float* in, int li, float* out, int lo) {
      F32Job j{};
      j.in[0] = in; j.ic[0] = net.cin(l); j.out = out;
      j.Hi = lv.H[li]; j.Wi = lv.W[li]; j.Ho = lv.H[lo]; j.Wo = lv.W[lo];
      job[l].push_back(j);
    };
    J(L_ENC2, t[i].e1, 1, t[i].e2, 2);
    J(L_ENC3, t[i].e2, 2, t[i].e3, 3);
    J(L_MU, t[i].e3, 3, train ? t[i].mu : t[i].z, 3);
    if (train) J(L_LV, t[i].e3, 3, t[i].lv, 3);
    J(L_DEC1, t[i].z, 3, t[i].d1, 2);
    J(L_DEC2, t[i].d1, 2, t[i].d2, 1);
    J(L_DEC3, t[i].d2, 1, t[i].d3, 0);
    if (train) {
      F32Lat& q = lat[i];
      q = F32Lat{};
      q.mu = t[i].mu; q.lv = t[i].lv; q.eps = eps[i]; q.z = t[i].z;
      q.mu_copy = t[i].mu_out; q.lv_copy = t[i].lv_out; q.eps_copy = t[i].eps_copy;
      q.n = (size_t)lv.H[3] * lv.W[3] * net.lat;
      max_lat = std::max(max_lat, q.n);
    }
  }
  Tables tb;
  const size_t o_img = tb.put(img), o_lat = tb.put(lat);
  size_t o_job[L_COUNT];
  for (int l = 0; l < L_COUNT; ++l) o_job[l] = tb.put(job[l]);
  sv_status s;
  if ((s = cuda(f32_tab.ensure(tb.host.size()), "alloc FP32 tables"))) return s;
  if ((s = upload(f32_tab.p, tb.host.data(), tb.host.size(), "upload FP32 tables", st))) return s;
  const unsigned char* d = (const unsigned char*)f32_tab.p;
  const F32Img* d_img = (const F32Img*)(d + o_img);
  const float *W = (const float*)w32.p, *P = (const float*)f32_w.p;
  {
    LaunchScope ls(*this, "enc1", st);
    if ((s = cuda(launch_f32_enc1(d_img, n, mH[1], mW[1], W + net.w_off(L_ENC1), W + net.b_off(L_ENC1), net.enc[0], st),
                  "enc1")))
      return s;
  }
  auto conv = [&](int l, const char* name, int lo, int act) {
    LaunchScope ls(*this, name, st);
    const F32Layer& L = train && l >= L_DEC1 ? f32_t[l] : f32_l[l];
    return cuda(launch_f32_conv(L, (const F32Job*)(d + o_job[l]), n, mH[lo], mW[lo], P, W + net.b_off(l), act,
                                st),
                name);
  };
  if ((s = conv(L_ENC2, "enc2", 2, 1))) return s;
  if ((s = conv(L_ENC3, "enc3", 3, 1))) return s;
  if ((s = conv(L_MU, "latent", 3, 0))) return s;
  if (train) {
    if ((s = conv(L_LV, "latent", 3, 0))) return s;
    LaunchScope ls(*this, "latent", st);
    if ((s = cuda(launch_f32_reparam((const F32Lat*)(d + o_lat), n, max_lat, st), "reparameterisation"))) return s;
  }
  if ((s = conv(L_DEC1, "dec1", 2, 1))) return s;
  if ((s = conv(L_DEC2, "dec2", 1, 1))) return s;
  if ((s = conv(L_DEC3, "dec3", 0, 1))) return s;
  LaunchScope ls(*this, "final", st);
  return cuda(launch_f32_final(d_img, n, mH[0], mW[0], W + net.w_off(L_FINAL), W + net.b_off(L_FINAL), net.dec[2],
                               train, st),
              "final");
}

// Floats of the activations e1 e2 e3 z d1 d2 d3 of one pair, each padded to 128 bytes.
static void act_sizes(const NetDims& net, const Levels& lv, size_t out[7]) {
  const size_t P0 = (size_t)lv.H[0] * lv.W[0], P1 = (size_t)lv.H[1] * lv.W[1], P2 = (size_t)lv.H[2] * lv.W[2],
               P3 = (size_t)lv.H[3] * lv.W[3];
  const size_t v[7] = {P1 * net.enc[0], P2 * net.enc[1], P3 * net.enc[2], P3 * net.lat,
                       P2 * net.dec[0], P1 * net.dec[1], P0 * net.dec[2]};
  for (int k = 0; k < 7; ++k) out[k] = pad32(v[k]);
}

// After an allocation failed: releases the workspaces that the call can do without.  True if there was
// one (another try may succeed).
bool Ctx::give_back(std::initializer_list<DevBuf*> spare) {
  bool any = false;
  for (DevBuf* b : spare)
    if (b->p) {
      b->release();
      any = true;
    }
  if (any) err.clear();
  return any;
}

sv_status Ctx::f32_refine(const sv_pair* pairs, const int16_t* const* coarse, int n, float* const* out,
                          cudaStream_t st) {
  size_t budget = kGroupBytes;
  for (int i0 = 0; i0 < n;) {
    std::vector<F32Tensors> t;
    std::vector<size_t> ofs;
    size_t total = 0;
    int i1 = i0;
    for (; i1 < n && i1 - i0 < kGroupPairs; ++i1) {
      size_t sz[7], sum = 0;
      act_sizes(net, Levels(pairs[i1].height, pairs[i1].width), sz);
      for (size_t v : sz) sum += v;
      if (i1 > i0 && (total + sum) * sizeof(float) > budget) break;
      ofs.push_back(total);
      total += sum;
    }
    sv_status s;
    if ((s = cuda(f32_act.ensure(total * sizeof(float)), "alloc activations"))) {
      if (s != SV_ERR_OOM) return s;
      if (!give_back({&train_scratch, &wgrad_slots})) {
        if (i1 - i0 == 1) return s;
        budget = total * sizeof(float) / 2;
        err.clear();
      }
      continue;
    }
    for (int i = i0; i < i1; ++i) {
      size_t sz[7];
      act_sizes(net, Levels(pairs[i].height, pairs[i].width), sz);
      float* q = (float*)f32_act.p + ofs[i - i0];
      auto take = [&](int k) { float* r = q; q += sz[k]; return r; };
      F32Tensors x{};
      x.e1 = take(0); x.e2 = take(1); x.e3 = take(2); x.z = take(3); x.d1 = take(4); x.d2 = take(5); x.d3 = take(6);
      t.push_back(x);
    }
    if ((s = f32_forward(pairs + i0, i1 - i0, t.data(), coarse + i0, nullptr, nullptr, out + i0, st))) return s;
    i0 = i1;
  }
  return SV_OK;
}

// ---------------------------------------------------------------- training

// Places the decoder activations and the latent of every pair, which the backward needs, in train_saved
// and the mean head's own output in train_mu.
sv_status Ctx::train_save_alloc(const sv_pair* pairs, int n, void* const* mu, void* const* lv) {
  size_t total = 0, lat_total = 0;
  for (int i = 0; i < n; ++i) {
    size_t sz[7];
    act_sizes(net, Levels(pairs[i].height, pairs[i].width), sz);
    for (int k = 3; k < 7; ++k) total += sz[k];
    total += 2 * sz[3];  // lv, eps
    lat_total += sz[3];
  }
  sv_status s;
  if ((s = cuda(train_saved.ensure(std::max<size_t>(total, 32) * sizeof(float)), "alloc saved activations"))) return s;
  if ((s = cuda(train_mu.ensure(std::max<size_t>(lat_total, 32) * sizeof(float)), "alloc latent scratch"))) return s;
  train_t.assign(n, F32Tensors{});
  float *q = (float*)train_saved.p, *m = (float*)train_mu.p;
  for (int i = 0; i < n; ++i) {
    size_t sz[7];
    act_sizes(net, Levels(pairs[i].height, pairs[i].width), sz);
    auto take = [&](int k) { float* r = q; q += sz[k]; return r; };
    F32Tensors& t = train_t[i];
    t.z = take(3); t.d1 = take(4); t.d2 = take(5); t.d3 = take(6);
    t.lv = take(3); t.eps_copy = take(3);
    t.mu = m;
    m += sz[3];
    t.mu_out = mu ? (float*)mu[i] : nullptr;
    t.lv_out = lv ? (float*)lv[i] : nullptr;
  }
  return SV_OK;
}

// Places e1 .. e3 of a pair at q.
static void place_encoder(F32Tensors& t, float* q, const size_t sz[7]) {
  t.e1 = q;
  t.e2 = q + sz[0];
  t.e3 = q + sz[0] + sz[1];
}

// Keeps the encoder's activations for the backward (train_enc) where they fit.  Else the forward goes
// through groups of pairs whose encoder activations are let go, and the backward recomputes them as it does
// for the BF16 form: the same kernels, the same bits.
sv_status Ctx::f32_train_forward(const sv_pair* pairs, const void* const* coarse, const void* const* eps, int n,
                                 void* const* Y, void* const* mu, void* const* lv, cudaStream_t st) {
  sv_status s;
  while ((s = train_save_alloc(pairs, n, mu, lv)))
    if (s != SV_ERR_OOM || !give_back({&train_scratch, &wgrad_slots, &f32_act, &train_enc})) return s;
  size_t enc_total = 0;
  for (int i = 0; i < n; ++i) {
    size_t sz[7];
    act_sizes(net, Levels(pairs[i].height, pairs[i].width), sz);
    enc_total += sz[0] + sz[1] + sz[2];
  }
  while ((s = cuda(train_enc.ensure(enc_total * sizeof(float)), "alloc encoder activations")))
    if (s != SV_ERR_OOM || !give_back({&train_scratch, &wgrad_slots, &f32_act})) break;
  if (s && s != SV_ERR_OOM) return s;
  const bool keep = s == SV_OK;
  err.clear();
  if (keep) {
    float* q = (float*)train_enc.p;
    for (int i = 0; i < n; ++i) {
      size_t sz[7];
      act_sizes(net, Levels(pairs[i].height, pairs[i].width), sz);
      place_encoder(train_t[i], q, sz);
      q += sz[0] + sz[1] + sz[2];
    }
  }
  train_pairs.assign(pairs, pairs + n);
  train_coarse.assign(coarse, coarse + n);
  train_elem = sizeof(float);
  size_t budget = kGroupBytes;
  for (int i0 = 0; i0 < n;) {
    size_t total = 0;
    int i1 = i0;
    std::vector<F32Tensors> t;
    std::vector<size_t> ofs;
    for (; i1 < n && i1 - i0 < kGroupPairs; ++i1) {
      size_t sz[7];
      act_sizes(net, Levels(pairs[i1].height, pairs[i1].width), sz);
      const size_t sum = keep ? 0 : sz[0] + sz[1] + sz[2];
      if (i1 > i0 && (total + sum) * sizeof(float) > budget) break;
      t.push_back(train_t[i1]);
      ofs.push_back(total);
      total += sum;
    }
    if (!keep) {
      if ((s = cuda(f32_act.ensure(total * sizeof(float)), "alloc encoder activations"))) {
        if (s != SV_ERR_OOM || i1 - i0 == 1) return s;
        budget = total * sizeof(float) / 2;
        err.clear();
        continue;
      }
      for (int i = i0; i < i1; ++i) {
        size_t sz[7];
        act_sizes(net, Levels(pairs[i].height, pairs[i].width), sz);
        place_encoder(t[i - i0], (float*)f32_act.p + ofs[i - i0], sz);
      }
    }
    if ((s = f32_forward(pairs + i0, i1 - i0, t.data(), nullptr, (const float* const*)coarse + i0,
                         (const float* const*)eps + i0, (float* const*)Y + i0, st)))
      return s;
    i0 = i1;
  }
  train_ready = true;
  return SV_OK;
}

// Training forward of the BF16 form: the tensor-core encoder and decoder (BF16 operands, FP32
// accumulation), the training latent and the final conv in FP32.  The decoder activations and
// the latent are saved as FP32 for the FP32 backward.
sv_status Ctx::train_forward_bf16(const sv_pair* pairs, const void* const* coarse, const void* const* eps, int n,
                                  void* const* Y, void* const* mu, void* const* lv, cudaStream_t st) {
  sv_status s;
  if (f32_n_descs == 0 && ((s = f32_plan(st)) || (s = f32_pack(st)))) {
    f32_n_descs = 0;  // the next call plans and packs again
    return s;
  }
  auto fitted = [&](auto alloc) {  // (a backward's scratch is not needed before the next backward)
    sv_status r = alloc();
    if (r == SV_ERR_OOM && give_back({&train_scratch, &wgrad_slots})) r = alloc();
    return r;
  };
  if ((s = fitted([&] { return train_save_alloc(pairs, n, mu, lv); }))) return s;
  train_pairs.assign(pairs, pairs + n);
  train_coarse.assign(coarse, coarse + n);
  train_elem = sizeof(float);
  std::vector<float*> outs(n);
  for (int i = 0; i < n; ++i) outs[i] = (float*)Y[i];
  TcRun r;
  if ((s = fitted([&] { return tc_prepare(pairs, nullptr, n, outs.data(), r, (const float* const*)coarse); }))) return s;
  std::vector<size_t> e3_ofs(n);
  size_t e3_total = 0;
  TcTrainLatent tl{};
  tl.n = n;
  for (int i = 0; i < n; ++i) {
    e3_ofs[i] = e3_total;
    e3_total += pad32(tc_len[i][2]);
    tl.max_e3 = std::max(tl.max_e3, tc_len[i][2]);
  }
  if ((s = fitted([&] { return cuda(f32_act.ensure(e3_total * sizeof(float)), "alloc latent input"); }))) return s;
  std::vector<F32Cvt> cvt_e3(n), cvt_d;
  std::vector<F32Job> jm(n), jl(n);
  std::vector<F32Lat> lat(n);
  size_t max_d = 0;
  for (int i = 0; i < n; ++i) {
    const Levels lv_(pairs[i].height, pairs[i].width);
    auto bf = [&](int k) { return (const __nv_bfloat16*)tc_act[k].p + tc_off[i][k]; };
    F32Tensors& t = train_t[i];
    float* e3 = (float*)f32_act.p + e3_ofs[i];
    cvt_e3[i] = {bf(2), e3, tc_len[i][2]};
    float* dst[3] = {t.d1, t.d2, t.d3};
    for (int k = 0; k < 3; ++k) {
      cvt_d.push_back({bf(4 + k), dst[k], tc_len[i][4 + k]});
      max_d = std::max(max_d, tc_len[i][4 + k]);
    }
    F32Job j{};
    j.in[0] = e3; j.ic[0] = net.enc[2]; j.out = t.mu;
    j.Hi = j.Ho = lv_.H[3]; j.Wi = j.Wo = lv_.W[3];
    jm[i] = j;
    j.out = t.lv;
    jl[i] = j;
    F32Lat& q = lat[i];
    q = F32Lat{};
    q.mu = t.mu; q.lv = t.lv; q.eps = (const float*)eps[i]; q.z = t.z; q.z16 = (__nv_bfloat16*)bf(3);
    q.mu_copy = t.mu_out; q.lv_copy = t.lv_out; q.eps_copy = t.eps_copy;
    q.n = (size_t)lv_.H[3] * lv_.W[3] * net.lat;
    tl.max_lat = std::max(tl.max_lat, q.n);
    tl.maxH3 = std::max(tl.maxH3, lv_.H[3]);
    tl.maxW3 = std::max(tl.maxW3, lv_.W[3]);
  }
  Tables tb;
  const size_t o_tc = tb.put(r.host), o_e3 = tb.put(cvt_e3), o_m = tb.put(jm), o_l = tb.put(jl), o_lat = tb.put(lat),
               o_d = tb.put(cvt_d);
  if ((s = cuda(tc_tables.ensure(tb.host.size()), "alloc tables"))) return s;
  if ((s = upload(tc_tables.p, tb.host.data(), tb.host.size(), "upload tables", st))) return s;
  const unsigned char* d = (const unsigned char*)tc_tables.p;
  tl.e3 = (const F32Cvt*)(d + o_e3);
  tl.mu = (const F32Job*)(d + o_m);
  tl.lv = (const F32Job*)(d + o_l);
  tl.lat = (const F32Lat*)(d + o_lat);
  if ((s = tc_launch(r, d + o_tc, st, &tl))) return s;
  {
    LaunchScope ls(*this, "save_bf16_to_f32", st);
    if ((s = cuda(launch_f32_convert((const F32Cvt*)(d + o_d), (int)cvt_d.size(), max_d, st), "save activations")))
      return s;
  }
  train_ready = true;
  return SV_OK;
}

// Backward of pairs grouped so that a group's gradients stay within the activation budget; every
// layer is one launch over the group's pairs.
sv_status Ctx::f32_backward(const void* const* gY, const void* const* gmu_ext, const void* const* glv_ext,
                            float* gparams, void* const* gcoarse, cudaStream_t st) {
  sv_status s;
  const int n = (int)train_pairs.size();
  const float *W = (const float*)w32.p, *P = (const float*)f32_w.p;
  auto GW = [&](int l) { return gparams + net.w_off(l); };
  auto GB = [&](int l) { return gparams + net.b_off(l); };
  if ((s = cuda(cudaMemsetAsync(gparams, 0, net.count() * sizeof(float), st), "zero grads"))) return s;
  bool recompute = n > 0 && train_t[0].e1 == nullptr;
  bool want_coarse = false;
  for (int i = 0; gcoarse && i < n; ++i) want_coarse |= gcoarse[i] != nullptr;
  // floats of one pair's gradients: e1 e2 e3 (and the recomputed activations), z, mu, lv, d1 d2 d3, x0
  auto pair_floats = [&](int i, size_t sz[7]) {
    const Levels lv(train_pairs[i].height, train_pairs[i].width);
    act_sizes(net, lv, sz);
    size_t t = 2 * sz[3];
    for (int k = 0; k < 7; ++k) t += sz[k];
    if (recompute) t += sz[0] + sz[1] + sz[2];
    if (want_coarse) t += pad32((size_t)2 * lv.H[0] * lv.W[0]);
    return t;
  };
  size_t budget = kGroupBytes, slot_budget = kSlotBytes;
  for (int i0 = 0; i0 < n;) {
    size_t total = 0;
    int i1 = i0;
    for (; i1 < n && i1 - i0 < kGroupPairs; ++i1) {
      size_t sz[7];
      const size_t f = pair_floats(i1, sz);
      if (i1 > i0 && (total + f) * sizeof(float) > budget) break;
      total += f;
    }
    const int m = i1 - i0;
    // The group again: with the forward's workspace given back, half the budget, or for a single pair
    // the encoder's kept activations given back too.
    auto again = [&] {
      if (give_back({&f32_act})) return true;
      if (m > 1) {
        budget = total * sizeof(float) / 2;
      } else {
        if (recompute || !give_back({&train_enc})) return false;
        for (F32Tensors& t : train_t) t.e1 = t.e2 = t.e3 = nullptr;
        recompute = true;
      }
      train_scratch.release();
      err.clear();
      return true;
    };
    if ((s = cuda(train_scratch.ensure(total * sizeof(float)), "alloc backward scratch"))) {
      if (s == SV_ERR_OOM && (give_back({&wgrad_slots}) || again())) continue;
      return s;
    }
    float* q = (float*)train_scratch.p;
    std::vector<F32Img> img(m);
    std::vector<F32Lat> lat(m);
    std::vector<F32Job> gj[L_COUNT], fj[L_COUNT];  // input gradients, recomputed layers
    std::vector<F32WJob> wj[L_COUNT];
    std::vector<float*> ge1s(m), gx0s(m);
    int mH[4] = {0, 0, 0, 0}, mW[4] = {0, 0, 0, 0};
    size_t max_lat = 0;
    for (int i = i0; i < i1; ++i) {
      const sv_pair& p = train_pairs[i];
      const Levels lv(p.height, p.width);
      size_t sz[7];
      pair_floats(i, sz);
      for (int k = 0; k < 4; ++k) {
        mH[k] = std::max(mH[k], lv.H[k]);
        mW[k] = std::max(mW[k], lv.W[k]);
      }
      auto take = [&](size_t c) { float* r = q; q += c; return r; };
      F32Tensors t = train_t[i];
      if (recompute) { t.e1 = take(sz[0]); t.e2 = take(sz[1]); t.e3 = take(sz[2]); }
      float *ge1 = take(sz[0]), *ge2 = take(sz[1]), *ge3 = take(sz[2]), *gz = take(sz[3]), *gmu = take(sz[3]),
            *glv = take(sz[3]), *gd1 = take(sz[4]), *gd2 = take(sz[5]), *gd3 = take(sz[6]);
      gx0s[i - i0] = want_coarse ? take(pad32((size_t)2 * lv.H[0] * lv.W[0])) : nullptr;
      ge1s[i - i0] = ge1;
      F32Img& g = img[i - i0];
      g = F32Img{};
      g.L = p.left; g.pitch = p.pitch; g.W = p.width; g.H = p.height; g.w = p.width / 4; g.h = p.height / 4;
      g.coarse_f = (const float*)train_coarse[i];
      g.e1 = t.e1; g.d3 = t.d3; g.gY = (const float*)gY[i]; g.gd3 = gd3; g.ge1 = ge1;
      g.W1 = lv.W[1]; g.H1 = lv.H[1];
      F32Lat& la = lat[i - i0];
      la = F32Lat{};
      la.lv = t.lv; la.eps = t.eps_copy; la.gz = gz; la.gmu = gmu; la.glv = glv;
      la.gmu_ext = gmu_ext ? (const float*)gmu_ext[i] : nullptr;
      la.glv_ext = glv_ext ? (const float*)glv_ext[i] : nullptr;
      la.n = (size_t)lv.H[3] * lv.W[3] * net.lat;
      max_lat = std::max(max_lat, la.n);
      // input gradient of layer l: from g (level lo) to gin (level li), masked by act
      auto G = [&](int l, const float* gg, int lo, const float* act, float* gin, int li) {
        F32Job j{};
        j.in[0] = gg; j.ic[0] = net.cout(l); j.mask = act; j.out = gin;
        j.Hi = lv.H[lo]; j.Wi = lv.W[lo]; j.Ho = lv.H[li]; j.Wo = lv.W[li];
        gj[l].push_back(j);
      };
      auto Wg = [&](int l, const float* gg, int lo, const float* x, int li) {
        wj[l].push_back({gg, x, lv.H[li], lv.W[li], lv.H[lo], lv.W[lo], 0, 0});
      };
      G(L_DEC3, gd3, 0, t.d2, gd2, 1);
      G(L_DEC2, gd2, 1, t.d1, gd1, 2);
      G(L_DEC1, gd1, 2, nullptr, gz, 3);
      Wg(L_FINAL, nullptr, 0, t.d3, 0);  // (g is the image table's gY)
      Wg(L_ENC1, ge1, 1, nullptr, 0);    // (x is built from the images)
      Wg(L_DEC3, gd3, 0, t.d2, 1);
      Wg(L_DEC2, gd2, 1, t.d1, 2);
      Wg(L_DEC1, gd1, 2, t.z, 3);
      G(L_MU, gmu, 3, t.e3, ge3, 3);
      G(L_LV, glv, 3, t.e3, ge3, 3);
      Wg(L_MU, gmu, 3, t.e3, 3);
      Wg(L_LV, glv, 3, t.e3, 3);
      G(L_ENC3, ge3, 3, t.e2, ge2, 2);
      Wg(L_ENC3, ge3, 3, t.e2, 2);
      G(L_ENC2, ge2, 2, t.e1, ge1, 1);
      Wg(L_ENC2, ge2, 2, t.e1, 1);
      if (recompute) {
        auto Fw = [&](int l, const float* in, int li, float* out, int lo) {
          F32Job j{};
          j.in[0] = in; j.ic[0] = net.cin(l); j.out = out;
          j.Hi = lv.H[li]; j.Wi = lv.W[li]; j.Ho = lv.H[lo]; j.Wo = lv.W[lo];
          fj[l].push_back(j);
        };
        Fw(L_ENC2, t.e1, 1, t.e2, 2);
        Fw(L_ENC3, t.e2, 2, t.e3, 3);
      }
    }
    static const int kinds[L_COUNT] = {FK_WENC1, FK_S2, FK_S2, FK_P1, FK_P1, FK_UP2, FK_UP2, FK_UP2, FK_WFINAL};
    F32WPlan wp[L_COUNT];
    for (;;) {
      size_t slots = 0;
      bool split = false;  // the largest ranges can be cut further
      for (int l = 0; l < L_COUNT; ++l) {
        wp[l] = f32_wgrad_plan(kinds[l], net.cout(l), net.cin(l), wj[l], slot_budget / sizeof(float));
        slots = std::max(slots, wp[l].slot_floats);
      }
      for (const F32WPlan& w : wp) split = split || (w.slot_floats == slots && (int)w.ranges.size() < m);
      s = cuda(wgrad_slots.ensure(slots * sizeof(float)), "alloc weight-gradient slots");
      if (s != SV_ERR_OOM || !split) break;
      slot_budget = std::min(slot_budget, slots * sizeof(float)) / 2;
      err.clear();
    }
    if (s) {
      if (s == SV_ERR_OOM && again()) continue;
      return s;
    }
    Tables tb;
    size_t og[L_COUNT], of[L_COUNT], ow[L_COUNT];
    const size_t o_img = tb.put(img), o_lat = tb.put(lat);
    for (int l = 0; l < L_COUNT; ++l) {
      og[l] = tb.put(gj[l]);
      of[l] = tb.put(fj[l]);
      ow[l] = tb.put(wj[l]);
    }
    if ((s = cuda(f32_tab.ensure(tb.host.size()), "alloc FP32 tables"))) return s;
    if ((s = upload(f32_tab.p, tb.host.data(), tb.host.size(), "upload FP32 tables", st))) return s;
    const unsigned char* d = (const unsigned char*)f32_tab.p;
    const F32Img* d_img = (const F32Img*)(d + o_img);
    float* sl = (float*)wgrad_slots.p;
#define SV_BW(name, expr)                   \
  {                                         \
    LaunchScope _ls(*this, name, st);       \
    if ((s = cuda((expr), name))) return s; \
  }
    auto dgrad = [&](int l, int li, int act = 0) {
      return launch_f32_conv(f32_g[l], (const F32Job*)(d + og[l]), m, mH[li], mW[li], P, nullptr, act, st);
    };
    auto wgrad = [&](int l) {
      const F32WJob* j = (const F32WJob*)(d + ow[l]);
      if (l == L_FINAL || l == L_ENC1) return launch_f32_edge_wgrad(wp[l], d_img, j, GW(l), GB(l), sl, st);
      return launch_f32_wgrad(wp[l], j, GW(l), GB(l), sl, st);
    };
    SV_BW("bwd_final_dgrad", launch_f32_final_dgrad(d_img, m, mH[0], mW[0], W + net.w_off(L_FINAL), net.dec[2], st));
    SV_BW("bwd_final_wgrad", wgrad(L_FINAL));
    SV_BW("bwd_dec3_dgrad", dgrad(L_DEC3, 1));
    SV_BW("bwd_dec3_wgrad", wgrad(L_DEC3));
    SV_BW("bwd_dec2_dgrad", dgrad(L_DEC2, 2));
    SV_BW("bwd_dec2_wgrad", wgrad(L_DEC2));
    SV_BW("bwd_dec1_dgrad", dgrad(L_DEC1, 3));
    SV_BW("bwd_dec1_wgrad", wgrad(L_DEC1));
    SV_BW("bwd_latent", launch_f32_latent_bwd((const F32Lat*)(d + o_lat), m, max_lat, st));
    if (recompute) {  // the encoder's FP32 activations (the tensor-core forward kept BF16 ones)
      SV_BW("recompute_enc1", launch_f32_enc1(d_img, m, mH[1], mW[1], W + net.w_off(L_ENC1), W + net.b_off(L_ENC1),
                                              net.enc[0], st));
      SV_BW("recompute_enc2", launch_f32_conv(f32_l[L_ENC2], (const F32Job*)(d + of[L_ENC2]), m, mH[2], mW[2], P,
                                              W + net.b_off(L_ENC2), 1, st));
      SV_BW("recompute_enc3", launch_f32_conv(f32_l[L_ENC3], (const F32Job*)(d + of[L_ENC3]), m, mH[3], mW[3], P,
                                              W + net.b_off(L_ENC3), 1, st));
    }
    SV_BW("bwd_mu_dgrad", dgrad(L_MU, 3));
    SV_BW("bwd_lv_dgrad", dgrad(L_LV, 3, 8));
    SV_BW("bwd_mu_wgrad", wgrad(L_MU));
    SV_BW("bwd_lv_wgrad", wgrad(L_LV));
    SV_BW("bwd_enc3_dgrad", dgrad(L_ENC3, 2));
    SV_BW("bwd_enc3_wgrad", wgrad(L_ENC3));
    SV_BW("bwd_enc2_dgrad", dgrad(L_ENC2, 1));
    SV_BW("bwd_enc2_wgrad", wgrad(L_ENC2));
    SV_BW("bwd_enc1_wgrad", wgrad(L_ENC1));
    for (int i = i0; want_coarse && i < i1; ++i) {
      if (!gcoarse[i]) continue;
      const sv_pair& p = train_pairs[i];
      const Levels lv(p.height, p.width);
      // through the network input (channel U / 256) and the residual Y = U + ...
      SV_BW("bwd_enc1_dgrad", launch_enc1_dgrad(ge1s[i - i0], lv.H[1], lv.W[1], net.enc[0], W + net.w_off(L_ENC1),
                                                p.height, p.width, gx0s[i - i0], st));
      SV_BW("bwd_upsample4", launch_up4_bwd<float>((const float*)gY[i], gx0s[i - i0], p.width, p.height, p.width / 4,
                                                   p.height / 4, (float*)gcoarse[i], st));
    }
#undef SV_BW
    i0 = i1;
  }
  return SV_OK;
}

}  // namespace sv
