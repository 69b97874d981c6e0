// C ABI, workspace planner and launch sequences of the attention coupling branch (Eq. 1).
// See include/revffn_attn.h for the contract of every entry point.  Included at the end of
// revffn_moe.cu: it uses that file's launch accounting, error macros and GEMM back ends.
//
// Attention core: with bf16 weights and heads of 128 both directions run as fused tcgen05 kernels
// (flash_attn.cuh) that never write the score matrix.  The CUDA-core cross-check path, fp32 weights
// and heads of another width materialise it: scores = Q K^T as one grouped product over all heads
// (fp32), a row kernel turns it into the causal softmax P (operand type), O = P V is a second grouped
// product; then dP = dO V^T, the row kernel for dS, dV = P^T dO and dK = dS^T Q as grouped
// weight-gradient-style products, dQ = dS K.
#pragma once

#include "../../include/revffn_attn.h"
#include "flash_attn.cuh"

namespace revffn {

struct AttnLayout {
  Buf status, rows_total, tile_group, group_off, cs, cs_t, n12, r12, u12, raw, qh, kh, vh, sc, p, oh, o, a;
  size_t fwd_bytes = 0;
  Buf dyb, da, dob, doh, ds, dqh, dkh, dvh, dq, dkv, du12, dn12, part, npart, lse_d;
  size_t bwd_bytes = 0;
  int T = 0, h = 0, hd = 0, d_kv = 0, Sp = 0, n_tiles = 0, groups = 0, strips = 0;
  int64_t rows = 0, kv_rows = 0;
};

static AttnLayout plan_attn(const revffn_attn_desc& D) {
  AttnLayout L;
  const size_t ts = D.weight_dtype == REVFFN_BF16 ? 2 : 4;
  const int64_t B = D.batch, S = D.seq_len, d = D.d_model, h = d / 2, nh = D.n_heads, nkv = D.n_kv_heads;
  const int64_t T = B * S, hd = d / nh, dkv = nkv * hd, Sp = round_up(S, ROW_PAD);
  L.T = (int)T; L.h = (int)h; L.hd = (int)hd; L.d_kv = (int)dkv; L.Sp = (int)Sp;
  L.rows = B * nh * Sp; L.kv_rows = B * nkv * Sp;
  L.n_tiles = (int)(L.rows / ROW_PAD);
  L.groups = (int)(B * nkv);
  L.strips = (int)ceil_div(T > 0 ? T : 1, STRIP);
  size_t off = 0;
  auto take = [&](Buf& b, size_t bytes) {
    b.off = off; b.bytes = bytes;
    off += (size_t)round_up((int64_t)(bytes > 0 ? bytes : 1), 256);
  };
  take(L.status, 256);
  take(L.rows_total, 256);
  take(L.tile_group, (size_t)L.n_tiles * 4);
  take(L.group_off, (size_t)(L.groups + 1) * 4);
  take(L.cs, (size_t)S * (hd / 2) * 8);
  // the fused kernels' own table, [pair, position]: a backward call may take up what a call on the other back end left
  take(L.cs_t, D.weight_dtype == REVFFN_BF16 && hd == FA_HD ? (size_t)S * (hd / 2) * 8 : 0);
  take(L.n12, (size_t)2 * T * h * ts);
  take(L.r12, (size_t)2 * T * 4);
  take(L.u12, (size_t)2 * T * d * ts);
  take(L.raw, (size_t)T * d * 4);
  take(L.qh, (size_t)L.rows * hd * ts);
  take(L.kh, (size_t)L.kv_rows * hd * ts);
  take(L.vh, (size_t)L.kv_rows * hd * ts);
  take(L.sc, (size_t)L.rows * Sp * 4);
  take(L.p, (size_t)L.rows * Sp * ts);
  take(L.oh, (size_t)L.rows * hd * ts);
  take(L.o, (size_t)T * d * ts);
  take(L.a, (size_t)T * d * ts);
  L.fwd_bytes = off;
  take(L.dyb, (size_t)T * h * ts);
  take(L.da, (size_t)T * d * ts);
  take(L.dob, (size_t)T * d * ts);
  take(L.doh, (size_t)L.rows * hd * ts);
  take(L.ds, (size_t)L.rows * Sp * ts);
  take(L.dqh, (size_t)L.rows * hd * 4);
  take(L.dkh, (size_t)L.kv_rows * hd * 4);
  take(L.dvh, (size_t)L.kv_rows * hd * 4);
  take(L.dq, (size_t)T * d * ts);
  take(L.dkv, (size_t)T * 2 * dkv * ts);
  take(L.du12, (size_t)2 * T * d * ts);
  take(L.dn12, (size_t)2 * T * h * 4);
  take(L.part, (size_t)L.strips * (d + 2 * dkv) * 4);
  take(L.npart, norm_part_floats(2 * T, (int)h) * 4);
  take(L.lse_d, (size_t)L.rows * 8);
  L.bwd_bytes = off;
  return L;
}

static int validate_attn_desc(const revffn_attn_desc* D) {
  if (!D) return REVFFN_ERR_NULL;
  if (D->batch < 0 || D->seq_len < 1 || D->d_model <= 0 || (D->d_model & 1)) return REVFFN_ERR_SHAPE;
  if (D->n_heads < 1 || D->d_model % D->n_heads) return REVFFN_ERR_SHAPE;
  if (D->n_kv_heads < 1 || D->n_heads % D->n_kv_heads) return REVFFN_ERR_SHAPE;
  if (D->weight_dtype != REVFFN_F32 && D->weight_dtype != REVFFN_BF16) return REVFFN_ERR_SHAPE;
  const int h = D->d_model / 2, hd = D->d_model / D->n_heads;
  if (hd & 1) return REVFFN_ERR_SHAPE;
  if (D->weight_dtype == REVFFN_BF16) {
    if (h % 128 || D->d_model % 128 || hd % 128) return REVFFN_ERR_SHAPE;
  } else if (h % 8 || D->d_model % 8 || hd % 8) {
    return REVFFN_ERR_SHAPE;
  }
  if (!(D->rope_theta > 0.f)) return REVFFN_ERR_SHAPE;
  if (D->flags & ~(REVFFN_FLAG_FORCE_SIMT | REVFFN_FLAG_REUSE_ACTIVATIONS | REVFFN_FLAG_SINGLE_STREAM)) return REVFFN_ERR_UNSUPPORTED;
  if (D->ld_stream < h || (D->ld_stream % 4)) return REVFFN_ERR_ALIGN;
  const int64_t Sp = round_up(D->seq_len, ROW_PAD);
  if ((int64_t)D->batch * D->n_heads * Sp > (int64_t)1 << 30 || (int64_t)D->batch * D->seq_len > (int64_t)1 << 28)
    return REVFFN_ERR_SHAPE;
  return REVFFN_OK;
}

static int validate_attn_weights(const revffn_attn_weights* w) {
  if (!w) return REVFFN_ERR_NULL;
  if (!w->w_up || !w->w_down || !w->w_q || !w->w_k || !w->w_v || !w->w_o) return REVFFN_ERR_NULL;
  const void* ps[] = {w->norm_gamma, w->w_up, w->w_down, w->w_q, w->w_k, w->w_v, w->w_o, w->b_q, w->b_k, w->b_v};
  for (const void* p : ps)
    if (p && !aligned16(p)) return REVFFN_ERR_ALIGN;
  return REVFFN_OK;
}

template <typename T>
struct ACtx {
  revffn_attn_desc D;
  revffn_attn_weights W;
  AttnLayout L;
  char* ws;
  cudaStream_t st;
  int* status;             // device status word: the workspace's own, or that of the block call this one is part of
  bool clear;              // this call clears it
  Overlap* ov = nullptr;   // non-null: the second stream is in use for this call
  bool tc;
  bool fused() const { return std::is_same<T, bf16>::value && tc && L.hd == FA_HD; }      // attention core as tcgen05 kernels
  // what is queued on `to` from now on follows everything queued on `from` so far (no-op without the second stream)
  int order(cudaStream_t from, cudaStream_t to) const { return ov ? ov->order(from, to) : REVFFN_OK; }
  ACtx on_side() const { ACtx c = *this; if (ov) c.st = ov->side; return c; }
  template <typename U> U* p(const Buf& b) const { return reinterpret_cast<U*>(ws + b.off); }
};

template <typename T>
static int a_gemm(const ACtx<T>& c, GemmProblem p, int tag) {
  p.status = c.status;
  ProfScope ps(tag, c.st);
  if constexpr (std::is_same<T, bf16>::value) {
    if (c.tc) return launch_gemm_tc(p, c.st);
  }
  return launch_gemm_simt<T>(p, c.st) == cudaSuccess ? REVFFN_OK : REVFFN_ERR_CUDA;
}

// What a pass needs before its first product: rotary table, zeroed padding rows of the head-major buffers, cleared
// status word; on the materialising path also the tables of the grouped products.  tables: the rotary table and the
// q / k / v padding (a gradient pass that reuses the key/value side finds them in place); d_o: its padding too.
// The two back ends have rotary tables of their own, and only the materialising path has tables of groups.  Where both can
// run (bf16, heads of 128) the slow one sees to both: it writes the fused kernels' table too, and makes its own
// tables again when it takes up a key/value side, which the fused path may have left.
template <typename T>
static int a_setup(const ACtx<T>& c, bool tables, bool d_o) {
  const revffn_attn_desc& D = c.D;
  const AttnLayout& L = c.L;
  cudaStream_t st = c.st;
  const int per = L.Sp - D.seq_len;
  if constexpr (std::is_same<T, bf16>::value) {
    if (c.fused()) {
      AttnPads pads;
      pads.n = 0;
      auto pad = [&](const Buf& b, int n_heads) {
        if (per == 0) return;
        pads.buf[pads.n] = c.template p<bf16>(b);
        pads.rows[pads.n++] = D.batch * n_heads * per;
      };
      if (tables) { pad(L.qh, D.n_heads); pad(L.kh, D.n_kv_heads); pad(L.vh, D.n_kv_heads); }
      if (d_o) pad(L.doh, D.n_heads);
      int64_t n = tables ? (int64_t)D.seq_len * 64 : 0;
      for (int j = 0; j < pads.n; ++j) n += (int64_t)pads.rows[j] * 16;
      if (n == 0 && !c.clear) return REVFFN_OK;
      ProfScope ps(TG_A_TABLES, st);
      CK(launch_k(attn_setup_kernel, (unsigned)ceil_div(std::max<int64_t>(n, 1), 256), 256, 0, st, D.seq_len, L.Sp,
                  (double)D.rope_theta, tables ? c.template p<float2>(L.cs_t) : nullptr, pads, c.clear ? c.status : nullptr));
      return REVFFN_OK;
    }
  }
  if (c.clear) CK(launch_k(clear_status_kernel, 1, 1, 0, st, c.status));
  const bool both = std::is_same<T, bf16>::value && L.hd == FA_HD;
  if (tables && both) {
    ProfScope ps(TG_A_TABLES, st);
    AttnPads none;
    none.n = 0;
    CK(launch_k(attn_setup_kernel, (unsigned)ceil_div((int64_t)D.seq_len * 64, 256), 256, 0, st, D.seq_len, L.Sp, (double)D.rope_theta,
                c.template p<float2>(L.cs_t), none, nullptr));
  }
  if (tables || both) {
    const int n_tab = L.n_tiles > L.groups + 1 ? L.n_tiles : L.groups + 1;
    { ProfScope ps(TG_A_TABLES, st);
    CK(launch_k(attn_tables_kernel, (unsigned)ceil_div(n_tab, 256), 256, 0, st, L.n_tiles, L.Sp / ROW_PAD,
                D.n_heads / D.n_kv_heads, L.groups, (D.n_heads / D.n_kv_heads) * L.Sp, c.template p<int32_t>(L.tile_group),
                c.template p<int32_t>(L.group_off), c.template p<int32_t>(L.rows_total)));
    }
    { ProfScope ps(TG_A_TABLES, st);
    CK(launch_k(rope_table_kernel, (unsigned)ceil_div((int64_t)D.seq_len * (L.hd / 2), 256), 256, 0, st, D.seq_len, L.hd,
                (double)D.rope_theta, c.template p<float2>(L.cs)));
    }
  }
  if (per != 0) {
    if (tables) {
      CK(cudaMemsetAsync(c.ws + L.qh.off, 0, L.qh.bytes, st));
      CK(cudaMemsetAsync(c.ws + L.kh.off, 0, L.kh.bytes, st));
      CK(cudaMemsetAsync(c.ws + L.vh.off, 0, L.vh.bytes, st));
    }
    if (d_o) CK(cudaMemsetAsync(c.ws + L.doh.off, 0, L.doh.bytes, st));
  }
  return REVFFN_OK;
}

// n = Norm(x), u = n W_up^T for one stream (side 0: query stream, side 1: key/value stream).
template <typename T>
static int a_norm_up(const ACtx<T>& c, const float* x, int side) {
  const revffn_attn_desc& D = c.D;
  const AttnLayout& L = c.L;
  const int Tn = L.T, d = D.d_model, h = L.h;
  T* n = c.template p<T>(L.n12) + (int64_t)side * Tn * h;
  { ProfScope ps(TG_NORM, c.st);
  launch_k(rmsnorm_fwd_kernel<T>, (unsigned)ceil_div((int64_t)Tn * 32, 128), 128, 0, c.st, 
      x, D.ld_stream, c.W.norm_gamma, D.norm_eps, 0, Tn, h, n, c.template p<float>(L.r12) + (int64_t)side * Tn);
  }
  CK(cudaGetLastError());
  GemmProblem p = blank_problem();
  p.M = Tn; p.N = d; p.K = h;
  p.A = n; p.lda = h;
  p.B0 = c.W.w_up; p.ldb = h;
  p.epilogue = EPI_STORE; p.C = c.template p<T>(L.u12) + (int64_t)side * Tn * d; p.ldc = d;
  return a_gemm(c, p, TG_PUP);
}

// heads = to_heads(u W^T + bias [, rotated])
template <typename T>
static int a_project(const ACtx<T>& c, int side, const void* W, const float* bias, int n, bool rotate, T* heads) {
  const revffn_attn_desc& D = c.D;
  const AttnLayout& L = c.L;
  const int Tn = L.T, d = D.d_model;
  GemmProblem p = blank_problem();
  p.M = Tn; p.N = n * L.hd; p.K = d;
  p.A = c.template p<T>(L.u12) + (int64_t)side * Tn * d; p.lda = d;
  p.B0 = W; p.ldb = d;
  if constexpr (std::is_same<T, bf16>::value) {
    if (c.fused()) {
      // bias, rotation and the head-major layout happen in the product's epilogue: no fp32 round trip
      p.epilogue = EPI_HEADS; p.C = heads;
      p.hm_bias = bias; p.hm_cs = rotate ? c.template p<float2>(L.cs_t) : nullptr; p.hm_S = D.seq_len; p.hm_Sp = L.Sp;
      return a_gemm(c, p, TG_A_QKV);
    }
  }
  p.epilogue = EPI_STORE; p.out_f32 = 1; p.C = c.template p<float>(L.raw); p.ldc = n * L.hd;
  CKR(a_gemm(c, p, TG_A_QKV));
  { ProfScope ps(TG_A_HEADS, c.st);
  CK((launch_to_heads<float, T>(c.template p<float>(L.raw), (int64_t)n * L.hd, bias,
                                rotate ? c.template p<float2>(L.cs) : nullptr, Tn, D.seq_len, L.Sp, n, L.hd, heads, c.st)));
  }
  return REVFFN_OK;
}

template <typename T>
static GemmProblem a_grouped_rows(const ACtx<T>& c) {
  const AttnLayout& L = c.L;
  GemmProblem p = blank_problem();
  p.M = (int)L.rows;
  p.group_mode = GROUP_M; p.n_groups = L.groups; p.b_group_stride = (int64_t)L.Sp * L.hd;
  p.group_off = c.template p<int32_t>(L.group_off); p.tile_group = c.template p<int32_t>(L.tile_group);
  p.rows_total = c.template p<int32_t>(L.rows_total);
  return p;
}

// O (token-major) from the head-major q, k, v.  need_p: the backward pass reads P afterwards, so the score
// matrix is materialised; otherwise the tcgen05 back end runs the attention core as one kernel.
template <typename T>
static int a_core(const ACtx<T>& c, bool need_p, bool grad = false) {
  const revffn_attn_desc& D = c.D;
  const AttnLayout& L = c.L;
  if constexpr (std::is_same<T, bf16>::value) {
    if (c.fused() && !need_p) {
      ProfScope ps(TG_A_FLASH, c.st);
      return launch_flash_fwd(c.template p<bf16>(L.qh), c.template p<bf16>(L.kh), c.template p<bf16>(L.vh), D.batch,
                              D.n_heads, D.n_kv_heads, D.seq_len, L.Sp, c.template p<bf16>(L.o), D.d_model,
                              grad ? c.template p<bf16>(L.doh) : nullptr, grad ? c.template p<float>(L.lse_d) : nullptr,
                              c.status, c.st);
    }
  }
  {
    GemmProblem p = a_grouped_rows(c);   // scores = Q K^T
    p.N = L.Sp; p.K = L.hd;
    p.A = c.template p<T>(L.qh); p.lda = L.hd;
    p.B0 = c.template p<T>(L.kh); p.ldb = L.hd;
    p.epilogue = EPI_STORE; p.out_f32 = 1; p.C = c.template p<float>(L.sc); p.ldc = L.Sp;
    CKR(a_gemm(c, p, TG_A_SCORES));
  }
  { ProfScope ps(TG_A_SOFTMAX, c.st);
  launch_k(softmax_causal_kernel<T>, (unsigned)ceil_div(L.rows * 32, 256), 256, 0, c.st, 
      c.template p<float>(L.sc), D.seq_len, L.Sp, 1.4426950408889634f / sqrtf((float)L.hd), L.rows, c.template p<T>(L.p));
  }
  CK(cudaGetLastError());
  {
    GemmProblem p = a_grouped_rows(c);   // O = P V
    p.N = L.hd; p.K = L.Sp;
    p.A = c.template p<T>(L.p); p.lda = L.Sp;
    p.B0 = c.template p<T>(L.vh); p.ldb = L.hd; p.b_mn_major = 1;
    p.epilogue = EPI_STORE; p.C = c.template p<T>(L.oh); p.ldc = L.hd;
    CKR(a_gemm(c, p, TG_A_PV));
  }
  { ProfScope ps(TG_A_HEADS, c.st);
  CK((launch_from_heads<T, T>(c.template p<T>(L.oh), nullptr, 1.f, L.T, D.seq_len, L.Sp, D.n_heads, L.hd,
                              c.template p<T>(L.o), D.d_model, 0, c.st)));
  }
  return REVFFN_OK;
}

// a = O W_o^T
template <typename T>
static int a_wo(const ACtx<T>& c) {
  const int d = c.D.d_model;
  GemmProblem p = blank_problem();
  p.M = c.L.T; p.N = d; p.K = d;
  p.A = c.template p<T>(c.L.o); p.lda = d;
  p.B0 = c.W.w_o; p.ldb = d;
  p.epilogue = EPI_STORE; p.C = c.template p<T>(c.L.a); p.ldc = d;
  return a_gemm(c, p, TG_A_WO);
}

// P_down fused with the coupling: out = resid + sign * (a W_down^T)
template <typename T>
static int a_couple(const ACtx<T>& c, const float* resid, float sign, float* out) {
  const int d = c.D.d_model;
  GemmProblem p = blank_problem();
  p.M = c.L.T; p.N = c.L.h; p.K = d;
  p.A = c.template p<T>(c.L.a); p.lda = d;
  p.B0 = c.W.w_down; p.ldb = d;
  p.epilogue = EPI_COUPLE; p.resid = resid; p.ld_resid = c.D.ld_stream; p.resid_sign = sign;
  p.C = out; p.ldc = c.D.ld_stream;
  return a_gemm(c, p, TG_PDOWN);
}

// Keys and values, on the fused path as one product with two matrices: of few heads each alone fills half of the GPU (4 heads at
// 4291 tokens: 34 pair tiles each for 74 pairs; attention step 963 -> 950 us, four d = 512 blocks 1579 -> 1521).  Its tiles are up to
// 256 columns, two heads, which must not lie in both matrices; an odd number of heads keeps two launches.
template <typename T>
static int a_keys_values(const ACtx<T>& c) {
  const AttnLayout& L = c.L;
  if constexpr (std::is_same<T, bf16>::value) {
    if (c.fused() && L.d_kv % 256 == 0) {
      GemmProblem p = blank_problem();
      p.M = L.T; p.N = 2 * L.d_kv; p.K = c.D.d_model;
      p.A = c.template p<T>(L.u12) + (int64_t)L.T * c.D.d_model; p.lda = c.D.d_model;
      p.B0 = c.W.w_k; p.B1 = c.W.w_v; p.ldb = c.D.d_model;
      p.epilogue = EPI_HEADS; p.C = c.template p<T>(L.kh); p.C1 = c.template p<T>(L.vh); p.hm_split = L.d_kv;
      p.hm_bias = c.W.b_k; p.hm_bias1 = c.W.b_v; p.hm_cs = c.template p<float2>(L.cs_t); p.hm_S = c.D.seq_len; p.hm_Sp = L.Sp;
      return a_gemm(c, p, TG_A_QKV);
    }
  }
  CKR(a_project(c, 1, c.W.w_k, c.W.b_k, c.D.n_kv_heads, true, c.template p<T>(L.kh)));
  return a_project(c, 1, c.W.w_v, c.W.b_v, c.D.n_kv_heads, false, c.template p<T>(L.vh));
}

template <typename T>
static int a_kv_side(const ACtx<T>& c, const float* x2) {
  CKR(a_norm_up(c, x2, 1));
  return a_keys_values(c);
}

// Query side up to the core's operands: norm, P_up, rotated q.
template <typename T>
static int a_query(const ACtx<T>& c, const float* x1) {
  CKR(a_norm_up(c, x1, 0));
  return a_project(c, 0, c.W.w_q, c.W.b_q, c.D.n_heads, true, c.template p<T>(c.L.qh));
}

// Forward pass: both streams are known at once, so the norm and P_up run over the 2T rows together.  The keys and
// values are projected on the second stream beside the queries.
template <typename T>
static int a_forward(const ACtx<T>& c, const float* x1, const float* x2, float* y1) {
  const revffn_attn_desc& D = c.D;
  const AttnLayout& L = c.L;
  const ACtx<T> cs = c.on_side();
  CKR(a_setup(c, true, false));
  { ProfScope ps(TG_NORM, c.st);
  CK(launch_k(rmsnorm2_fwd_kernel<T>, (unsigned)ceil_div((int64_t)2 * L.T * 32, 128), 128, 0, c.st, x1, x2, D.ld_stream,
              c.W.norm_gamma, D.norm_eps, L.T, L.h, c.template p<T>(L.n12), c.template p<float>(L.r12)));
  }
  {
    GemmProblem p = blank_problem();
    p.M = 2 * L.T; p.N = D.d_model; p.K = L.h;
    p.A = c.template p<T>(L.n12); p.lda = L.h;
    p.B0 = c.W.w_up; p.ldb = L.h;
    p.epilogue = EPI_STORE; p.C = c.template p<T>(L.u12); p.ldc = D.d_model;
    CKR(a_gemm(c, p, TG_PUP));
  }
  CKR(c.order(c.st, cs.st));
  CKR(a_keys_values(cs));
  CKR(a_project(c, 0, c.W.w_q, c.W.b_q, D.n_heads, true, c.template p<T>(L.qh)));
  CKR(c.order(cs.st, c.st));
  CKR(a_core(c, false));
  CKR(a_wo(c));
  return a_couple(c, x1, 1.f, y1);
}

template <typename T>
static int a_inverse(const ACtx<T>& c, const float* y1, const float* x2, float* x1, int n_iter) {
  const AttnLayout& L = c.L;
  if (n_iter == 0) {
    if (c.clear) CK(launch_k(clear_status_kernel, 1, 1, 0, c.st, c.status));
    if (x1 != y1) {
      ++g_prof.launches;
      CK(launch_k(copy_stream_kernel, (unsigned)ceil_div((int64_t)L.T * L.h, 4 * 256), 256, 0, c.st, y1, c.D.ld_stream, L.T,
                  L.h, x1, c.D.ld_stream));
    }
    return REVFFN_OK;
  }
  const ACtx<T> cs = c.on_side();
  CKR(a_setup(c, true, false));
  CKR(c.order(c.st, cs.st));
  CKR(a_kv_side(cs, x2));                  // beside the first iteration's query side
  const float* cur = y1;
  for (int it = 0; it < n_iter; ++it) {
    CKR(a_query(c, cur));
    if (it == 0) CKR(c.order(cs.st, c.st));
    CKR(a_core(c, false));
    CKR(a_wo(c));
    CKR(a_couple(c, y1, -1.f, x1));
    cur = x1;
  }
  return REVFFN_OK;
}

template <typename T>
static int a_backward(const ACtx<T>& c, const float* x1, const float* x2, const float* dy1, float* dx1, float* dx2,
                      const revffn_attn_grads& G) {
  const revffn_attn_desc& D = c.D;
  const AttnLayout& L = c.L;
  const int Tn = L.T, d = D.d_model, h = L.h, hd = L.hd, dkv = L.d_kv, Sp = L.Sp;
  const int acc = G.accumulate ? 1 : 0;
  cudaStream_t st = c.st;
  const ACtx<T> cs = c.on_side();

  // out2: second output of a product whose M is two stacked gradients.  Gradients of few tiles are split over K as in the MoE
  // branch; the partial sums take the score matrix's place, which the fused core does not write, where they fit in it.
  auto wgrad = [&](const ACtx<T>& on, float* out, int M, int N, const void* A, int64_t lda, int a_col0, const void* B, int64_t ldb,
                   int K, float* out2 = nullptr) -> int {
    GemmProblem p = blank_problem();
    p.M = M; p.N = N; p.K = K;
    p.a_mn_major = 1; p.b_mn_major = 1;
    p.A = A; p.lda = lda; p.a_col0 = a_col0;
    p.B0 = B; p.ldb = ldb;
    p.epilogue = EPI_WGRAD; p.accumulate = acc;
    p.C = out; p.ldc = N;
    if (out2) { p.C2 = out2; p.split_m = M / 2; }
    int n_split = 1;
    if constexpr (std::is_same<T, bf16>::value) {
      if (on.fused()) n_split = wgrad_splits(M, N, K, L.sc.bytes);
    }
    if (n_split <= 1) return a_gemm(on, p, TG_A_WGRAD);
    const int64_t count = (int64_t)M * N;
    p.group_mode = GROUP_K; p.n_groups = n_split;
    p.C = on.template p<float>(L.sc); p.C2 = nullptr; p.split_m = 0; p.c_group_stride = count; p.accumulate = 0;
    CKR(a_gemm(on, p, TG_A_WGRAD));
    ProfScope ps(TG_A_WGRAD, on.st);
    CK(launch_k(splitk_reduce_kernel<T>, (unsigned)ceil_div(count, 4 * 256), 256, 0, on.st, on.template p<float>(L.sc), n_split, count, out,
                out2, out2 ? count / 2 : count, acc, nullptr, nullptr, UpdRule{}, nullptr, nullptr));
    return REVFFN_OK;
  };
  auto dgrad = [&](const ACtx<T>& on, int tag, int M, int N, int K, const void* A, int64_t lda, const void* W, int64_t ldw, void* C,
                   bool f32) -> int {
    GemmProblem p = blank_problem();   // C = A W  with W stored [K, N]
    p.M = M; p.N = N; p.K = K;
    p.A = A; p.lda = lda;
    p.B0 = W; p.ldb = ldw; p.b_mn_major = 1;
    p.epilogue = EPI_STORE; p.out_f32 = f32 ? 1 : 0; p.C = C; p.ldc = N;
    return a_gemm(on, p, tag);
  };

  // Recompute the branch's intermediates (Sec. 3.1: nothing was cached).
  // REUSE: an inverse call (at least one iteration) on this workspace with the same x2 and weights has left the
  // tables and the key/value side (n2, u2, k, v head-major) behind; only the query side is evaluated again.
  // tcgen05 back end: the attention core runs fused in both directions and P is never written;
  // otherwise the score matrix is materialised and the gradient pass reads P from memory.
  // The upstream gradient's way down to dO needs none of it: it runs on the second stream beside the query side.
  const bool reuse_kv = (D.flags & REVFFN_FLAG_REUSE_ACTIVATIONS) != 0;
  const bool fused = c.fused();
  CKR(a_setup(c, !reuse_kv, true));
  CKR(c.order(st, cs.st));
  { ProfScope ps(TG_CAST, cs.st);
  CK(launch_k(cast_stream_kernel<T>, (unsigned)ceil_div((int64_t)Tn * h, 4 * 256), 256, 0, cs.st, dy1, D.ld_stream, Tn, h,
              c.template p<T>(L.dyb)));
  }
  CKR(dgrad(cs, TG_A_DGRAD, Tn, d, h, c.template p<T>(L.dyb), h, c.W.w_down, d, c.template p<T>(L.da), false));
  if (fused) {
    GemmProblem p = blank_problem();   // dO = da W_o, written head-major by the product's epilogue
    p.M = Tn; p.N = d; p.K = d;
    p.A = c.template p<T>(L.da); p.lda = d;
    p.B0 = c.W.w_o; p.ldb = d; p.b_mn_major = 1;
    p.epilogue = EPI_HEADS; p.C = c.template p<T>(L.doh); p.hm_S = D.seq_len; p.hm_Sp = Sp;
    CKR(a_gemm(cs, p, TG_A_DGRAD));
  } else {
    CKR(dgrad(cs, TG_A_DGRAD, Tn, d, d, c.template p<T>(L.da), d, c.W.w_o, d, c.template p<T>(L.dob), false));
    { ProfScope ps(TG_A_HEADS, cs.st);
    CK((launch_to_heads<T, T>(c.template p<T>(L.dob), d, nullptr, nullptr, Tn, D.seq_len, Sp, D.n_heads, hd,
                              c.template p<T>(L.doh), cs.st)));
    }
  }
  if (!reuse_kv) CKR(a_kv_side(c, x2));
  CKR(a_query(c, x1));
  CKR(c.order(cs.st, st));              // the fused core reads dO: it leaves the rows' statistics for the two kernels below
  CKR(a_core(c, !fused, fused));

  // attention core backward
  if (fused) {
    if constexpr (std::is_same<T, bf16>::value) {
      CKR(c.order(st, cs.st));
      { ProfScope ps(TG_A_FLASH, st);
      // the two launches also undo the rotation and write dq and dk|dv token-major in the operand type
      CKR(launch_flash_bwd(c.template p<bf16>(L.qh), c.template p<bf16>(L.kh), c.template p<bf16>(L.vh),
                           c.template p<bf16>(L.doh), c.template p<float>(L.lse_d), c.template p<float2>(L.cs_t), D.batch,
                           D.n_heads, D.n_kv_heads, D.seq_len, Sp, c.template p<bf16>(L.dq), d, c.template p<bf16>(L.dkv),
                           2 * (int64_t)dkv, dkv, c.status, st, cs.st));
      ++g_prof.launches;
      }
    }
  } else {
    {
      GemmProblem p = a_grouped_rows(c);   // dP = dO V^T
      p.N = Sp; p.K = hd;
      p.A = c.template p<T>(L.doh); p.lda = hd;
      p.B0 = c.template p<T>(L.vh); p.ldb = hd;
      p.epilogue = EPI_STORE; p.out_f32 = 1; p.C = c.template p<float>(L.sc); p.ldc = Sp;
      CKR(a_gemm(c, p, TG_A_DP));
    }
    { ProfScope ps(TG_A_SOFTMAX, st);
    CK(launch_k(dsoftmax_causal_kernel<T>, (unsigned)ceil_div(L.rows * 32, 256), 256, 0, st, c.template p<T>(L.p),
                c.template p<float>(L.sc), D.seq_len, Sp, 1.f / sqrtf((float)hd), L.rows, c.template p<T>(L.ds)));
    }
    auto kv_grad = [&](const T* A, const T* Bm, float* out) -> int {
      GemmProblem p = blank_problem();   // out[g] = A_g^T B_g over the query rows of key/value group g
      p.M = Sp; p.N = hd; p.K = (int)L.rows;
      p.a_mn_major = 1; p.b_mn_major = 1;
      p.A = A; p.lda = Sp;
      p.B0 = Bm; p.ldb = hd;
      p.epilogue = EPI_WGRAD; p.accumulate = 0;
      p.C = out; p.ldc = hd; p.c_group_stride = (int64_t)Sp * hd;
      p.group_mode = GROUP_K; p.n_groups = L.groups; p.group_off = c.template p<int32_t>(L.group_off);
      return a_gemm(c, p, TG_A_DKV);
    };
    CKR(kv_grad(c.template p<T>(L.p), c.template p<T>(L.doh), c.template p<float>(L.dvh)));    // dV = P^T dO
    CKR(kv_grad(c.template p<T>(L.ds), c.template p<T>(L.qh), c.template p<float>(L.dkh)));    // dK = dS^T Q
    {
      GemmProblem p = a_grouped_rows(c);   // dQ = dS K
      p.N = hd; p.K = Sp;
      p.A = c.template p<T>(L.ds); p.lda = Sp;
      p.B0 = c.template p<T>(L.kh); p.ldb = hd; p.b_mn_major = 1;
      p.epilogue = EPI_STORE; p.out_f32 = 1; p.C = c.template p<float>(L.dqh); p.ldc = hd;
      CKR(a_gemm(c, p, TG_A_DQ));
    }
    // back to token-major; the rotation is undone by its transpose
    { ProfScope ps(TG_A_HEADS, st);
    CK((launch_from_heads<float, T>(c.template p<float>(L.dqh), c.template p<float2>(L.cs), -1.f, Tn, D.seq_len, Sp,
                                    D.n_heads, hd, c.template p<T>(L.dq), d, 0, st)));
    }
    { ProfScope ps(TG_A_HEADS, st);
    CK((launch_from_heads<float, T>(c.template p<float>(L.dkh), c.template p<float2>(L.cs), -1.f, Tn, D.seq_len, Sp,
                                    D.n_kv_heads, hd, c.template p<T>(L.dkv), 2 * (int64_t)dkv, 0, st)));
    }
    { ProfScope ps(TG_A_HEADS, st);
    CK((launch_from_heads<float, T>(c.template p<float>(L.dvh), nullptr, 1.f, Tn, D.seq_len, Sp, D.n_kv_heads, hd,
                                    c.template p<T>(L.dkv), 2 * (int64_t)dkv, dkv, st)));
    }
    CKR(c.order(st, cs.st));
  }

  // Input gradients on the caller's stream; every weight gradient is a leaf and goes to the second one (dq is already
  // there, dk | dv are ordered in).
  const T* u1 = c.template p<T>(L.u12);
  const T* u2 = u1 + (int64_t)Tn * d;
  T* du1 = c.template p<T>(L.du12);
  T* du2 = du1 + (int64_t)Tn * d;
  CKR(c.order(cs.st, st));
  CKR(c.order(st, cs.st));
  CKR(dgrad(c, TG_A_DGRAD, Tn, d, d, c.template p<T>(L.dq), d, c.W.w_q, d, du1, false));
  {
    GemmProblem p = blank_problem();   // dU2 = dK W_k + dV W_v
    p.M = Tn; p.N = d; p.K = 2 * dkv;
    p.A = c.template p<T>(L.dkv); p.lda = 2 * (int64_t)dkv;
    p.B0 = c.W.w_k; p.B1 = c.W.w_v; p.ldb = d; p.b_mn_major = 1; p.concat = CONCAT_K;
    p.epilogue = EPI_STORE; p.C = du2; p.ldc = d;
    CKR(a_gemm(c, p, TG_A_DGRAD));
  }
  if (G.w_down) {
    CKR(a_wo(cs));                     // a = O W_o^T is wanted for this gradient only
    CKR(wgrad(cs, G.w_down, h, d, c.template p<T>(L.dyb), h, 0, c.template p<T>(L.a), d, Tn));
  }
  if (G.w_o) CKR(wgrad(cs, G.w_o, d, d, c.template p<T>(L.da), d, 0, c.template p<T>(L.o), d, Tn));
  if (G.w_q) CKR(wgrad(cs, G.w_q, d, d, c.template p<T>(L.dq), d, 0, u1, d, Tn));
  // dk | dv is one buffer and both gradients read u2: one product where both are wanted (on the CUDA cores it has one output)
  if (G.w_k && G.w_v && c.tc) {
    CKR(wgrad(cs, G.w_k, 2 * dkv, d, c.template p<T>(L.dkv), 2 * (int64_t)dkv, 0, u2, d, Tn, G.w_v));
  } else {
    if (G.w_k) CKR(wgrad(cs, G.w_k, dkv, d, c.template p<T>(L.dkv), 2 * (int64_t)dkv, 0, u2, d, Tn));
    if (G.w_v) CKR(wgrad(cs, G.w_v, dkv, d, c.template p<T>(L.dkv), 2 * (int64_t)dkv, dkv, u2, d, Tn));
  }
  {
    ColSegs<T> s;
    int n = 0, cols = 0;
    auto seg = [&](const T* X, int64_t ld, int width, float* out) {
      if (!out) return;
      cols += width;
      s.X[n] = X; s.ld[n] = ld; s.end[n] = cols; s.out[n++] = out;
    };
    seg(c.template p<T>(L.dq), d, d, G.b_q);
    seg(c.template p<T>(L.dkv), 2 * (int64_t)dkv, dkv, G.b_k);
    seg(c.template p<T>(L.dkv) + dkv, 2 * (int64_t)dkv, dkv, G.b_v);
    for (int i = n; i < 3; ++i) { s.X[i] = nullptr; s.ld[i] = 0; s.end[i] = cols; s.out[i] = nullptr; }
    if (n > 0) {
      { ProfScope ps(TG_A_BIAS, cs.st);
      CK(launch_k(colsum_segs_partial_kernel<T>, dim3((unsigned)ceil_div(cols, 4 * 128), (unsigned)L.strips), 128, 0, cs.st, s, Tn,
                  cols, STRIP, c.template p<float>(L.part)));
      }
      { ProfScope ps(TG_A_BIAS, cs.st);
      CK(launch_k(colsum_segs_final_kernel<T>, (unsigned)ceil_div(cols, COLSUM_FINAL_COLS), 256, 0, cs.st,
                  c.template p<float>(L.part), L.strips, cols, acc, s));
      }
    }
  }

  // P_up and the norm, both streams at once: their rows are independent and share the weights
  CKR(dgrad(c, TG_DN, 2 * Tn, h, d, du1, d, c.W.w_up, h, c.template p<float>(L.dn12), true));
  if (G.w_up) {
    CKR(c.order(st, cs.st));
    CKR(wgrad(cs, G.w_up, d, h, du1, d, 0, c.template p<T>(L.n12), h, 2 * Tn));
  }
  const float* dn1 = c.template p<float>(L.dn12);
  const float* r1 = c.template p<float>(L.r12);
  const NormBwdRows s0 = {dn1, x1, r1, dy1, dx1}, s1 = {dn1 + (int64_t)Tn * h, x2, r1 + Tn, dx2, dx2};
  CKR(norm_backward(st, s0, s1, 2, D.ld_stream, c.W.norm_gamma, 0, Tn, h, G.norm_gamma, acc, c.template p<float>(L.npart)));
  return c.order(cs.st, st);           // the caller's stream ends after the weight gradients too
}

enum APass { APASS_FWD = 3, APASS_INV = 4, APASS_BWD = 5 };

template <typename T>
static int a_dispatch(APass pass, const revffn_attn_desc& D, const revffn_attn_weights& W, const AttnLayout& L, void* ws,
                      cudaStream_t st, const float* in1, const float* x2, const float* dy1, float* out1, float* dx2,
                      int n_iter, const revffn_attn_grads* G, int* status) {
  ACtx<T> c;
  c.D = D; c.W = W; c.L = L; c.ws = reinterpret_cast<char*>(ws); c.st = st;
  g_prof.pass = (int)pass;
  c.tc = std::is_same<T, bf16>::value && !(D.flags & REVFFN_FLAG_FORCE_SIMT);
  c.status = status ? status : c.template p<int>(L.status);
  c.clear = status == nullptr;
  if (c.tc) CKR(tc_prepare());
  SideStream side;
  if (c.fused() && !g_prof.on && !(D.flags & REVFFN_FLAG_SINGLE_STREAM)) CKR(side.take(st));
  c.ov = side.lane;
  if (L.T == 0) {
    if (c.clear) CK(launch_k(clear_status_kernel, 1, 1, 0, st, c.status));
    return REVFFN_OK;
  }
  if (pass == APASS_FWD) return a_forward(c, in1, x2, out1);
  if (pass == APASS_INV) return a_inverse(c, in1, x2, out1, n_iter);
  return a_backward(c, in1, x2, dy1, out1, dx2, *G);
}

static int a_entry(APass pass, const revffn_attn_desc* desc, const revffn_attn_weights* w, const float* in1,
                   const float* x2, const float* dy1, float* out1, float* dx2, int n_iter,
                   const revffn_attn_grads* grads, void* ws, size_t ws_bytes, void* cuda_stream, int* status = nullptr) {
  CKR(validate_attn_desc(desc));
  CKR(validate_attn_weights(w));
  if (!ws) return REVFFN_ERR_NULL;
  if (n_iter < 0) return REVFFN_ERR_SHAPE;
  const bool bwd = pass == APASS_BWD;
  if (bwd && !grads) return REVFFN_ERR_NULL;
  if ((int64_t)desc->batch * desc->seq_len > 0 && (!in1 || !x2 || !out1 || (bwd && (!dy1 || !dx2)))) return REVFFN_ERR_NULL;
  if (!aligned16(in1) || !aligned16(x2) || !aligned16(dy1) || !aligned16(out1) || !aligned16(dx2) ||
      (reinterpret_cast<uintptr_t>(ws) & 255u))
    return REVFFN_ERR_ALIGN;
  if (grads) {
    const float* gs[] = {grads->norm_gamma, grads->w_up, grads->w_down, grads->w_q, grads->w_k, grads->w_v,
                         grads->w_o, grads->b_q, grads->b_k, grads->b_v};
    for (const float* g : gs)
      if (g && !aligned16(g)) return REVFFN_ERR_ALIGN;
  }
  AttnLayout L = plan_attn(*desc);
  if (ws_bytes < (bwd ? L.bwd_bytes : L.fwd_bytes)) return REVFFN_ERR_WORKSPACE;
  CKR(check_device());
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  if (desc->weight_dtype == REVFFN_BF16)
    return a_dispatch<bf16>(pass, *desc, *w, L, ws, st, in1, x2, dy1, out1, dx2, n_iter, grads, status);
  return a_dispatch<float>(pass, *desc, *w, L, ws, st, in1, x2, dy1, out1, dx2, n_iter, grads, status);
}

}  // namespace revffn

extern "C" {

int revffn_attn_workspace_size(const revffn_attn_desc* desc, size_t* fwd_bytes, size_t* bwd_bytes) {
  int r = revffn::validate_attn_desc(desc);
  if (r != REVFFN_OK) return r;
  revffn::AttnLayout L = revffn::plan_attn(*desc);
  if (fwd_bytes) *fwd_bytes = L.fwd_bytes;
  if (bwd_bytes) *bwd_bytes = L.bwd_bytes;
  return REVFFN_OK;
}

int revffn_attn_forward(const revffn_attn_desc* desc, const revffn_attn_weights* w, const float* x1, const float* x2,
                        float* y1, void* ws, size_t ws_bytes, void* cuda_stream) {
  return revffn::a_entry(revffn::APASS_FWD, desc, w, x1, x2, nullptr, y1, nullptr, 0, nullptr, ws, ws_bytes, cuda_stream);
}

int revffn_attn_inverse(const revffn_attn_desc* desc, const revffn_attn_weights* w, const float* y1, const float* x2,
                        float* x1, int32_t n_iter, void* ws, size_t ws_bytes, void* cuda_stream) {
  if (n_iter > 1 && x1 == y1) return REVFFN_ERR_UNSUPPORTED;
  return revffn::a_entry(revffn::APASS_INV, desc, w, y1, x2, nullptr, x1, nullptr, n_iter, nullptr, ws, ws_bytes,
                         cuda_stream);
}

int revffn_attn_backward(const revffn_attn_desc* desc, const revffn_attn_weights* w, const float* x1, const float* x2,
                         const float* dy1, float* dx1, float* dx2_inout, const revffn_attn_grads* grads, void* ws,
                         size_t ws_bytes, void* cuda_stream) {
  return revffn::a_entry(revffn::APASS_BWD, desc, w, x1, x2, dy1, dx1, dx2_inout, 0, grads, ws, ws_bytes, cuda_stream);
}

int revffn_attn_status(const void* ws, void* cuda_stream, int32_t* device_status) {
  return revffn_moe_status(ws, cuda_stream, device_status);
}

}  // extern "C"
