// The launch sequence of the base-model forward and what each kernel touches before its dependency wait.
//
// Every kernel of the forward is launched programmatically dependent on its predecessor: it may start while the
// kernel in front is still running, and it executes griddepcontrol.wait before it touches what that kernel writes.
// Every kernel also releases its own dependents only AFTER its own wait, and no CTA leaves without having waited (a launch whose
// CTAs all had would be complete while the kernel in front runs).  So when kernel i runs, kernel i - 2 and
// everything older is complete, and kernel i may read, ahead of its wait, any buffer whose youngest writer is at
// least two launches older.  This file states, per kernel, what it writes and what it reads ahead of its wait;
// launch_order_violations() checks the rule over the cyclic layer sequence, and the host controller steps
// through the same table while it launches (forward_rows), so that the table cannot drift from the code.
// An attention that takes two launches (a rest of items, the second window of a wide tree) is one entry: the second one reads what is complete when
// the first one runs, and waits for that one at its end.
#include <stdio.h>
#include <string.h>

#include "cerb_internal.cuh"

namespace cerb {

namespace {

// buffers (bits)
enum : unsigned {
  B_X = 1u << 0,       // residual stream (fp32)
  B_XN = 1u << 1,      // norm output = GEMM input
  B_PART = 1u << 2,    // fp32 partial slots of the last GEMM
  B_Q = 1u << 3,       // rotated queries
  B_KV = 1u << 4,      // this step's tree slots of the K/V pools
  B_ATTN = 1u << 5,    // attention output
  B_ACT = 1u << 6,     // SwiGLU output
  B_HIDDEN = 1u << 7,  // final-norm output
  B_STATE = 1u << 8,   // per-sequence state the step starts from: lengths, live node counts (written before the forward)
  B_CONST = 1u << 9,   // never written during a forward: weights, gains, tree arrays, page table, rotation table,
                       // committed (prefix) K/V
};

struct Entry {
  int id;
  const char* name;
  unsigned writes;
  unsigned prewait_reads;
};

// The launches of one layer, then the tail.  Ids are what forward_rows announces, in this order.
const Entry kSetActive = {LO_SET_ACTIVE, "set_active / gate (live node counts)", B_STATE, 0};
const Entry kNormAttn = {LO_NORM_ATTN, "fused_norm (embedding or residual add, attention norm)", B_X | B_XN, B_X | B_CONST};
const Entry kQkv = {LO_GEMM_QKV, "gemm qkv", B_PART, B_CONST};
const Entry kRope = {LO_ROPE, "rope_append", B_Q | B_KV, B_STATE | B_CONST};
const Entry kAttn = {LO_ATTN, "tree attention", B_ATTN, B_STATE | B_CONST};
const Entry kWo = {LO_GEMM_WO, "gemm wo", B_PART, B_CONST};
const Entry kNormMlp = {LO_NORM_MLP, "fused_norm (residual add, MLP norm)", B_X | B_XN, B_X | B_CONST};
const Entry kGu = {LO_GEMM_GU, "gemm gate-up", B_PART, B_CONST};
const Entry kSwiglu = {LO_SWIGLU, "swiglu", B_ACT, 0};
const Entry kDown = {LO_GEMM_DOWN, "gemm down", B_PART, B_CONST};
const Entry kNormFinal = {LO_NORM_FINAL, "fused_norm (residual add, final norm)", B_X | B_HIDDEN, B_X | B_CONST};
const Entry kLm = {LO_GEMM_LM, "gemm lm_head", B_PART, B_CONST};
const Entry kArgmax = {LO_ARGMAX, "argmax_rows", 0, 0};
// SwiGLU in the gate-up GEMM's epilogue: that GEMM writes the activations itself.  RoPE + cache append in the QKV GEMM's.
const Entry kGuSwiglu = {LO_GEMM_GU, "gemm gate-up + swiglu epilogue", B_PART | B_ACT, B_CONST};
const Entry kQkvRope = {LO_GEMM_QKV, "gemm qkv + rope / append epilogue", B_PART | B_Q | B_KV, B_CONST};
// The residual add in the O and down GEMMs' epilogues: the norms then read nothing ahead of their wait (the
// embedding gather in front of the first layer writes it, as ever).
const Entry kWoAdd = {LO_GEMM_WO, "gemm wo + residual add epilogue", B_PART | B_X, B_CONST};
const Entry kDownAdd = {LO_GEMM_DOWN, "gemm down + residual add epilogue", B_PART | B_X, B_CONST};
const Entry kNormAttnRead = {LO_NORM_ATTN, "row_norm (embedding; attention norm)", B_X | B_XN, 0};
const Entry kNormMlpRead = {LO_NORM_MLP, "row_norm (MLP norm)", B_XN, 0};
const Entry kNormFinalRead = {LO_NORM_FINAL, "row_norm (final norm)", B_HIDDEN, 0};

// The norms in the GEMMs that read them, which then read the residual stream after their wait; the embedding gather with the
// first attention norm stays, in front of the layers.
const Entry kNormEmbed = {LO_NORM_ATTN, "row_norm (embedding, attention norm)", B_X | B_XN, 0};
const Entry kQkvNorm = {LO_GEMM_QKV, "gemm norm + qkv + rope / append epilogue", B_Q | B_KV, B_CONST};
const Entry kGuNorm = {LO_GEMM_GU, "gemm norm + gate-up + swiglu epilogue", B_ACT, B_CONST};

// Variants 0, 1, 2 and 4 are the steps of 9 to 128 rows (bf16): a tile per SM finishes SwiGLU, RoPE + cache append or both, where the matrix has the size
// for it (gemm_rows.cu); and of up to 256 rows where O and down leave parts of k for the norm.  Those with a residual add in the GEMMs occur above and up to 8 rows, the norms in
// the GEMMs (8) with as many of those as gemm_few_normalises allows.  fp32 models take 8 or, above kF32NormMax columns, 3 as long as their
// GEMMs have few output tiles, 0 otherwise.
constexpr int kVariants = 9;
const Fusion kFusion[kVariants] = {  // {swiglu, rope, residual, norm}
    {false, false, false}, {true, false, false}, {true, true, false}, {true, true, true},
    {false, true, false},  {false, false, true}, {true, false, true}, {false, true, true}, {true, true, true, true}};

int layer(int variant, const Entry** out) {
  const Fusion& f = kFusion[variant];
  int n = 0;
  if (!f.norm) out[n++] = f.residual ? &kNormAttnRead : &kNormAttn;
  out[n++] = f.norm ? &kQkvNorm : f.rope ? &kQkvRope : &kQkv;
  if (!f.rope) out[n++] = &kRope;
  out[n++] = &kAttn;
  out[n++] = f.residual ? &kWoAdd : &kWo;
  if (!f.norm) out[n++] = f.residual ? &kNormMlpRead : &kNormMlp;
  out[n++] = f.norm ? &kGuNorm : f.swiglu ? &kGuSwiglu : &kGu;
  if (!f.swiglu) out[n++] = &kSwiglu;
  out[n++] = f.residual ? &kDownAdd : &kDown;
  return n;
}

int build(int variant, const Entry** out) {
  // set-up, three layers (enough to close the cycle between layers), tail
  int n = 0;
  out[n++] = &kSetActive;
  if (kFusion[variant].norm) out[n++] = &kNormEmbed;
  for (int l = 0; l < 3; ++l) n += layer(variant, out + n);
  out[n++] = kFusion[variant].residual ? &kNormFinalRead : &kNormFinal;
  out[n++] = &kLm;
  out[n++] = &kArgmax;
  return n;
}

}  // namespace

int launch_order_variant(Fusion f) {
  for (int v = 0; v < kVariants; ++v)
    if (kFusion[v].swiglu == f.swiglu && kFusion[v].rope == f.rope && kFusion[v].residual == f.residual && kFusion[v].norm == f.norm) return v;
  return -1;
}

int launch_order_layer(int variant, int* ids_out) {
  const Entry* seq[kLayerLaunches];
  const int n = layer(variant, seq);
  for (int i = 0; i < n; ++i) ids_out[i] = seq[i]->id;
  return n;
}

// Number of (kernel, buffer) pairs that break the rule; the tail after the last layer counts as the "next layer"
// (its first kernel is a fused_norm as well).
int launch_order_violations(int variant) {
  const Entry* seq[64];
  const int n = build(variant, seq);
  int bad = 0;
  for (int i = 1; i < n; ++i) {
    for (unsigned bit = 1; bit <= B_STATE; bit <<= 1) {
      if (!(seq[i]->prewait_reads & bit)) continue;
      int j = i - 1;
      while (j >= 0 && !(seq[j]->writes & bit)) --j;
      if (j >= 0 && i - j < 2) ++bad;           // the youngest writer is the kernel right in front
    }
  }
  return bad;
}

}  // namespace cerb

extern "C" int cerb_launch_order_table(int32_t variant, char* buf, size_t cap) {
  using namespace cerb;
  if (!buf || cap < 64 || variant < 0 || variant >= kVariants) return CERB_E_ARG;
  const Entry* seq[64];
  const int n = build(variant, seq);
  size_t off = 0;
  for (int i = 0; i < n; ++i) {
    int w = snprintf(buf + off, cap - off, "%d|%s|%u|%u\n", seq[i]->id, seq[i]->name, seq[i]->writes, seq[i]->prewait_reads);
    if (w < 0 || (size_t)w >= cap - off) return CERB_E_NOMEM;
    off += (size_t)w;
  }
  return launch_order_violations(variant) == 0 ? CERB_OK : CERB_E_STATE;
}
