// Host-side dispatch of kmq_linear: picks a kernel variant for (bits, M, N, K, layout).
#include "kmq_common.cuh"
#include "kmq_linear_variants.cuh"
#include "kmq_rows.cuh"

namespace kmq {

LinearPlan plan_linear(int64_t N, int64_t K, int bits, int64_t M, int layout, size_t scratch_limit) {
  LinearPlan p;
  p.workspace = 0;
  p.split_k = 1;
  if (layout == KMQ_LAYOUT_TABLE && bits != 4) {
    if (!linear_lut_supports(N, K, bits, M)) {
      p.variant = kVariantUnsupported;
      p.launches = 0;
      p.name = "unsupported";
      return p;
    }
    p.variant = kVariantLut;
    p.workspace = linear_lut_scratch_bytes(N, K, bits);
    p.launches = (int)(p.workspace ? 2 * M : M);
    p.name = bits == 1 ? "table_lookup_b1" : "table_lookup_b2";
    return p;
  }
  if (layout == KMQ_LAYOUT_TABLE) layout = KMQ_LAYOUT_TUNED;   // b = 4: the two layouts are the same
  if (layout == KMQ_LAYOUT_CANONICAL) {
    const bool mma = linear_mma_selected(N, K, bits, M);
    p.variant = mma ? kVariantMma : kVariantRows;
    p.launches = (int)((M + linear_rows_per_launch() - 1) / linear_rows_per_launch());
    if (mma) p.name = bits == 2 ? "staged_prmt_b2" : "staged_select_b1";
    else p.name = bits == 4 ? "staged_pairtable_b4" : bits == 2 ? "staged_pairtable_b2" : "staged_pairtable_b1";
    return p;
  }
  // (the balanced pairs of kernels, whose callers bring scratch for them, keep their shapes)
  const bool few = linear_umma_few_rows(N, K, bits, M) && !linear_split_ctas(N, K, bits, M) &&
                   !(M >= linear_multi_min_rows(bits, N, K) && linear_multi_split(N, K, bits, M).ctas);
  if (few || linear_umma_selected(N, K, bits, M)) {
    const int64_t per = linear_umma_rows_per_launch();
    p.variant = kVariantUmma;
    p.launches = (int)((M + per - 1) / per);
    p.name = bits == 4 ? "tcgen05_prmt_b4" : bits == 2 ? "tcgen05_prmt_b2" : "tcgen05_select_b1";
    return p;
  }
  if (M >= linear_multi_min_rows(bits, N, K)) {
    const int64_t per = linear_multi_rows_per_launch();
    p.variant = kVariantMulti;
    p.launches = (int)((M + per - 1) / per);
    p.name = bits == 4 ? "multi_prmt_b4" : bits == 2 ? "multi_prmt_b2" : "multi_select_b1";
    const MultiSplit sp = linear_multi_split(N, K, bits, M);
    if (sp.ctas && scratch_limit >= sp.scratch) {
      p.launches = 2;
      p.split_k = sp.ctas;
      p.workspace = sp.scratch;
      p.name = bits == 4 ? "multi_balanced_b4" : bits == 2 ? "multi_balanced_b2" : "multi_balanced_b1";
    }
    return p;
  }
  if (const int ctas = linear_split_ctas(N, K, bits, M)) {
    p.variant = kVariantSplit;
    p.launches = 2;
    p.split_k = ctas;
    p.workspace = linear_split_scratch_bytes(ctas);
    p.name = bits == 4 ? "split_pairtable_b4" : bits == 2 ? "split_prmt_b2" : "split_select_b1";
    return p;
  }
  p.variant = kVariantTiled;
  p.launches = (int)((M + 7) / 8);
  p.name = bits == 4 ? "tiled_pairtable_b4" : bits == 2 ? "tiled_prmt_b2" : "tiled_select_b1";
  return p;
}

cudaError_t launch_linear(const LinearPlan& plan, const uint32_t* packed, const uint16_t* cb, const uint16_t* x,
                          uint16_t* y, int64_t N, int64_t K, int bits, int64_t M, int layout, void* workspace,
                          cudaStream_t s) {
  if (layout == KMQ_LAYOUT_TABLE && bits == 4) layout = KMQ_LAYOUT_TUNED;
  switch (plan.variant) {
    case kVariantLut:
      return launch_linear_lut(packed, cb, x, y, N, K, bits, M, workspace, s);
    case kVariantUnsupported:
      return cudaErrorNotSupported;
    case kVariantSplit:
      return launch_linear_split(packed, cb, x, y, N, K, bits, M, workspace, plan.split_k, s);
    case kVariantUmma:
      return launch_linear_umma(packed, cb, x, y, N, K, bits, M, s);
    case kVariantMulti:
      return launch_linear_multi(packed, cb, x, y, N, K, bits, M, plan.workspace ? workspace : nullptr, s);
    case kVariantMma:
      return launch_linear_mma(packed, cb, x, y, N, K, bits, M, s);
    case kVariantRows:
      return launch_linear_rows(packed, cb, x, y, N, K, bits, M, s);
    case kVariantTiled:
    default:
      return launch_linear_tiled(packed, cb, x, y, N, K, bits, M, s);
  }
}

}  // namespace kmq
