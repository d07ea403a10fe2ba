// ksg_inst_k7_d1.cu -- compiled specialisations of the fused KSG kernel for
// any k <= 7 (runtime), dx = 1, dy = 1 and 2, 32 jobs per CTA, z buckets 1, 2,
// 3, 6, 10, 16 (a wider row costs the list building and the full scans, not the
// walks, so there are fewer than for k = 4).  Against the generic one (four x
// columns, 16 warps an SM): N = 2503, two x, one y and three z columns, k = 7,
// 21 estimates, list kernel 172 -> 98 us, the call 0.55 -> 0.41 ms.
#include "ksg_list.cuh"

namespace idtx {

int ksg_variants_k7_d1(KsgVariant *out)
{
    int n = 0;
    out[n++] = make_variant<1, 1, 1, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 1, 2, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 1, 3, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 1, 6, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 1, 10, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 1, 16, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 2, 1, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 2, 2, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 2, 3, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 2, 6, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 2, 10, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    out[n++] = make_variant<1, 2, 16, 8, false, IDTX_FAST_QC, IDTX_FAST_NW>();
    return n;
}

}  // namespace idtx
