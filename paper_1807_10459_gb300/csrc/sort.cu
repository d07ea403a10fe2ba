// sort.cu -- the library's one use of a vendor primitive: CUB's device radix
// sort, of (32-bit key, int32 index) pairs to order the samples before the
// estimator runs, and of a single short column's values for counts in it.  Kept
// in its own translation unit so the template instantiations compile in parallel.
#include <cub/device/device_radix_sort.cuh>

#include "ksg_common.cuh"

namespace idtx {

cudaError_t sort_pairs_u32(void *tmp, size_t &tmp_bytes, const uint32_t *keys_in,
                           uint32_t *keys_out, const int32_t *vals_in, int32_t *vals_out, int n,
                           int end_bit, cudaStream_t stream)
{
    return cub::DeviceRadixSort::SortPairs(tmp, tmp_bytes, keys_in, keys_out, vals_in, vals_out, n,
                                           0, end_bit, stream);
}

cudaError_t sort_floats(void *tmp, size_t &tmp_bytes, const float *in, float *out, int n,
                        cudaStream_t stream)
{
    return cub::DeviceRadixSort::SortKeys(tmp, tmp_bytes, in, out, n, 0, 32, stream);
}

}  // namespace idtx
