// mesh_rule.h -- which texel of the neighbouring ring closes a triangle of VaFR_Rep's
// mesh (device code of the reprojection; plain C++ for the tests).
#pragma once

#ifdef __CUDACC__
#define VAFR_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define VAFR_HOST_DEVICE inline
#endif

namespace vafr {

// Row of the ring of n2 texels that closes the triangle over the step from row j to
// row j + 1 of a ring of n texels (0 <= j < n), modulo n2:
//   s = 0 (towards the next column)      max{k : (2k+1) n <  (2j+3) n2}
//   s = 1 (towards the column before)    max{k : (2k+1) n <= (2j+3) n2}
// Rings below 32,768 texels keep the products within 32 bits.  k, at most 3/2 n2,
// needs one correction and no remainder (the raster pass takes 38 us, with 64-bit
// divisions and remainders 42).
VAFR_HOST_DEVICE int ring_partner(int n, int n2, int j, int s) {
    long long k;
    if ((n | n2) < 32768) {
        const unsigned d = (unsigned)n, num = (2u * (unsigned)j + 3u) * (unsigned)n2;
        k = s == 0 ? ((int)((num + d - 1u) / d) - 2) >> 1 : ((int)(num / d) - 1) >> 1;
    } else {
        const long long d = n, num = (2ll * j + 3) * n2;
        k = s == 0 ? ((num + d - 1) / d - 2) >> 1 : (num / d - 1) >> 1;
    }
    if (k < 0) k += n2;
    else if (k >= n2) k -= n2;
    return (int)k;
}

}  // namespace vafr
