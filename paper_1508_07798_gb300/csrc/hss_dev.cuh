// Device helpers shared by the kernels of the HSS construction.
#pragma once
#include "hss.h"

namespace hssnd {

// 16 bytes of a shared-memory column (4 floats or 2 doubles), 16-byte aligned.
template <class T> __device__ __forceinline__ void ld16(const T *p, T *a) {
    if constexpr (std::is_same<T, float>::value) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        a[0] = v.x;
        a[1] = v.y;
        a[2] = v.z;
        a[3] = v.w;
    } else {
        const double2 v = *reinterpret_cast<const double2 *>(p);
        a[0] = v.x;
        a[1] = v.y;
    }
}
template <class T> __device__ __forceinline__ void st16(T *p, const T *a) {
    if constexpr (std::is_same<T, float>::value)
        *reinterpret_cast<float4 *>(p) = make_float4(a[0], a[1], a[2], a[3]);
    else
        *reinterpret_cast<double2 *>(p) = make_double2(a[0], a[1]);
}

}  // namespace hssnd
