// Instances of the one-block kernel with asynchronous exchange.
#pragma once

#include "rank2_async.cuh"

namespace romk {

template <typename T, int KI, bool MANY>
void* async_instance_for(int cb) {
    return cb == 1   ? (void*)&rank2_async_kernel<T, KI, 1, MANY>
           : cb == 2 ? (void*)&rank2_async_kernel<T, KI, 2, MANY>
                     : (void*)&rank2_async_kernel<T, KI, 4, MANY && sizeof(T) == 8>;  // (FP32: one form)
}
template <typename T, bool MANY>
void* async_instance(int KI, int cb) {
    switch (KI) {
        case 1: return async_instance_for<T, 1, MANY>(cb);
        case 2: return async_instance_for<T, 2, MANY>(cb);
        case 3: return async_instance_for<T, 3, MANY>(cb);
        case 4: return async_instance_for<T, 4, MANY>(cb);
        default: break;
    }
    if constexpr (sizeof(T) == 4) {
        switch (KI) {
            case 5: return async_instance_for<T, 5, MANY>(cb);
            case 6: return async_instance_for<T, 6, MANY>(cb);
            case 7: return async_instance_for<T, 7, MANY>(cb);
            case 8: return async_instance_for<T, 8, MANY>(cb);
            default: break;
        }
    }
    return nullptr;
}

// The instance for many receivers (FP32: at most 2 columns a group).
void* async_many_kernel(bool f64, int KI, int cb);

}  // namespace romk
