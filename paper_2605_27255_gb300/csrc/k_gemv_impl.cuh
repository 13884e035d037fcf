// Launch handles of the CUDA-core GEMV kernels of one weight type T (included
// by k_gemv_bf16.cu and k_gemv_f32.cu).
#pragma once

#include "gemv_block.cuh"
#include "gemv_stream.cuh"
#include "kernel_tables.h"
#include "kernels.cuh"

namespace pipo {

constexpr int kStreamDepth = 4;  // chunks per register batch (two batches in flight)

template <typename T>
void* pick_block_t(int ru) {
    return ru == 2 ? reinterpret_cast<void*>(&gemv_kernel<T, 2>) : reinterpret_cast<void*>(&gemv_kernel<T, 1>);
}

template <typename T, int NB, int RU>
void* stream_fn(bool rows) {
    return rows ? reinterpret_cast<void*>(&gemv_rows_kernel<T, NB, RU, kStreamDepth>)
                : reinterpret_cast<void*>(&gemv_stream_kernel<T, NB, RU, kStreamDepth>);
}

// rows: every weight row is a whole number of 512-byte chunks (fast kernel)
template <typename T>
void* pick_stream_t(int nb, int ru, bool rows) {
    switch (nb) {
        case 1: return ru == 2 ? stream_fn<T, 1, 2>(rows) : stream_fn<T, 1, 1>(rows);
        case 2: return ru == 2 ? stream_fn<T, 2, 2>(rows) : stream_fn<T, 2, 1>(rows);
        default: return ru == 2 ? stream_fn<T, 4, 2>(rows) : stream_fn<T, 4, 1>(rows);
    }
}

}  // namespace pipo
