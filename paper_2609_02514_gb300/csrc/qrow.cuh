// Draft rows (float32) in 16-byte chunks, on or off the 16-byte grid.
#pragma once
#include "common.cuh"

namespace aces {

// A draft row in 16-byte chunks: element e of chunk c is id c * 4 + e - head
// (rows off the 16-byte grid start inside chunk 0); 0 outside the row.
struct QChunks {
    const float *base;
    int head, V, nch;
    __device__ __forceinline__ QChunks(const float *row, int V_) : V(V_) {
        head = (int)((uintptr_t)row & 15u) >> 2;
        base = row - head;
        nch = (V + head + 3) >> 2;
    }
    static __device__ __noinline__ uint4 edge(const float *row, int V, int x0) {
        uint32_t v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = x0 + e >= 0 && x0 + e < V ? __float_as_uint(__ldg(row + x0 + e)) : 0u;
        return make_uint4(v[0], v[1], v[2], v[3]);
    }
    __device__ __forceinline__ uint4 load(int c) const {
        if (c * 4 >= head && c * 4 + 4 <= V + head) return ldg16(base + (size_t)c * 4);
        return edge(base + head, V, c * 4 - head);
    }
};

}  // namespace aces
