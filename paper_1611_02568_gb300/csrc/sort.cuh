// Bitonic sort of 32 V 64-bit keys in a warp's registers, ascending: key v of
// lane l is element l V + v, so that the strides below V stay inside a lane and
// only the others cost shuffles.
#pragma once

#include "common.cuh"

namespace pxsne {

template <int V>
__device__ __forceinline__ void sort_keys(u64 (&key)[V], int lane) {
#pragma unroll
    for (int k2 = 2; k2 <= 32 * V; k2 <<= 1) {
#pragma unroll
        for (int j = k2 >> 1; j > 0; j >>= 1) {
            if (j >= V) {
                const int lj = j / V;
                const bool upper = lane & lj;
#pragma unroll
                for (int v = 0; v < V; v++) {
                    const bool up = ((lane * V + v) & k2) == 0;
                    const u64 o = __shfl_xor_sync(0xffffffffu, key[v], lj);
                    const bool less = o < key[v];
                    // the lower element of an ascending pair keeps the smaller key
                    key[v] = (less == (up != upper)) ? o : key[v];
                }
            } else {
#pragma unroll
                for (int v = 0; v < V; v++) {
                    const int w = v ^ j;
                    if (w > v) {
                        const bool up = ((lane * V + v) & k2) == 0;
                        const u64 x = key[v], y = key[w];
                        const bool sw = (x > y) == up;
                        key[v] = sw ? y : x;
                        key[w] = sw ? x : y;
                    }
                }
            }
        }
    }
}

}  // namespace pxsne
