// fine_tiles.cuh -- the polynomial fine step for fields that no cluster holds
// (fine_tiles.cu), as the entry points of fine_big.cu and fine3d.cu call it.
#pragma once

#include "fine.cuh"

namespace acpr {

// Field f = g * per_group + i of a batch is field map[g] * gs + off + i of the
// array at `base` (map NULL: identity).
struct FieldMap {
    float* base;
    int per_group;
    long long gs, off;
    const int* map;
    __host__ __device__ float* at(int f, long long cells) const {
        const int g = f / per_group, i = f % per_group;
        const long long pg = map ? map[g] : g;
        return base + (pg * gs + off + i) * cells;
    }
};

constexpr int kSumWords = 56;

// `steps` >= 1 steps of `fields` 1024 x 1024 fields by a degree-2 polynomial.
// tmp: as many contiguous fields; sum_words: kSumWords words per field (mass model).
int big_tiles_run(const SolvePoly& poly, double a, double dt, int mass, int fields, int steps, FieldMap src, FieldMap dst,
                  float* tmp, long long* sum_words, cudaStream_t st);

// The same on the cube (n = 32, 64 or 128); u_in may equal u_out.
int cube_run(const ac_params* p, const SolvePoly& poly, int steps, int fields, const float* u_in, float* u_out, float* tmp,
             long long* sum_words, cudaStream_t st);

}  // namespace acpr
