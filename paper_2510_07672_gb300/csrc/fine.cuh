// fine.cuh -- launch arguments shared by the fine-step kernels of fine.cu
// (Fourier solve) and fine_stencil.cu (polynomial solve), and the polynomial.
#pragma once

#include "common.cuh"

namespace acpr {

struct FineArgs {
    const void* in;
    void* out;
    int num_fields;
    int steps;
    // Field f = g * per_group + i reads field (map[g] * in_gs + in_off + i) of
    // `in` and writes field (map[g] * out_gs + out_off + i) of `out` (map NULL:
    // identity).  Plain batched calls use per_group = num_fields.
    int per_group;
    long long in_gs, in_off, out_gs, out_off;
    const int* map;
    // Work list (overrides the mapping above and `steps`): field f reads field
    // work[f].x of `in`, writes field work[f].y of `out`, runs work[f].z steps.
    const int4* work;
    int mass;        // 1: hold the (0,0) mode at the entry mean
    // adjoint = 1 runs the transposed steps: lambda_n = a mu + dt f'(u_n) * (mu -
    // [mass] mean mu), mu = A^{-1} lambda_{n+1}, with u_n read from
    // states[n][field] (n = steps-1 .. 0, plain field index).
    int adjoint;
    const void* states;
    // traj != NULL stores the state before the first step and after every
    // step: traj[s][field] for s = 0..steps (plain field index).
    void* traj;
    double a;        // 1 + S dt
    double dt;
    double lam_scale;  // dt eps^2 (4 / h^2)
};

// Degrees of the solve polynomials that are built.
constexpr int kMaxDegree = 6;

// p(T) = sum_j b_j T^j, T the sum of a cell's 2 d neighbours, with
// p(Laplacian) = (a - dt eps^2 Lap_h)^{-1} to the precision of the fields.
struct SolvePoly {
    int degree = 0;              // 0: no polynomial of a built degree is exact enough
    double b[kMaxDegree + 1] = {};
};

// The polynomial of the least degree in [min_degree, max_degree] for a step of
// the given 1 + S dt and dt eps^2 4 / h^2 in `dims` dimensions (degree 0: none).
SolvePoly solve_poly(double a, double lam_scale, int dims, int precision, int min_degree, int max_degree);

// Fine propagation by the polynomial solve (fine_stencil.cu); *taken = false
// (and nothing is launched) when the size, the precision or the step is not
// one it is built for.
template <typename T>
int launch_stencil(int n, const FineArgs& args, cudaStream_t stream, bool* taken);

// The adjoint steps of `adj` and the forward steps of `fwd` (same step, other
// fields) side by side in one launch, where the polynomial solve serves them.
int launch_stencil_pair(int n, int precision, const FineArgs& adj, const FineArgs& fwd, cudaStream_t stream, bool* taken);

}  // namespace acpr
