// Molecular dynamics with the potential: velocity Verlet, neighbour lists with a skin.
//
// The neighbour list is built once for the search radius R_cut + skin and kept, together with the
// build-time displacements r0_ij and positions x0, while no atom has moved more than skin / 2 (then
// no pair can cross R_cut unseen).  Between rebuilds every step refreshes
//   r_ij = r0_ij + (u_j - u_i),   u = x - x0,
// where u is small, so the float path keeps full float accuracy in r_ij.  Units: Angstrom, fs, eV,
// amu; 1 amu Angstrom^2 / fs^2 = 103.6427 eV.
#include <cuda_runtime.h>
#include "mtp_internal.h"
#include "mtp_common.cuh"

namespace mtp {

namespace {

constexpr double kMvv2eV = 103.642696;  // amu Angstrom^2 fs^-2 in eV

// u_i = x_i - x0_i in the working precision, one vector per atom
template <class T>
__device__ __forceinline__ void put_displacement(int i, const double* x, const double* x0, Vec4<T>* u, int* err) {
    const double u0 = x[3 * (size_t)i] - x0[3 * (size_t)i];
    const double u1 = x[3 * (size_t)i + 1] - x0[3 * (size_t)i + 1];
    const double u2 = x[3 * (size_t)i + 2] - x0[3 * (size_t)i + 2];
    if (!(isfinite(u0) && isfinite(u1) && isfinite(u2))) atomicOr(err, kErrNonFinite);
    u[i] = Vec4<T>{(T)u0, (T)u1, (T)u2, T(0)};
}

template <class T>
__global__ void k_displacements(int n, const double* x, const double* x0, Vec4<T>* u, int* err) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        put_displacement<T>(i, x, x0, u, err);
}

// r_ij = r0_ij + (u_j - u_i), one thread per atom and kPairSlots list slots (blockIdx.y): the loads of a
// few independent pairs per thread and a block per slot group keep enough of them in flight; one thread
// walking an atom's whole list took 40 us at 16,384 atoms (42 pairs each), this takes 5.9.
constexpr int kPairSlots = 4;
template <class T>
__global__ void __launch_bounds__(128) k_update_pairs(int n, const int* count, const PairRec<T>* r0,
                                                      const Vec4<T>* u, PairRec<T>* pr, int* queue) {
    const size_t N = (size_t)n;
    // the evaluation kernels' work queues start at zero (the neighbour build clears them otherwise)
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 2) queue[threadIdx.x] = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int cnt = count[i], p0 = blockIdx.y * kPairSlots;
        if (p0 >= cnt) continue;
        const Vec4<T> ui = u[i];
#pragma unroll
        for (int q = 0; q < kPairSlots; ++q) {
            if (p0 + q < cnt) {
                const size_t o = (size_t)(p0 + q) * N + i;
                PairRec<T> rec = r0[o];
                const Vec4<T> uj = u[rec.jz & 0xffffff];
                rec.x = rec.x + (uj.x - ui.x);
                rec.y = rec.y + (uj.y - ui.y);
                rec.z = rec.z + (uj.z - ui.z);
                pr[o] = rec;
            }
        }
    }
}

__device__ __forceinline__ int species(const int* types, int i, int S) {
    const int z = types[i];  // out-of-range species are reported by the neighbour build
    return z < 0 ? 0 : (z >= S ? S - 1 : z);
}

// Second half kick of a step and the kinetic energy of the new velocities (kick = false: the kinetic
// energy alone); clears the rebuild flag (flag[0]) for the drift that follows and keeps the error word of the
// evaluation for it (flag[1]).
__global__ void k_kick_kinetic(int n, int S, double* v, const double* F, const int* types, const double* masses,
                               double half_dt, bool kick, double* out, int* flag, const int* err) {
    __shared__ double s[256];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        flag[0] = 0;
        flag[1] = *err;
    }
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double m = masses[species(types, i, S)];
        double w[3];
        for (int c = 0; c < 3; ++c) w[c] = v[3 * (size_t)i + c];
        if (kick) {
            const double q = half_dt / (m * kMvv2eV);
            for (int c = 0; c < 3; ++c) {
                w[c] += q * F[3 * (size_t)i + c];
                v[3 * (size_t)i + c] = w[c];
            }
        }
        acc += 0.5 * m * kMvv2eV * (w[0] * w[0] + w[1] * w[1] + w[2] * w[2]);
    }
    s[threadIdx.x] = acc;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(out, s[0]);
}

// First half kick, x += dt v, and the displacements since the build for the refresh of the pairs; flags
// a rebuild when |x - x0| exceeds skin / 2.  Launched before the host has seen whether the evaluation that
// gave F succeeded: if it did not (flag[1], which this kernel does not write: all blocks agree), positions and
// velocities stay those of the failing step.
template <class T>
__global__ void k_kick_drift(int n, int S, double* x, double* v, const double* F, const int* types,
                             const double* masses, double half_dt, const double* x0, double dt, double lim2,
                             Vec4<T>* u, int* flag, int* err) {
    if (flag[1] != 0) return;
    bool far = false;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double q = half_dt / (masses[species(types, i, S)] * kMvv2eV);
        double d2 = 0.0;
        for (int c = 0; c < 3; ++c) {
            const size_t o = 3 * (size_t)i + c;
            const double w = v[o] + q * F[o];
            v[o] = w;
            const double xn = x[o] + dt * w;
            x[o] = xn;
            const double d = xn - x0[o];
            d2 += d * d;
        }
        put_displacement<T>(i, x, x0, u, err);
        far = far || !(d2 <= lim2);  // a NaN displacement forces a rebuild, whose checks report it
    }
    if (__syncthreads_or(far) && threadIdx.x == 0) atomicOr(flag, 1);
}

int grid_for(int n, int threads, int n_sm) {
    int b = (n + threads - 1) / threads;
    if (b > n_sm * 8) b = n_sm * 8;
    return b < 1 ? 1 : b;
}

}  // namespace

int launch_update_pairs(const NbrState& nb, const double* x, bool have_u, cudaStream_t st, int n_sm) {
    const int n = nb.n_atoms;
    const dim3 grid((unsigned)((n + 127) / 128), (unsigned)((nb.cap + kPairSlots - 1) / kPairSlots));
    int* queue = nb.counters.as<int>() + 4;
    auto go = [&](auto zero) {
        using T = decltype(zero);
        if (!have_u)
            k_displacements<T><<<grid_for(n, 256, n_sm), 256, 0, st>>>(n, x, nb.x0.as<double>(), nb.disp.as<Vec4<T>>(),
                                                                       nb.err.as<int>());
        k_update_pairs<T><<<grid, 128, 0, st>>>(n, nb.count.as<int>(), nb.pr.as<PairRec<T>>(), nb.disp.as<Vec4<T>>(),
                                                nb.cpr.as<PairRec<T>>(), queue);
    };
    if (nb.fp64)
        go(double(0));
    else
        go(float(0));
    return have_u ? 1 : 2;
}

int launch_kick_kinetic(const NbrState& nb, int S, double* v, const double* F, const int* types, const double* masses,
                        double half_dt, bool kick, double* e_kin, int* flag, cudaStream_t st, int n_sm) {
    const int n = nb.n_atoms;
    k_kick_kinetic<<<grid_for(n, 256, n_sm), 256, 0, st>>>(n, S, v, F, types, masses, half_dt, kick, e_kin, flag,
                                                          nb.err.as<int>());
    return 1;
}

int launch_kick_drift(const NbrState& nb, int S, double* x, double* v, const double* F, const int* types,
                      const double* masses, double dt, double lim2, int* flag, cudaStream_t st, int n_sm) {
    const int n = nb.n_atoms, grid = grid_for(n, 256, n_sm);
    if (nb.fp64)
        k_kick_drift<double><<<grid, 256, 0, st>>>(n, S, x, v, F, types, masses, 0.5 * dt, nb.x0.as<double>(), dt, lim2,
                                                   nb.disp.as<Vec4<double>>(), flag, nb.err.as<int>());
    else
        k_kick_drift<float><<<grid, 256, 0, st>>>(n, S, x, v, F, types, masses, 0.5 * dt, nb.x0.as<double>(), dt, lim2,
                                                  nb.disp.as<Vec4<float>>(), flag, nb.err.as<int>());
    return 1;
}

}  // namespace mtp
