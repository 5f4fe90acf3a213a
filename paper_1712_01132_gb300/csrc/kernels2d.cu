// kernels2d.cu -- sm_103a kernels of one source iteration (arXiv:1712.01132, Sec. 3.1) in 2D, apart from the
// transport sweeps (sweep2d_f32x2.cu, sweep2d_f64.cu).
//
// finalize2d: step (iii) completion: sums the per-quadrant moment partials, forms the wall
//             densities of Eq. 6 in FP64, the source terms and wall terms of the next sweep, and
//             the FP64 sum of u1 for the permeability of Eq. 11-12.
// init2d    : the zero-perturbation start in the kernels' source-form variables.
#include <cuda_runtime.h>

#include <cstdint>

#include "dvm_internal.h"
#include "dvm_device.cuh"

namespace dvm {

// ---------------------------------------------------------------- finalize

// rho'_s of face (y, axis j, side sigma) (Eq. 6) in FP64 from the quadrant partials of u_j at y:
// sum_{sigma v_j > 0} W |v_j| h / D = sigma * sum_{quadrants with sign(v_j) = sigma} P_uj / D.
template <typename T>
__device__ __forceinline__ double wall_density(const Prob2D<T>* P, int y, int j, int sigma, const double* dinv) {
    double num = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int neg = (q >> j) & 1;
        if (neg == (sigma < 0 ? 1 : 0)) num += (double)P->P[((size_t)q * 3 + 1 + j) * P->N + y];
    }
    return sigma * num * dinv[j];
}

// Points per finalize thread: a block of 256 threads covers 1024 consecutive points, thread t the
// points t, t + 256, t + 512 and t + 768 of its block (coalesced), with all of their loads issued
// before any store.
constexpr int kFinPPT = 4;

template <typename T>
__global__ void __launch_bounds__(256) finalize2d_kernel(const FinArgs2D<T> a) {
    using V = typename Vec4<T>::type;
    __shared__ double s_red[8];
    __shared__ int s_last;
    const int b = a.blk_prob[blockIdx.x];
    const Prob2D<T>* __restrict__ P = a.prob + b;
    const size_t N = P->N;
    double u1d = 0.0;
    int idk[kFinPPT];
    uint16_t code[kFinPPT];
    T pu[kFinPPT][4][3];     // quadrant partials (rho, u1, u2) of each point
#pragma unroll
    for (int k = 0; k < kFinPPT; ++k) {
        idk[k] = a.blk_start[blockIdx.x] + threadIdx.x + k * 256;
        code[k] = idk[k] < P->N ? P->code[idk[k]] : kSolidBit;
    }
#pragma unroll
    for (int k = 0; k < kFinPPT; ++k)
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int m = 0; m < 3; ++m)
                pu[k][q][m] = idk[k] < P->N ? P->P[((size_t)q * 3 + m) * N + idk[k]] : T(0);   // zero at solid points
#pragma unroll
    for (int k = 0; k < kFinPPT; ++k) {
        const int id = idk[k];
        if (id >= P->N) continue;
        V s = Vec4<T>::make(0, 0, 0, 0), e = s;
        if (!(code[k] & kSolidBit)) {
            T rho = T(0), u1 = T(0), u2 = T(0);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                rho += pu[k][q][0];
                u1 += pu[k][q][1];
                u2 += pu[k][q][2];
            }
            const T nu = (T)P->nu;
            s = Vec4<T>::make(nu * rho, T(2) * nu * u1 + T(1), T(2) * nu * u2, T(0));
            u1d += (double)u1;
            T ev[4];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int c = (code[k] >> (2 * (2 * j + u))) & 3;
                    const int sigma = u ? 1 : -1;
                    double val = 0.0;
                    if (c == 2) {
                        // first-order stencil: wall value of face (x, j, sigma) (Eq. 6, rho'_s in
                        // FP64 from the partials of u_j of the quadrants moving toward the wall:
                        // sigma * sum / D), shifted by the source-form offset sigma dx on x1 faces
                        // (Eq. 5: alpha times the diffuse value, through the alpha-scaled
                        // denominators; the specular part is added per velocity by the sweep)
                        double num = 0.0;
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            if (((q >> j) & 1) == (sigma < 0 ? 1 : 0)) num += (double)pu[k][q][1 + j];
                        val = sigma * num * P->dinvw[j] + (j == 0 ? sigma * P->dx : 0.0);
                    }
                    // case 1 (only the second upstream point solid) is first order on the fluid
                    // neighbour: no wall term
                    ev[2 * j + u] = (T)val;
                }
            }
            e = Vec4<T>::make(ev[0], ev[1], ev[2], ev[3]);
        }
        reinterpret_cast<V*>(P->src)[id] = s;
        reinterpret_cast<V*>(P->E)[id] = e;
    }
    // FP64 block sum of u1 (fixed tree), then the last block of the problem adds the block sums in
    // block order: the permeability is independent of scheduling.
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) u1d += __shfl_xor_sync(0xffffffffu, u1d, off);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = u1d;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += s_red[w];
        P->kpart[blockIdx.x - P->fin_block0] = tot;
        __threadfence();
        const unsigned prev = atomicAdd(P->fin_counter, 1u);
        s_last = (prev == (unsigned)P->fin_nblocks - 1u);
    }
    __syncthreads();
    if (s_last) {
        // all threads of the last block: strided partial sums in a fixed order, then a fixed tree
        __threadfence();
        double acc = 0.0;
        for (int k = threadIdx.x; k < P->fin_nblocks; k += blockDim.x) acc += __ldcg(P->kpart + k);
#pragma unroll
        for (int off = 16; off >= 1; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        __syncthreads();
        if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double tot = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += s_red[w];
            const double gp = tot / (double)P->N;
            P->kval[0] = 2.0 / sqrt(3.14159265358979323846) * P->kn * gp;
            P->kval[1] = gp;
            P->kval[2] = tot;
            *P->fin_counter = 0u;
        }
    }
}

// ---------------------------------------------------------------- init and readout

// Zero-perturbation start h = 0 in the paper's variables, i.e. h' = x1 in the kernels' variables:
// moment partials x1 * sum_{k in q} W_k (1, v1, v2) and ghost layers carrying x1 of their source
// points.  A finalize pass afterwards derives the source and wall terms.
template <typename T>
__global__ void init2d_kernel(const Prob2D<T>* prob, int NL, const double* qw /*[4][3]*/) {
    const Prob2D<T>* P = prob;
    const int n1 = P->n1, n2 = P->n2, N = P->N;
    const size_t nl = NL;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (size_t idx = t0; idx < (size_t)4 * 3 * N; idx += stride) {
        const int id = idx % N;
        const int qm = idx / N;
        const double x1 = (id % n1) * P->dx;
        P->P[idx] = (P->code[id] & kSolidBit) ? T(0) : (T)(x1 * qw[qm]);
    }
    const int nxs = P->nxslots;
    for (size_t idx = t0; idx < (size_t)2 * 4 * nxs * n2 * 2 * nl; idx += stride) {
        const int layer = (idx / nl) % 2;
        const int sl = (idx / (nl * 2 * n2)) % nxs;
        const int q = (idx / (nl * 2 * n2 * nxs)) % 4;
        const int ico = P->xslot_col[q * nxs + sl] - 1 - layer;     // oriented source column
        const int col = (q & 1) ? n1 - 1 - ico : ico;
        P->gx1[idx] = (T)(col * P->dx);
    }
    for (size_t idx = t0; idx < (size_t)2 * 4 * P->nslots * n1 * 2 * nl; idx += stride) {
        const int ic = (idx / (nl * 2)) % n1;
        const int q = (idx / (nl * 2 * n1 * P->nslots)) % 4;
        const int col = (q & 1) ? n1 - 1 - ic : ic;
        P->glat[idx] = (T)(col * P->dx);
    }
    if (P->spec > 0.0)   // face stores of both parities: h' = x1 at the face's fluid point
        for (size_t idx = t0; idx < (size_t)2 * P->nfaces * 2 * nl; idx += stride) {
            const int id = P->faces[(idx / (2 * nl)) % P->nfaces] >> 2;
            P->F[idx] = (T)((id % n1) * P->dx);
        }
}

// Warm start: the state an iteration leaves when it produced the local linearised equilibrium
// h0 = rho0 + 2 u0 . v at every fluid point (source form: h0' = h0 + x1).  Moment partials are the
// quadrant quadratures of h0' (closed form through qw2[q][m][n] = sum_{k in q} W phi_m psi_n with
// phi = psi = (1, v1, v2)); the lagged ghost layers read at parity `par` hold h0' at the points the
// sweep would have captured them from (same slot layout as the sweep kernels write).
template <typename T>
__global__ void warm2d_kernel(const Prob2D<T>* P, int NL, int par, const double* __restrict__ qw2,
                              const double* __restrict__ vel, const double* __restrict__ rho0,
                              const double* __restrict__ u0) {
    const int n1 = P->n1, n2 = P->n2, N = P->N;
    const size_t nl = NL;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    const size_t t0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    auto h0 = [&](int x, int y, const double* v) -> double {
        const int id = y * n1 + x;
        if (P->code[id] & kSolidBit) return 0.0;
        return rho0[id] + x * P->dx + 2.0 * (u0[id] * v[0] + u0[N + id] * v[1]);
    };
    for (size_t idx = t0; idx < (size_t)4 * 3 * N; idx += stride) {
        const int id = idx % N;
        const int qm = idx / N;
        double val = 0.0;
        if (!(P->code[id] & kSolidBit)) {
            const double* c = qw2 + (size_t)qm * 3;
            const double r = rho0[id] + (id % n1) * P->dx;
            val = r * c[0] + 2.0 * (u0[id] * c[1] + u0[N + id] * c[2]);
        }
        P->P[idx] = (T)val;
    }
    // lagged x1 layers: slot (q, s, oriented row, layer) holds h at the oriented column
    // xslot_col[q][s] - 1 - layer (slot 0: the x1 ghosts, columns n1 - 1 - layer)
    const int nxs = P->nxslots;
    for (size_t idx = t0; idx < (size_t)4 * nxs * n2 * 2 * nl; idx += stride) {
        const int l = idx % nl;
        const int layer = (idx / nl) % 2;
        const int yo = (idx / (nl * 2)) % n2;
        const int sl = (idx / (nl * 2 * n2)) % nxs;
        const int q = idx / (nl * 2 * n2 * nxs);
        const int ico = P->xslot_col[q * nxs + sl] - 1 - layer;
        const int x = (q & 1) ? n1 - 1 - ico : ico;
        const int y = (q & 2) ? n2 - 1 - yo : yo;
        P->gx1[(size_t)par * 4 * nxs * n2 * 2 * nl + idx] = (T)h0(x, y, vel + ((size_t)q * nl + l) * 2);
    }
    // lagged x2 layers: quadrant q writes the oriented rows below slot s (slot 0: its top rows
    // n2 - 1 - layer) into the slot of the quadrant that reads them (slot 0: itself when periodic,
    // the x2-reflected quadrant when specular; subdomain slots: itself)
    const int ns = P->nslots;
    for (size_t idx = t0; idx < (size_t)4 * ns * n1 * 2 * nl; idx += stride) {
        const int l = idx % nl;
        const int layer = (idx / nl) % 2;
        const int ic = (idx / (nl * 2)) % n1;
        const int sl = (idx / (nl * 2 * n1)) % ns;
        const int q = idx / (nl * 2 * n1 * ns);
        const int x = (q & 1) ? n1 - 1 - ic : ic;
        const int yo = P->slot_row[q * ns + sl] - 1 - layer;
        const int y = (q & 2) ? n2 - 1 - yo : yo;
        const int qd = (sl > 0 || P->lateral == 1) ? q : (q ^ 2);
        P->glat[(((((size_t)par * 4 + qd) * ns + sl) * n1 + ic) * 2 + layer) * nl + l] =
            (T)h0(x, y, vel + ((size_t)q * nl + l) * 2);
    }
    // face stores (specular wall part, Eq. 5): h0' at the face's fluid point for the velocity slot
    // of the quadrant that moves into the face (s_j = the face side, other-axis sign bit o)
    if (P->spec > 0.0)
        for (size_t idx = t0; idx < (size_t)P->nfaces * 2 * nl; idx += stride) {
            const int l = idx % nl;
            const int o = (idx / nl) % 2;
            const int f = P->faces[idx / (2 * nl)];
            const int id = f >> 2, j = (f >> 1) & 1, u = f & 1;
            const int qw = (j == 0) ? ((1 - u) | (o << 1)) : (o | ((1 - u) << 1));
            P->F[(size_t)par * P->nfaces * 2 * nl + idx] = (T)h0(id % n1, id / n1, vel + ((size_t)qw * nl + l) * 2);
        }
}

// rho (paper variables, ramp restored) and u of one problem into double buffers; solid = 0.
template <typename T>
__global__ void moments2d_kernel(const Prob2D<T>* prob, double* rho, double* u) {
    const Prob2D<T>* P = prob;
    const int N = P->N;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        if (P->code[id] & kSolidBit) {
            rho[id] = 0.0;
            u[id] = 0.0;
            u[N + id] = 0.0;
            continue;
        }
        T r = T(0), u1 = T(0), u2 = T(0);
        for (int q = 0; q < 4; ++q) {
            r += P->P[((size_t)q * 3 + 0) * N + id];
            u1 += P->P[((size_t)q * 3 + 1) * N + id];
            u2 += P->P[((size_t)q * 3 + 2) * N + id];
        }
        rho[id] = (double)r - (id % P->n1) * P->dx;
        u[id] = (double)u1;
        u[N + id] = (double)u2;
    }
}

// Wall densities [2][2][N] (axis, side) in the paper's variables; 0 where there is no face.
template <typename T>
__global__ void wall2d_kernel(const Prob2D<T>* prob, double* out) {
    const Prob2D<T>* P = prob;
    const int N = P->N;
    for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < N; id += gridDim.x * blockDim.x) {
        const uint16_t code = P->code[id];
        for (int j = 0; j < 2; ++j)
            for (int u = 0; u < 2; ++u) {
                double v = 0.0;
                if (!(code & kSolidBit) && ((code >> (2 * (2 * j + u))) & 3) == 2)
                    v = wall_density(P, id, j, u ? 1 : -1, P->dinv) - (id % P->n1) * P->dx;
                out[(size_t)(2 * j + u) * N + id] = v;
            }
    }
}

// ---------------------------------------------------------------- launchers

template <typename T>
cudaError_t launch_finalize2d(const FinArgs2D<T>& a, int nblocks, cudaStream_t st) {
    finalize2d_kernel<T><<<nblocks, 256, 0, st>>>(a);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_init2d(const Prob2D<T>* prob_dev, int NL, const double* qw_dev, cudaStream_t st) {
    init2d_kernel<T><<<304, 256, 0, st>>>(prob_dev, NL, qw_dev);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_warm2d(const Prob2D<T>* prob_dev, int NL, int par, const double* qw2, const double* vel,
                          const double* rho0, const double* u0, cudaStream_t st) {
    warm2d_kernel<T><<<304, 256, 0, st>>>(prob_dev, NL, par, qw2, vel, rho0, u0);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_moments2d(const Prob2D<T>* prob_dev, double* rho, double* u, cudaStream_t st) {
    moments2d_kernel<T><<<304, 256, 0, st>>>(prob_dev, rho, u);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_wall2d(const Prob2D<T>* prob_dev, double* out, cudaStream_t st) {
    wall2d_kernel<T><<<304, 256, 0, st>>>(prob_dev, out);
    return cudaGetLastError();
}

#define DVM_INSTANTIATE(T)                                                                      \
    template cudaError_t launch_finalize2d<T>(const FinArgs2D<T>&, int, cudaStream_t);          \
    template cudaError_t launch_init2d<T>(const Prob2D<T>*, int, const double*, cudaStream_t);  \
    template cudaError_t launch_warm2d<T>(const Prob2D<T>*, int, int, const double*, const double*, \
                                          const double*, const double*, cudaStream_t);            \
    template cudaError_t launch_moments2d<T>(const Prob2D<T>*, double*, double*, cudaStream_t); \
    template cudaError_t launch_wall2d<T>(const Prob2D<T>*, double*, cudaStream_t);

DVM_INSTANTIATE(float)
DVM_INSTANTIATE(double)

}  // namespace dvm
