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
    T v[2];   // the two quadrants whose sign bit of axis j is (sigma < 0), ascending
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int q = j == 0 ? (2 * i + (sigma < 0)) : (i + 2 * (sigma < 0));
        v[i] = P->P[((size_t)q * 3 + 1 + j) * P->N + y];
    }
    const double num = widen(v[0]) + widen(v[1]);
    return num * (sigma < 0 ? -dinv[j] : dinv[j]);
}

// Bound by FP64 issue when every lane of a warp with a wall point computed wall densities and a shuffle tree added
// the u1 of 32 points (a warp instruction per ~16 cycles and SM): a warp now lists its wall faces and computes
// them a lane per face, and a thread adds the u1 of its points before the tree.  Solid points are neither read
// nor written (nothing reads their sources).  1,048,576 points of the 512^2 medium at four Knudsen numbers:
// 64 -> 29 us; a 32^2 cell in FP64: 16 -> 8 us.
// A block of 256 threads covers ppt x 256 consecutive points, thread t the points t, t + 256, ... of its block.
template <typename T>
__global__ void __launch_bounds__(256) finalize2d_kernel(const FinArgs2D<T> a, const int ppt) {
    using V = typename Vec4<T>::type;
    __shared__ double s_red[8];
    __shared__ T s_ev[8][32 * 4];
    __shared__ unsigned char s_face[8][32 * 4];
    const Prob2D<T>* __restrict__ P = a.prob + a.blk_prob[blockIdx.x];
    const size_t N = P->N;
    const T nu = (T)P->nu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int start = a.blk_start[blockIdx.x];
    auto code_of = [&](int k) -> int {
        const int id = start + k * 256 + threadIdx.x;
        return k < ppt && id < P->N ? P->code[id] : kSolidBit;
    };
    double sum1 = 0.0;
    int next = code_of(0);
    for (int k = 0; k < ppt; ++k) {
        const int id = start + k * 256 + threadIdx.x;
        const int code = next;
        next = code_of(k + 1);
        const bool fluid = !(code & kSolidBit);
        T rho = T(0), u1 = T(0), u2 = T(0);
        if (fluid) {
            T pu[4][3];          // quadrant partials (rho, u1, u2)
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int m = 0; m < 3; ++m) pu[q][m] = P->P[((size_t)q * 3 + m) * N + id];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                rho += pu[q][0];
                u1 += pu[q][1];
                u2 += pu[q][2];
            }
        }
        if (fluid) sum1 += widen(u1);
        // the warp's faces (upstream point of (axis j, side u) solid: case 2), a lane each
        int nface = 0, mine[4];
#pragma unroll
        for (int ju = 0; ju < 4; ++ju) {
            const bool f = fluid && ((code >> (2 * ju)) & 3) == 2;
            const unsigned m = __ballot_sync(0xffffffffu, f);
            mine[ju] = f ? nface + __popc(m & ((1u << lane) - 1u)) : -1;
            if (f) s_face[warp][mine[ju]] = (unsigned char)(lane * 4 + ju);
            nface += __popc(m);
        }
        __syncwarp();
        for (int e = lane; e < nface; e += 32) {
            const int f = s_face[warp][e], ju = f & 3, j = ju >> 1, sigma = (ju & 1) ? 1 : -1;
            // wall value of face (x, j, sigma) (Eq. 6, rho'_s in FP64 from the partials of u_j of the quadrants
            // moving toward the wall), shifted by the source-form offset sigma dx on x1 faces (Eq. 5: alpha
            // times the diffuse value, through the alpha-scaled denominators; the specular part is added per
            // velocity by the sweep).  Case 1 (only the second upstream point solid) has no wall term.
            const double val = wall_density(P, id - lane + (f >> 2), j, sigma, P->dinvw) + (j == 0 ? (sigma < 0 ? -P->dx : P->dx) : 0.0);
            s_ev[warp][e] = (T)val;
        }
        __syncwarp();
        if (fluid) {
            T ev[4];
#pragma unroll
            for (int ju = 0; ju < 4; ++ju) ev[ju] = mine[ju] >= 0 ? s_ev[warp][mine[ju]] : T(0);
            reinterpret_cast<V*>(P->src)[id] = Vec4<T>::make(nu * rho, T(2) * nu * u1 + T(1), T(2) * nu * u2, T(0));
            reinterpret_cast<V*>(P->E)[id] = Vec4<T>::make(ev[0], ev[1], ev[2], ev[3]);
        }
        __syncwarp();
    }
    finish_u1_sum(P, sum1, s_red);
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
cudaError_t launch_finalize2d(const FinArgs2D<T>& a, int nblocks, int ppt, cudaStream_t st) {
    finalize2d_kernel<T><<<nblocks, 256, 0, st>>>(a, ppt);
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
    template cudaError_t launch_finalize2d<T>(const FinArgs2D<T>&, int, int, cudaStream_t);          \
    template cudaError_t launch_init2d<T>(const Prob2D<T>*, int, const double*, cudaStream_t);  \
    template cudaError_t launch_warm2d<T>(const Prob2D<T>*, int, int, const double*, const double*, \
                                          const double*, const double*, cudaStream_t);            \
    template cudaError_t launch_moments2d<T>(const Prob2D<T>*, double*, double*, cudaStream_t); \
    template cudaError_t launch_wall2d<T>(const Prob2D<T>*, double*, cudaStream_t);

DVM_INSTANTIATE(float)
DVM_INSTANTIATE(double)

}  // namespace dvm
