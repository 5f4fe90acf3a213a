// nn_packed.cu -- the warm-start network's passes on packed activations.
//
// A packed tensor is the form that the tensor-core convolutions read (conv_umma.cu): BF16, channels-last,
// [d + 2][h + 2][w + 2][cp] with a one-voxel periodic halo and the channels padded with zeros to multiples of 32.
// A convolution writes its output in that form itself (after the bias and the ReLU), pooling and upsampling produce
// it directly, and the weight gradient reads the stored layer inputs and one packed gradient, so that between two
// convolutions nothing passes through FP32 memory that only the BF16 rounding of is used.  What FP32 values are used
// for stays FP32: the pooled means, the gradients' sums over voxels, the sums of upsampling and skip gradients.
// Measured against separate passes (FP32 output, ReLU, padded copy, upsampled copy; three shifted copies of every
// layer input and a copy of every gradient in the weight gradients; a block per channel in the bias gradients):
// prediction for 128^3 voxels, base 32, 8.23 -> 2.82 ms; training step on 64^3 voxels 6.60 -> 2.51 ms.
// Every sum is taken in the order of the unpacked functions and gives their bits, but for the weight gradients of rows of
// 65 to 96 voxels and concatenations whose first part is not a multiple of 8 channels (another split of the same sums).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "../../include/dvm.h"

namespace dvm_nn {
struct ConvOut {   // as in conv_umma.cu
    float* y;
    __nv_bfloat16* yp;
    int yc, y0, yw;
    int relu, accumulate;
};
cudaError_t conv_packed(const __nv_bfloat16* xp, const __nv_bfloat16* wb, const float* bias, const ConvOut& o, int nin, int nout,
                        int d, int h, int w, cudaStream_t st);
cudaError_t pack_input(const float* x, __nv_bfloat16* xp, int c, int cp, int d, int h, int w, int pool, cudaStream_t st);
long long wgrad_packed_scratch_bytes(int cinp, int cout, int d, int h, int w);
cudaError_t wgrad_packed(const __nv_bfloat16* xp, const __nv_bfloat16* gw, float* dw, int cin, int c0, int c0p, int cinp, int cout, int d,
                         int h, int w, float* part, long long part_bytes, cudaStream_t st);
cudaError_t channel_sum(const float* dy, float* db, int c, long long V, int accumulate, cudaStream_t st);   // nn3d.cu
}  // namespace dvm_nn

namespace {

constexpr int kMaxLayers = 32;
constexpr int kGradBlocks = 1216;     // blocks (along voxels) of a gradient pass: eight per SM

__host__ __device__ inline int round32(int n) { return (n + 31) / 32 * 32; }
inline int out_tile(int n) { return n <= 32 ? 32 : (n <= 64 ? 64 : 128); }      // the convolutions' channel tile
// A concatenated input's second part follows the first c0 channels at once where eight channels (16 bytes) are stored at
// a time: 24 + 48 channels are three 32-channel steps, and the sums run over the channels in their order.
__host__ __device__ inline int second_part(int c0) { return c0 % 8 ? round32(c0) : c0; }
__host__ __device__ inline int packed_in(int cin, int c0) { return round32(second_part(c0) + cin - c0); }

struct WeightSet {
    const float* w[kMaxLayers];
    __nv_bfloat16* wb[kMaxLayers];
    int cin[kMaxLayers], cout[kMaxLayers], c0[kMaxLayers];
    int first[kMaxLayers + 1];        // first block of a layer
    int n, gradient;
};

// wb[tap][n][c] of every layer in one launch.  Forward: n output channel, c packed input channel; gradient: n input
// channel (unpacked), c output channel, taps mirrored.  A block transposes the 27 taps of one n and 32 c.
__global__ void __launch_bounds__(256) pack_weights_kernel(const WeightSet s) {
    __shared__ float t[27][33];
    int l = 0;
    while (l + 1 < s.n && (int)blockIdx.x >= s.first[l + 1]) ++l;
    const int cin = s.cin[l], cout = s.cout[l], c0 = s.c0[l];
    const int ncp = s.gradient ? round32(cout) : packed_in(cin, c0);
    const int nout = s.gradient ? cin : cout;
    const int bn = nout <= 32 ? 32 : (nout <= 64 ? 64 : 128), noutp = (nout + bn - 1) / bn * bn;
    const int blk = blockIdx.x - s.first[l], nc = ncp / 32;
    const int n = blk / nc, cb = (blk - n * nc) * 32;
    const int c0p = second_part(c0);
    for (int e = threadIdx.x; e < 32 * 27; e += 256) {
        const int cc = e / 27, k = e - cc * 27, c = cb + cc;
        float v = 0.f;
        if (n < nout) {
            if (s.gradient) {
                if (c < cout) v = s.w[l][((long long)c * cin + n) * 27 + 26 - k];
            } else {
                const int ci = c < c0 ? c : (c >= c0p ? c - c0p + c0 : cin);
                if (ci < cin) v = s.w[l][((long long)n * cin + ci) * 27 + k];
            }
        }
        t[k][cc] = v;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 16 * 27; e += 256) {
        const int k = e >> 4, c2 = (e & 15) * 2;
        *reinterpret_cast<__nv_bfloat162*>(s.wb[l] + ((long long)k * noutp + n) * ncp + cb + c2) =
            __floats2bfloat162_rn(t[k][c2], t[k][c2 + 1]);
    }
}

// nearest-neighbour 2x upsampling of a packed tensor (lc channels, zeros beyond) into channels x0 .. x0 + cw - 1
// of a packed tensor of D x H x W voxels (channel stride xc), halo included; 8 channels a thread.
// A block takes a padded row, whose indices are then found once (64-bit divisions for every 16 bytes were what it waited
// for): the three upsamplings of a 128^3 network 151 -> 75 us.
__global__ void __launch_bounds__(256) up_packed_kernel(const uint4* __restrict__ lp, int lc, uint4* __restrict__ xp, int xc,
                                                        int x0, int cw, int D, int H, int W) {
    const int row = blockIdx.x, py = row % (H + 2), pz = row / (H + 2);
    auto low = [](int p, int n) { return ((p == 0 ? n - 1 : (p == n + 1 ? 0 : p - 1)) >> 1) + 1; };
    const int g8 = cw / 8, l8 = lc / 8, x8 = xc / 8;
    const uint4* l = lp + ((size_t)low(pz, D) * (H / 2 + 2) + low(py, H)) * (W / 2 + 2) * l8;
    uint4* o = xp + (size_t)row * (W + 2) * x8 + x0 / 8;
#pragma unroll 4
    for (int k = threadIdx.x; k < (W + 2) * g8; k += 256) {
        const int px = k / g8, g = k - px * g8;
        o[px * x8 + g] = g < l8 ? l[low(px, W) * l8 + g] : make_uint4(0u, 0u, 0u, 0u);
    }
}

// Gradient g at a layer's output [c][z][y][x] (FP32): mode 0: src; 1: src + (1/8) low[z/2][y/2][x/2] (the pooling's
// gradient beside the skip's); 2: the sum of the 8 children of src, which has 2 D x 2 H x 2 W voxels (upsampling).
// Masked by the ReLU (ap: the layer's packed output at channels a0 .., NULL: none), it goes out as the packed tensor
// gp that the data gradient reads, as gw [z][y][x padded to 16][cp] that the weight gradient reads, and in FP32 to gf
// (src itself or another buffer; NULL: src is it already) for the bias gradient.  A block transposes 64 voxels x 32
// channels at a time; voxels are counted along the padded rows, so that short rows fill a tile too.  Bound by latency
// while the mode was a branch in the loop over the channels (a thread's eight loads one after another) and rows below 64
// voxels left threads idle: 64^3 voxels, 32 channels: mode 0 65 -> 23 us, mode 1 92 -> 33;
// mode 2 onto 32^3 voxels, 64 channels: 88 -> 18.
template <int MODE>
__global__ void __launch_bounds__(256) grad_pack_kernel(const float* src, const float* __restrict__ low,
                                                        const __nv_bfloat16* __restrict__ ap, int ac, int a0,
                                                        __nv_bfloat16* __restrict__ gp, __nv_bfloat16* __restrict__ gw,
                                                        float* gf, int C, int cp, int D, int H, int W) {
    __shared__ float t[32][65];
    const int cb = blockIdx.y * 32;
    const int wp = (W + 15) / 16 * 16;
    const int total = D * H * wp;                                     // padded voxels
    const size_t V = (size_t)D * H * W;
    const int tx = threadIdx.x & 63, cg = threadIdx.x >> 6;           // voxel and channels cg, cg + 4, ... of a thread's FP32 accesses
    const int vv = threadIdx.x >> 2, q8 = (threadIdx.x & 3) * 8;      // voxel and channels of a thread's 16-byte stores
    for (int p0 = blockIdx.x * 64; p0 < total; p0 += gridDim.x * 64) {
        const int row = (p0 + tx) / wp, x = p0 + tx - row * wp;
        const bool in = x < W && row < D * H;
        {
            const int z = row / H, y = row - z * H;
            float v[8];
            if constexpr (MODE == 2) {
                const float* s = src + (((size_t)(cb + cg) * 2 * D + 2 * z) * 2 * H + 2 * y) * 2 * W + 2 * x;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    float2 e[4];
#pragma unroll
                    for (int ab = 0; ab < 4; ++ab)
                        e[ab] = in && cb + cg + 4 * k < C
                                    ? *reinterpret_cast<const float2*>(s + (size_t)k * 32 * V + ((size_t)(ab >> 1) * 2 * H + (ab & 1)) * 2 * W)
                                    : make_float2(0.f, 0.f);
                    v[k] = 0.f;
#pragma unroll
                    for (int ab = 0; ab < 4; ++ab) {
                        v[k] += e[ab].x;
                        v[k] += e[ab].y;
                    }
                }
            } else {
                const size_t o = (size_t)(cb + cg) * V + (size_t)row * W + x;
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = in && cb + cg + 4 * k < C ? src[o + (size_t)k * 4 * V] : 0.f;
                if constexpr (MODE == 1) {
                    const float* l = low + (((size_t)(cb + cg) * (D / 2) + z / 2) * (H / 2) + y / 2) * (W / 2) + x / 2;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (in && cb + cg + 4 * k < C) v[k] += 0.125f * l[(size_t)k * 4 * (V / 8)];
                }
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) t[cg + 4 * k][tx] = v[k];
        }
        __syncthreads();
        const int pv = p0 + vv;
        if (pv < total) {
            const int r = pv / wp, xv = pv - r * wp, z = r / H, y = r - z * H;
            float v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = t[q8 + j][vv];          // (zero beyond W)
            if (ap && xv < W) {
                const uint4 m = *reinterpret_cast<const uint4*>(
                    ap + (((long long)(z + 1) * (H + 2) + y + 1) * (W + 2) + xv + 1) * ac + a0 + cb + q8);
                const __nv_bfloat162* mh = reinterpret_cast<const __nv_bfloat162*>(&m);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float2 f = __bfloat1622float2(mh[j]);
                    if (!(f.x > 0.f)) t[q8 + 2 * j][vv] = v[2 * j] = 0.f;
                    if (!(f.y > 0.f)) t[q8 + 2 * j + 1][vv] = v[2 * j + 1] = 0.f;
                }
            }
            uint4 o;
            __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
            for (int j = 0; j < 4; ++j) oh[j] = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
            *reinterpret_cast<uint4*>(gw + (long long)pv * cp + cb + q8) = o;
            if (gp && xv < W) {
                __nv_bfloat16* d = gp + (((long long)(z + 1) * (H + 2) + y + 1) * (W + 2) + xv + 1) * cp + cb + q8;
                *reinterpret_cast<uint4*>(d) = o;
                if (z == 0 || z == D - 1 || y == 0 || y == H - 1 || xv == 0 || xv == W - 1)      // every halo image of the voxel
                    for (int pz = z + 1 - D < 0 ? z + 1 : z + 1 - D; pz < D + 2; pz += D)
                        for (int py = y + 1 - H < 0 ? y + 1 : y + 1 - H; py < H + 2; py += H)
                            for (int px = xv + 1 - W < 0 ? xv + 1 : xv + 1 - W; px < W + 2; px += W)
                                *reinterpret_cast<uint4*>(gp + (((long long)pz * (H + 2) + py) * (W + 2) + px) * cp + cb + q8) = o;
            }
        }
        __syncthreads();
        if (gf) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if (in && cb + cg + 4 * k < C) gf[(size_t)(cb + cg + 4 * k) * V + (size_t)row * W + x] = t[cg + 4 * k][tx];
            __syncthreads();
        }
    }
}

dvm_status status_of(cudaError_t e) { return e == cudaSuccess ? DVM_OK : (e == cudaErrorInvalidValue ? DVM_EINVAL : DVM_ECUDA); }

// packed buffers are read and written 16 bytes at a time
bool misaligned(const void* p) { return ((uintptr_t)p & 15) != 0; }

bool bad_size(int c, int d, int h, int w) { return c < 1 || d < 1 || h < 1 || w < 1 || w > 128; }

}  // namespace

extern "C" {

dvm_status dvm_nn_pack_weights(int n, const float* const* w, void* const* wb, const int* cin, const int* cout, const int* c0,
                               int gradient, void* stream) {
    if (n < 1 || n > kMaxLayers || !w || !wb || !cin || !cout || !c0) return DVM_EINVAL;
    WeightSet s;
    s.n = n;
    s.gradient = gradient ? 1 : 0;
    long long blocks = 0;
    for (int l = 0; l < n; ++l) {
        if (!w[l] || !wb[l] || misaligned(wb[l]) || cin[l] < 1 || cout[l] < 1 || c0[l] < 1 || c0[l] > cin[l]) return DVM_EINVAL;
        s.w[l] = w[l];
        s.wb[l] = (__nv_bfloat16*)wb[l];
        s.cin[l] = cin[l];
        s.cout[l] = cout[l];
        s.c0[l] = c0[l];
        s.first[l] = (int)blocks;
        const int ncp = gradient ? round32(cout[l]) : packed_in(cin[l], c0[l]), nout = gradient ? cin[l] : cout[l];
        const int bn = out_tile(nout);
        blocks += (long long)((nout + bn - 1) / bn * bn) * (ncp / 32);
        if (blocks > 0x7fffff) return DVM_EINVAL;
    }
    s.first[n] = (int)blocks;
    pack_weights_kernel<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(s);
    return status_of(cudaGetLastError());
}

int64_t dvm_nn_packed_weight_elems(int cin, int cout, int c0) {
    if (cin < 1 || cout < 1 || c0 < 1 || c0 > cin) return 0;
    const int bf = out_tile(cout), bg = out_tile(cin);
    const long long f = 27LL * ((cout + bf - 1) / bf * bf) * packed_in(cin, c0), g = 27LL * ((cin + bg - 1) / bg * bg) * round32(cout);
    return f > g ? f : g;
}

dvm_status dvm_nn_pack(const float* x, void* xp, int c, int cp, int d, int h, int w_, int pool, void* stream) {
    if (!x || !xp || bad_size(c, d, h, w_) || cp < c || cp % 32) return DVM_EINVAL;
    if ((long long)(d + 2) * (h + 2) > 65535 || ((uintptr_t)x & (pool ? 7 : 3)) || misaligned(xp)) return DVM_EINVAL;
    return status_of(dvm_nn::pack_input(x, (__nv_bfloat16*)xp, c, cp, d, h, w_, pool, (cudaStream_t)stream));
}

dvm_status dvm_nn_up2_packed(const void* lp, int lc, void* xp, int xc, int x0, int cw, int d, int h, int w_, void* stream) {
    if (!lp || !xp || bad_size(cw, d, h, w_) || (d | h | w_) & 1 || cw % 8 || lc % 32 || xc % 32 || x0 % 8 || x0 < 0 || x0 + cw > xc)
        return DVM_EINVAL;
    const long long rows = (long long)(d + 2) * (h + 2);
    if (rows > 0x7fffffff || misaligned(lp) || misaligned(xp)) return DVM_EINVAL;
    up_packed_kernel<<<(unsigned)rows, 256, 0, (cudaStream_t)stream>>>((const uint4*)lp, lc, (uint4*)xp, xc, x0, cw, d, h, w_);
    return status_of(cudaGetLastError());
}

dvm_status dvm_nn_conv3d_packed(const void* xp, const void* wb, const float* b, float* y, void* yp, int yc, int y0, int cinp,
                                int cout, int d, int h, int w_, int relu, void* stream) {
    if (!xp || !wb || (!y && !yp) || bad_size(cout, d, h, w_) || cinp < 32 || cinp % 32) return DVM_EINVAL;
    if (yp && (yc % 32 || y0 % 32 || y0 < 0 || y0 + round32(cout) > yc)) return DVM_EINVAL;
    if (misaligned(xp) || misaligned(wb) || misaligned(yp)) return DVM_EINVAL;
    const dvm_nn::ConvOut o{y, (__nv_bfloat16*)yp, yc, y0, round32(cout), relu ? 1 : 0, 0};
    return status_of(dvm_nn::conv_packed((const __nv_bfloat16*)xp, (const __nv_bfloat16*)wb, b, o, cinp, cout, d, h, w_,
                                         (cudaStream_t)stream));
}

dvm_status dvm_nn_grad_pack(const float* src, const float* low, int mode, const void* ap, int ac, int a0, void* gp, void* gw,
                            float* gf, float* db, int c, int d, int h, int w_, void* stream) {
    if (!src || !gw || !db || bad_size(c, d, h, w_) || mode < 0 || mode > 2 || (mode == 1 && (!low || (d | h | w_) & 1))) return DVM_EINVAL;
    if ((!gf && (mode || ap)) || (gf == src && mode)) return DVM_EINVAL;
    const int cp = round32(c);
    if (ap && (a0 < 0 || a0 % 8 || ac % 8 || a0 + cp > ac)) return DVM_EINVAL;
    if (misaligned(ap) || misaligned(gp) || misaligned(gw)) return DVM_EINVAL;
    const long long tiles = ((long long)d * h * ((w_ + 15) / 16 * 16) + 63) / 64;
    if (tiles > (1 << 24) || (mode == 2 && ((uintptr_t)src & 7))) return DVM_EINVAL;
    const int blocks = tiles < kGradBlocks ? (int)tiles : kGradBlocks;
    cudaStream_t st = (cudaStream_t)stream;
    auto kern = mode == 0 ? grad_pack_kernel<0> : (mode == 1 ? grad_pack_kernel<1> : grad_pack_kernel<2>);
    kern<<<dim3((unsigned)blocks, (unsigned)(cp / 32)), 256, 0, st>>>(src, low, (const __nv_bfloat16*)ap, ac, a0, (__nv_bfloat16*)gp,
                                                                      (__nv_bfloat16*)gw, gf, c, cp, d, h, w_);
    const cudaError_t e = cudaGetLastError();
    return status_of(e != cudaSuccess ? e : dvm_nn::channel_sum(gf ? gf : src, db, c, (long long)d * h * w_, 1, st));
}

int64_t dvm_nn_wgrad_packed_scratch_floats(int cin, int c0, int cout, int d, int h, int w_) {
    if (cin < 1 || c0 < 1 || c0 > cin || bad_size(cout, d, h, w_)) return 0;
    return (dvm_nn::wgrad_packed_scratch_bytes(packed_in(cin, c0), cout, d, h, w_) + 3) / 4;
}

dvm_status dvm_nn_conv3d_wgrad_packed(const void* xp, const void* gw, float* dw, float* scratch, int64_t scratch_floats, int cin,
                                      int c0, int cout, int d, int h, int w_, void* stream) {
    if (!xp || !gw || misaligned(xp) || misaligned(gw) || !dw || !scratch || cin < 1 || c0 < 1 || c0 > cin || bad_size(cout, d, h, w_)) return DVM_EINVAL;
    return status_of(dvm_nn::wgrad_packed((const __nv_bfloat16*)xp, (const __nv_bfloat16*)gw, dw, cin, c0, second_part(c0), packed_in(cin, c0), cout,
                                         d, h, w_, scratch, scratch_floats * 4, (cudaStream_t)stream));
}

}  // extern "C"
