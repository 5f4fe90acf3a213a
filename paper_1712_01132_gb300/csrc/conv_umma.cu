// conv_umma.cu -- the warm-start network's 3 x 3 x 3 periodic convolutions as implicit GEMMs on the
// fifth-generation tensor cores (tcgen05.mma, BF16 operands, FP32 accumulators in tensor memory).
//
//   y[co][v] (+)= b[co] + sum_ci sum_k w[co][ci][k] x[ci][v + off(k)]
//
// GEMM view: M = voxels (a tile of `by` whole x rows of one z plane, at most 128 voxels, one per
// TMEM lane), N = output channels (a tile of BN), K = 27 taps x input channels (chunks of 32).
// Before the GEMM the input is written once as a BF16, channels-last copy with a one-voxel
// periodic halo, xp[z + 1][y + 1][x + 1][c] (channels padded to a multiple of 32 with zeros), and
// the weights as BF16 wb[tap][co][ci] (padded likewise): the A operand of a tap and channel chunk
// is then one box of xp (32 channels x W x by x 1) and the B operand one box of wb (32 x BN x 1),
// both brought to shared memory by the tensor memory accelerator (cp.async.bulk.tensor, 64-byte
// swizzle, the K-major layout tcgen05.mma reads).  One thread streams the boxes through a ring of
// stages, one thread issues the MMAs (K = 16 each, accumulating in TMEM) and releases a stage when
// its MMAs complete (tcgen05.commit); the four warps then read the accumulators back (tcgen05.ld,
// each warp its 32 lanes) and write y channel-major.  Every wait is bounded (a device status word
// records an expiry and the CTA returns after releasing its tensor memory).
//
// The data gradient is the same convolution of dy with the transposed channel roles and mirrored
// taps (wb[tap][ci][co] = w[co][ci][26 - tap]).
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

namespace dvm_nn {

constexpr int kBM = 128;       // GEMM rows per tile (TMEM lanes)
constexpr int kBK = 32;        // input channels per K chunk: 64-byte rows
constexpr int kStages = 4;
constexpr int kThreads = 128;
constexpr long long kTimeoutNs = 2000000000LL;

struct ConvGeom {
    int cin, cout;        // channels of this convolution's input and output
    int D, H, W;
    int cinp, coutp;      // padded to multiples of kBK and of BN
    int by, ytiles;       // x rows per tile, tiles per z plane
    int nk;               // K chunks per tap
};

// What a convolution writes: FP32 channel-major (y, optional) and / or the packed BF16 form that the next
// convolution reads (yp, optional: channels-last with a one-voxel periodic halo, channel stride yc, channels
// y0 .. y0 + yw - 1, yw = cout rounded up to 32 and zero beyond cout), after the bias and an optional ReLU.
struct ConvOut {
    float* y;
    __nv_bfloat16* yp;
    int yc, y0, yw;
    int relu, accumulate;
};

// the 16 channels c0 .. c0 + 15 (of n0 + ...) of voxel (z, y, x)
__device__ __forceinline__ void conv_store16(const unsigned (&a)[16], int co, int z, int yy, int xx, const float* __restrict__ bias,
                                             const ConvGeom& g, const ConvOut& o) {
    float val[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        val[j] = __uint_as_float(a[j]) + ((bias && co + j < g.cout) ? bias[co + j] : 0.f);
        if (o.relu) val[j] = fmaxf(val[j], 0.f);
    }
    if (o.y) {
        const long long V = (long long)g.D * g.H * g.W;
        float* d = o.y + (long long)co * V + ((long long)z * g.H + yy) * g.W + xx;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (co + j < g.cout) d[j * V] = o.accumulate ? d[j * V] + val[j] : val[j];
    }
    if (o.yp && co < o.yw) {
        uint4 q[2];
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(q);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            h[j] = __floats2bfloat162_rn(co + 2 * j < g.cout ? val[2 * j] : 0.f, co + 2 * j + 1 < g.cout ? val[2 * j + 1] : 0.f);
        auto put = [&](int pz, int py, int px) {
            uint4* d = reinterpret_cast<uint4*>(o.yp + (((long long)pz * (g.H + 2) + py) * (g.W + 2) + px) * o.yc + o.y0 + co);
            d[0] = q[0];
            d[1] = q[1];
        };
        put(z + 1, yy + 1, xx + 1);
        if (z == 0 || z == g.D - 1 || yy == 0 || yy == g.H - 1 || xx == 0 || xx == g.W - 1) {   // its halo images
            for (int pz = z + 1 - g.D; pz < g.D + 2; pz += g.D)
                for (int py = yy + 1 - g.H; py < g.H + 2; py += g.H)
                    for (int px = xx + 1 - g.W; px < g.W + 2; px += g.W)
                        if (pz >= 0 && py >= 0 && px >= 0 && !(pz == z + 1 && py == yy + 1 && px == xx + 1)) put(pz, py, px);
        }
    }
}

__device__ int g_conv_status;   // nonzero after a bounded wait expired

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long gtime() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// bounded wait for the phase with the given parity to complete; false on expiry
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity) {
    const unsigned a = smem_u32(bar);
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(a), "r"(parity) : "memory");
        if (done) return true;
        if ((it & 255u) == 0u) {
            const unsigned long long t = gtime();
            if (it == 0) t0 = t;
            else if ((long long)(t - t0) > kTimeoutNs) return false;
            if (*reinterpret_cast<volatile int*>(&g_conv_status) != 0 && it > 0) return false;
        }
    }
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                            uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
                   "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2),
                   "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1, int c2, int c3, int c4,
                                            uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
                 ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4),
                   "r"(smem_u32(bar))
                 : "memory");
}

// shared-memory matrix descriptor of a K-major operand in the 64-byte swizzled layout: rows of 64
// bytes, eight-row groups 512 bytes apart (stride byte offset), descriptor version 1
__device__ __forceinline__ uint64_t smem_desc_sw64(const void* p) {
    const uint64_t addr = (smem_u32(p) >> 4) & 0x3FFFu;
    return addr | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// instruction descriptor: FP32 accumulator, BF16 A and B, both K-major, M = 128, N = BN
template <int BN>
__device__ __forceinline__ unsigned idesc_bf16() {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(BN >> 3) << 17) | ((unsigned)(kBM >> 4) << 24);
}

__device__ __forceinline__ void umma_bf16(unsigned tmem_d, uint64_t adesc, uint64_t bdesc, unsigned idesc, int acc) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
                 : "memory");
}

// the mbarrier completes one phase when every MMA this thread issued so far has finished
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// MT row tiles per CTA share every B box and write MT accumulators (TMEM columns t BN .. t BN + BN - 1)
template <int BN, int MT, int GRP, int NST>
__global__ void __launch_bounds__(kThreads) conv3d_umma_kernel(const __grid_constant__ CUtensorMap tmA,
                                                               const __grid_constant__ CUtensorMap tmB,
                                                               const float* __restrict__ bias, const ConvOut o,
                                                               const ConvGeom g) {
    constexpr int kABytes = kBM * kBK * 2;            // 8 KB per row tile
    constexpr int kBBytes = BN * kBK * 2;
    constexpr int kEntryBytes = MT * kABytes + kBBytes;   // a multiple of 1024 (BN multiple of 16)
    constexpr int kStageBytes = GRP * kEntryBytes;        // GRP entries (tap, chunk), one after the other
    static_assert(27 % GRP == 0, "whole stages");
    constexpr unsigned kTmemCols = MT * BN <= 32 ? 32u : (MT * BN <= 64 ? 64u : (MT * BN <= 128 ? 128u : 256u));
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sbase = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[NST], empty[NST], done;
    __shared__ unsigned s_tmem;
    __shared__ int s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.y * BN;
    const int rows = g.by * g.W;                      // valid GEMM rows of a tile (<= 128)
    int tz[MT], ty0[MT];                              // row tile t: z plane and first y row
#pragma unroll
    for (int t = 0; t < MT; ++t) {
        const int tile = blockIdx.x * MT + t;         // beyond the grid: z >= D, never written
        tz[t] = tile / g.ytiles;
        ty0[t] = (tile - tz[t] * g.ytiles) * g.by;
    }

    if (rows < kBM) {   // rows beyond the boxes stay zero in every stage (the boxes never write them)
        for (int i = threadIdx.x * 16; i < NST * kStageBytes; i += kThreads * 16)
            *reinterpret_cast<uint4*>(sbase + i) = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before the tensor cores read them
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_d = s_tmem;
    const int niter = 27 / GRP * g.nk;
    const unsigned box_bytes = (unsigned)(GRP * (MT * kBK * 2 * g.W * g.by + kBBytes));

    if (warp == 0 && lane == 0) {
        // producer: the A box of (tap, chunk) and the B box of the same (tap, chunk) per entry
        for (int i = 0; i < niter; ++i) {
            const int s = i % NST;
            if (i >= NST && !mbar_wait(&empty[s], ((i / NST) - 1) & 1)) {
                s_fail = 1;
                break;
            }
            mbar_expect_tx(&full[s], box_bytes);
#pragma unroll
            for (int j = 0; j < GRP; ++j) {
                const int e = GRP * i + j, tap = e / g.nk, kc = e - tap * g.nk;
                const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
                unsigned char* st = sbase + (size_t)s * kStageBytes + j * kEntryBytes;
#pragma unroll
                for (int t = 0; t < MT; ++t)
                    tma_load_4d(st + t * kABytes, &tmA, kc * kBK, 1 + dx, ty0[t] + 1 + dy, tz[t] + 1 + dz, &full[s]);
                tma_load_3d(st + MT * kABytes, &tmB, kc * kBK, n0, tap, &full[s]);
            }
        }
    } else if (warp == 1 && lane == 0) {
        // MMA issuer: K = 16 per instruction, two per chunk; the first one overwrites the accumulator
        const unsigned idesc = idesc_bf16<BN>();
        for (int i = 0; i < niter; ++i) {
            const int s = i % NST;
            if (!mbar_wait(&full[s], (i / NST) & 1)) {
                s_fail = 1;
                break;
            }
            tc_fence_after();
#pragma unroll
            for (int j = 0; j < GRP; ++j) {
                const unsigned char* st = sbase + (size_t)s * kStageBytes + j * kEntryBytes;
                const uint64_t bd = smem_desc_sw64(st + MT * kABytes);
#pragma unroll
                for (int t = 0; t < MT; ++t) {
                    const uint64_t ad = smem_desc_sw64(st + t * kABytes);
#pragma unroll
                    for (int kk = 0; kk < kBK / 16; ++kk)    // 32 bytes of K per step: +2 in the 16-byte address field
                        umma_bf16(tmem_d + t * BN, ad + 2 * kk, bd + 2 * kk, idesc, (i > 0 || j > 0 || kk > 0) ? 1 : 0);
                }
            }
            umma_commit(&empty[s]);
        }
        umma_commit(&done);
    }
    __syncwarp();
    const bool ok = mbar_wait(&done, 0);
    tc_fence_after();
    if (!ok || s_fail) {
        if (threadIdx.x == 0) atomicCAS(&g_conv_status, 0, -4);
    } else {
        // accumulator row r of tile t = voxel r of the tile (TMEM lane r), column t BN + j = output
        // channel n0 + j
        const int r = warp * 32 + lane;
#pragma unroll
        for (int t = 0; t < MT; ++t) {
        const int yy = ty0[t] + r / g.W, xx = r % g.W;
        const bool valid = r < rows && yy < g.H && tz[t] < g.D;
#pragma unroll
        for (int c0 = 0; c0 < BN; c0 += 16) {
            unsigned a[16];
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                         "%13, %14, %15}, [%16];"
                         : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
                           "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]),
                           "=r"(a[14]), "=r"(a[15])
                         : "r"(tmem_d + ((unsigned)(32 * warp) << 16) + (unsigned)(t * BN + c0))
                         : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (valid) conv_store16(a, n0 + c0, tz[t], yy, xx, bias, g, o);
        }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(kTmemCols) : "memory");
}

// The same convolution with the A operand shared by the three y taps: when a tile is whole x rows
// (W a multiple of 8 dividing 128, by = 128 / W rows) and a CTA's MT tiles are consecutive rows of one z plane, one box of MT by + 2 rows (the tiles' rows and a halo row on each side) per (dz, dx,
// channel chunk) holds the A rows of all three dy taps: tap dy of tile t starts (t by + dy + 1) W
// rows into the box, a multiple of eight 64-byte rows, so it is a plain shift of the swizzled
// operand's start address.  A stage is that box and the three dy taps' B boxes: 9 stages per chunk
// instead of 27, and a third of the A bytes per tap.
template <int BN, int MT, int NST>
__global__ void __launch_bounds__(kThreads) conv3d_umma_dy_kernel(const __grid_constant__ CUtensorMap tmA,
                                                                  const __grid_constant__ CUtensorMap tmB,
                                                                  const float* __restrict__ bias, const ConvOut o,
                                                                  const ConvGeom g, int abox_bytes, int stage_bytes) {
    constexpr int kBBytes = BN * kBK * 2;
    constexpr unsigned kTmemCols = MT * BN <= 32 ? 32u : (MT * BN <= 64 ? 64u : (MT * BN <= 128 ? 128u : 256u));
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sbase = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[NST], empty[NST], done;
    __shared__ unsigned s_tmem;
    __shared__ int s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.y * BN;
    const int tile0 = blockIdx.x * MT;                // first tile: z plane, first y row
    const int z = tile0 / g.ytiles;
    const int yb = (tile0 - z * g.ytiles) * g.by;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_d = s_tmem;
    const int niter = 9 * g.nk;                       // (dz, dx) x channel chunks
    const unsigned box_bytes = (unsigned)(abox_bytes + 3 * kBBytes);

    if (warp == 0 && lane == 0) {
        // producer: the A box of (dz, dx, chunk) and the B boxes of its three dy taps per stage
        for (int i = 0; i < niter; ++i) {
            const int s = i % NST;
            if (i >= NST && !mbar_wait(&empty[s], ((i / NST) - 1) & 1)) {
                s_fail = 1;
                break;
            }
            const int zx = i / g.nk, kc = i - zx * g.nk;
            const int dz = zx / 3 - 1, dx = zx % 3 - 1;
            unsigned char* st = sbase + (size_t)s * stage_bytes;
            mbar_expect_tx(&full[s], box_bytes);
            tma_load_4d(st, &tmA, kc * kBK, 1 + dx, yb, z + 1 + dz, &full[s]);   // padded rows yb .. yb + MT by + 1
#pragma unroll
            for (int j = 0; j < 3; ++j)
                tma_load_3d(st + abox_bytes + j * kBBytes, &tmB, kc * kBK, n0, (dz + 1) * 9 + j * 3 + (dx + 1), &full[s]);
        }
    } else if (warp == 1 && lane == 0) {
        // MMA issuer: per stage, for each dy tap and row tile two K = 16 steps
        const unsigned idesc = idesc_bf16<BN>();
        for (int i = 0; i < niter; ++i) {
            const int s = i % NST;
            if (!mbar_wait(&full[s], (i / NST) & 1)) {
                s_fail = 1;
                break;
            }
            tc_fence_after();
            const unsigned char* st = sbase + (size_t)s * stage_bytes;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const uint64_t bd = smem_desc_sw64(st + abox_bytes + j * kBBytes);
#pragma unroll
                for (int kk = 0; kk < kBK / 16; ++kk)
#pragma unroll
                    for (int t = 0; t < MT; ++t) {
                        const uint64_t ad = smem_desc_sw64(st + (size_t)((t * g.by + j) * g.W) * (kBK * 2));
                        umma_bf16(tmem_d + t * BN, ad + 2 * kk, bd + 2 * kk, idesc, (i > 0 || j > 0 || kk > 0) ? 1 : 0);
                    }
            }
            umma_commit(&empty[s]);
        }
        umma_commit(&done);
    }
    __syncwarp();
    const bool ok = mbar_wait(&done, 0);
    tc_fence_after();
    if (!ok || s_fail) {
        if (threadIdx.x == 0) atomicCAS(&g_conv_status, 0, -4);
    } else {
        // accumulator row r of tile t = voxel r of the tile (TMEM lane r), column t BN + j = output
        // channel n0 + j; every row of every tile is a voxel (by W = 128, whole tiles)
        const int r = warp * 32 + lane;
#pragma unroll
        for (int t = 0; t < MT; ++t) {
            const int yy = yb + t * g.by + r / g.W, xx = r % g.W;
#pragma unroll
            for (int c0 = 0; c0 < BN; c0 += 16) {
                unsigned a[16];
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                             "%13, %14, %15}, [%16];"
                             : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
                               "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]),
                               "=r"(a[14]), "=r"(a[15])
                             : "r"(tmem_d + ((unsigned)(32 * warp) << 16) + (unsigned)(t * BN + c0))
                             : "memory");
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                conv_store16(a, n0 + c0, z, yy, xx, bias, g, o);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(kTmemCols) : "memory");
}

// xp[pz][py][px][c] = bf16(v[c][pz - 1][py - 1][px - 1]) with periodic wrap, zero for c >= cin, where v is x or (POOL)
// its 2 x 2 x 2 mean (x then has 2 D x 2 H x 2 W voxels).  A block transposes 64 padded voxels of one z plane by 32
// channels through shared memory: reads are coalesced along x, and four threads write the 64 bytes of a voxel.
// Voxels are counted along the padded plane: with a row of W + 2 per group of blocks, 128 + 2 voxels filled two of
// three blocks.  A thread's eight loads are issued together.  128^3 voxels, 3 channels: 91 -> 62 us;
// the three poolings of a 128^3 network 113 -> 83.
template <bool POOL>
__global__ void __launch_bounds__(256) pad_bf16_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ xp,
                                                       int cin, int cinp, int D, int H, int W) {
    __shared__ float t[32][65];
    const int plane = (H + 2) * (W + 2), p0 = blockIdx.x * 64, pz = blockIdx.y, c0 = blockIdx.z * 32;
    {
        const int p = p0 + (threadIdx.x & 63), cc = threadIdx.x >> 6;
        const int py = p / (W + 2), px = p - py * (W + 2);
        const int sx = px == 0 ? W - 1 : (px == W + 1 ? 0 : px - 1);
        const int sy = py == 0 ? H - 1 : (py == H + 1 ? 0 : py - 1);
        const int sz = pz == 0 ? D - 1 : (pz == D + 1 ? 0 : pz - 1);
        const size_t V = (size_t)D * H * W;            // of the result
        float v[8];
        if constexpr (POOL) {
            const float* xc = x + (((size_t)(c0 + cc) * 2 * D + 2 * sz) * 2 * H + 2 * sy) * 2 * W + 2 * sx;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                float2 e[4];
#pragma unroll
                for (int ab = 0; ab < 4; ++ab)
                    e[ab] = p < plane && c0 + cc + 4 * k < cin
                                ? *reinterpret_cast<const float2*>(xc + (size_t)k * 32 * V + ((size_t)(ab >> 1) * 2 * H + (ab & 1)) * 2 * W)
                                : make_float2(0.f, 0.f);
                float s = 0.f;
#pragma unroll
                for (int ab = 0; ab < 4; ++ab) {
                    s += e[ab].x;
                    s += e[ab].y;
                }
                v[k] = 0.125f * s;
            }
        } else {
            const float* xc = x + (size_t)(c0 + cc) * V + ((size_t)sz * H + sy) * W + sx;
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = p < plane && c0 + cc + 4 * k < cin ? xc[(size_t)k * 4 * V] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) t[cc + 4 * k][threadIdx.x & 63] = v[k];
    }
    __syncthreads();
    const int vv = threadIdx.x >> 2, q = threadIdx.x & 3;
    if (p0 + vv < plane) {
        uint4 o;
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
        for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(t[8 * q + 2 * j][vv], t[8 * q + 2 * j + 1][vv]);
        *reinterpret_cast<uint4*>(xp + ((size_t)pz * plane + p0 + vv) * cinp + c0 + 8 * q) = o;
    }
}

inline dim3 pad_grid(int cinp, int d, int h, int w) {
    return dim3((unsigned)(((h + 2) * (w + 2) + 63) / 64), (unsigned)(d + 2), (unsigned)(cinp / 32));
}

// wb[tap][n][c] = bf16(w[n sn + c sc + (flip ? 26 - tap : tap)]) for n < nout, c < nin, else 0
__global__ void weights_bf16_kernel(const float* __restrict__ w, __nv_bfloat16* __restrict__ wb, int nout, int nin,
                                    int noutp, int ninp, int sn, int sc, int flip) {
    const long long total = 27LL * noutp * ninp;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int c = (int)(i % ninp);
    const int n = (int)((i / ninp) % noutp);
    const int tap = (int)(i / ((long long)ninp * noutp));
    float val = 0.f;
    if (n < nout && c < nin) val = w[(long long)n * sn + (long long)c * sc + (flip ? 26 - tap : tap)];
    wb[i] = __float2bfloat16_rn(val);
}

using EncodeFn = PFN_cuTensorMapEncodeTiled_v12000;

EncodeFn encode_fn() {
    static EncodeFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeFn>(p);
    });
    return fn;
}

inline int bn_for(int cout) { return cout <= 32 ? 32 : (cout <= 64 ? 64 : 128); }
inline long long align1k(long long b) { return (b + 1023) & ~1023LL; }

template <int BN, int MT, int GRP, int NST>
cudaError_t launch_bn(const CUtensorMap& ta, const CUtensorMap& tb, const float* bias, const ConvOut& o, const ConvGeom& g,
                      cudaStream_t st) {
    const int smem = NST * GRP * (MT * kBM * kBK * 2 + BN * kBK * 2) + 1024;
    auto kern = conv3d_umma_kernel<BN, MT, GRP, NST>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    const int tiles = g.D * g.ytiles;
    dim3 grid((unsigned)((tiles + MT - 1) / MT), (unsigned)((g.cout + BN - 1) / BN));
    kern<<<grid, kThreads, smem, st>>>(ta, tb, bias, o, g);
    return cudaGetLastError();
}

template <int BN, int MT, int NST>
cudaError_t launch_dy(const CUtensorMap& ta, const CUtensorMap& tb, const float* bias, const ConvOut& o, const ConvGeom& g,
                      cudaStream_t st) {
    const int abox = (MT * g.by + 2) * g.W * kBK * 2;
    const int stage = (abox + 3 * BN * kBK * 2 + 1023) / 1024 * 1024;
    const int smem = NST * stage + 1024;
    auto kern = conv3d_umma_dy_kernel<BN, MT, NST>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)(g.D * g.ytiles / MT), (unsigned)((g.cout + BN - 1) / BN));
    kern<<<grid, kThreads, smem, st>>>(ta, tb, bias, o, g, abox, stage);
    return cudaGetLastError();
}

}  // namespace dvm_nn

// Scratch bytes of one convolution with nin input and nout output channels on a d x h x w grid: the
// padded BF16 input copy and the BF16 weights, each 1 KB aligned.
long long conv_umma_scratch_bytes(int nin, int nout, int d, int h, int w) {
    using namespace dvm_nn;
    const int cinp = (nin + kBK - 1) / kBK * kBK;
    const int bn = bn_for(nout);
    const int coutp = (nout + bn - 1) / bn * bn;
    return align1k((long long)(d + 2) * (h + 2) * (w + 2) * cinp * 2) + align1k(27LL * coutp * cinp * 2) + 1024;
}

namespace dvm_nn {

// The convolution of a packed input xp (channels-last BF16 with halo, g.cinp channels) with packed weights wb.
cudaError_t conv_packed(const __nv_bfloat16* xp, const __nv_bfloat16* wb, const float* bias, const ConvOut& o, int nin, int nout,
                        int d, int h, int w_, cudaStream_t st) {
    EncodeFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    ConvGeom g;
    g.cin = nin;
    g.cout = nout;
    g.D = d;
    g.H = h;
    g.W = w_;
    g.cinp = (nin + kBK - 1) / kBK * kBK;
    int bn = bn_for(nout);
    g.coutp = (nout + bn - 1) / bn * bn;
    g.by = kBM / w_ < h ? kBM / w_ : h;
    g.ytiles = (h + g.by - 1) / g.by;
    g.nk = g.cinp / kBK;
    // Whole-row tiles of 128 voxels in pairs (single ones with more than 64 output channels): the A box is shared by the
    // dy taps.  The rule decides the order in which the taps are summed as well, so it does not follow the tile chosen
    // below: a network's rounding does not depend on how a layer is spread over the chip.
    const bool whole = w_ % 8 == 0 && kBM % w_ == 0 && g.by * w_ == kBM && h % g.by == 0 && g.ytiles % (bn == 128 ? 1 : 2) == 0;
    // Two row tiles per CTA share a weight box (four on large grids, see below, one with 128 output channels); a grid
    // with fewer CTAs than SMs takes one, then fewer channels per CTA: every CTA runs all taps and input channels in
    // turn, so on the small grids of the deep levels it is their number that counts (256 -> 256 channels on 8^3 voxels: 16 CTAs 70 us, 64 CTAs
    // 34 us; 128 -> 128 on 16^3: 32 CTAs 48 us, 128 CTAs 23 us).
    int mt = bn == 128 ? 1 : 2;
    if (nout % 128 > 64 && nout % 128 <= 96) bn = 96;              // (no columns of padding)
    else if (bn == 128 && nout % 128 > 0 && nout % 128 <= 64) bn = 64;
    auto ctas = [&] { return (long long)(d * g.ytiles + mt - 1) / mt * ((nout + bn - 1) / bn); };
    if (ctas() < 152) mt = 1;
    while (ctas() < 152 && bn > 32) bn = bn == 96 ? 32 : bn / 2;
    // four row tiles per CTA on grids of four waves of such CTAs or more (on 64^3, 512 CTAs, 46 us become 50)
    if (whole && bn == 32 && mt == 2 && g.ytiles % 4 == 0 && ctas() >= 2 * 4 * 304) mt = 4;
    CUtensorMap ta, tb;
    {
        const cuuint64_t dims[4] = {(cuuint64_t)g.cinp, (cuuint64_t)(w_ + 2), (cuuint64_t)(h + 2), (cuuint64_t)(d + 2)};
        const cuuint64_t strides[3] = {(cuuint64_t)g.cinp * 2, (cuuint64_t)g.cinp * 2 * (w_ + 2),
                                       (cuuint64_t)g.cinp * 2 * (w_ + 2) * (h + 2)};
        const cuuint32_t box[4] = {(cuuint32_t)kBK, (cuuint32_t)w_, (cuuint32_t)g.by, 1u};
        const cuuint32_t es[4] = {1u, 1u, 1u, 1u};
        if (enc(&ta, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(xp), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
            CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[3] = {(cuuint64_t)g.cinp, (cuuint64_t)g.coutp, 27u};
        const cuuint64_t strides[2] = {(cuuint64_t)g.cinp * 2, (cuuint64_t)g.cinp * 2 * g.coutp};
        const cuuint32_t box[3] = {(cuuint32_t)kBK, (cuuint32_t)bn, 1u};
        const cuuint32_t es[3] = {1u, 1u, 1u};
        if (enc(&tb, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(wb), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
            CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    if (whole) {
        CUtensorMap td;
        const cuuint64_t dims[4] = {(cuuint64_t)g.cinp, (cuuint64_t)(w_ + 2), (cuuint64_t)(h + 2), (cuuint64_t)(d + 2)};
        const cuuint64_t strides[3] = {(cuuint64_t)g.cinp * 2, (cuuint64_t)g.cinp * 2 * (w_ + 2),
                                       (cuuint64_t)g.cinp * 2 * (w_ + 2) * (h + 2)};
        const cuuint32_t box[4] = {(cuuint32_t)kBK, (cuuint32_t)w_, (cuuint32_t)(mt * g.by + 2), 1u};
        const cuuint32_t es[4] = {1u, 1u, 1u, 1u};
        if (enc(&td, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(xp), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
            CUDA_SUCCESS)
            return cudaErrorInvalidValue;
        // Stages: as few as let two CTAs share an SM (three on 64-wide rows), whose prologues and epilogues then run
        // beside the other's MMAs (a CTA's life is 10 to 18 us, a third of it outside its MMAs); six where a small grid
        // leaves an SM one CTA.  128^3 voxels, 32 -> 32 channels: 3 stages (115 KB, one CTA) 646 us, 2 stages 377, and
        // four row tiles 321 (an MMA of 32 columns takes longer than its operands: more of them in flight); 96 -> 32:
        // 1180, 729, 594; 64^3, 64 -> 64: 109, 98; 32 -> 96: 75, 67.  With one row tile and 64 or 128 channels a third
        // stage gains 5 to 20 %; four tiles of 64 channels or two of 128 lose 10 to 60 %.
        if (mt == 4) return launch_dy<32, 4, 2>(td, tb, bias, o, g, st);
        if (bn == 32) return mt == 2 ? launch_dy<32, 2, 2>(td, tb, bias, o, g, st) : launch_dy<32, 1, 6>(td, tb, bias, o, g, st);
        if (bn == 64) return mt == 2 ? launch_dy<64, 2, 2>(td, tb, bias, o, g, st) : launch_dy<64, 1, 3>(td, tb, bias, o, g, st);
        if (bn == 96) return launch_dy<96, 1, 2>(td, tb, bias, o, g, st);
        return launch_dy<128, 1, 3>(td, tb, bias, o, g, st);
    }
    // One tile of 32 channels a CTA and at most one CTA an SM: nine entries a stage, since a stage's wait and commit cost as
    // much as its MMAs (256 -> 256 channels on 8^3 voxels: 69 us with one entry, 40 with three, 34 with nine).  Two row
    // tiles of 32 channels: three stages (four: three CTAs an SM, not four; 96 x 100 x 108 voxels, 32 -> 32 channels
    // 190 -> 167 us).
    if (bn == 32 && mt == 1 && ctas() <= 152) return launch_bn<32, 1, 9, 2>(ta, tb, bias, o, g, st);
    if (bn == 32) return mt == 2 ? launch_bn<32, 2, 1, 3>(ta, tb, bias, o, g, st) : launch_bn<32, 1, 1, 4>(ta, tb, bias, o, g, st);
    if (bn == 64) return mt == 2 ? launch_bn<64, 2, 1, 4>(ta, tb, bias, o, g, st) : launch_bn<64, 1, 1, 4>(ta, tb, bias, o, g, st);
    if (bn == 96) return launch_bn<96, 1, 1, 4>(ta, tb, bias, o, g, st);
    return launch_bn<128, 1, 1, 4>(ta, tb, bias, o, g, st);
}

}  // namespace dvm_nn

// One convolution (flip = 0: y = conv(x, w) + b with w[nout][nin][27]; flip = 1: the data gradient,
// nout = the forward input channels, w[nin][nout][27] read with mirrored taps).  Returns a CUDA error,
// cudaErrorInvalidValue for a grid wider than 128 voxels, or cudaErrorNotSupported when the driver
// lacks the tensor-map encoder.
cudaError_t conv_umma(const float* x, const float* w, const float* bias, float* y, int nin, int nout, int d, int h,
                      int w_, int flip, int accumulate, void* scratch, long long scratch_bytes, cudaStream_t st) {
    using namespace dvm_nn;
    if (w_ > kBM || scratch_bytes < conv_umma_scratch_bytes(nin, nout, d, h, w_)) return cudaErrorInvalidValue;
    const int cinp = (nin + kBK - 1) / kBK * kBK, bn = bn_for(nout), coutp = (nout + bn - 1) / bn * bn;
    const uintptr_t base = (reinterpret_cast<uintptr_t>(scratch) + 1023) & ~uintptr_t(1023);
    __nv_bfloat16* xp = reinterpret_cast<__nv_bfloat16*>(base);
    __nv_bfloat16* wb =
        reinterpret_cast<__nv_bfloat16*>(base + align1k((long long)(d + 2) * (h + 2) * (w_ + 2) * cinp * 2));
    pad_bf16_kernel<false><<<pad_grid(cinp, d, h, w_), 256, 0, st>>>(x, xp, nin, cinp, d, h, w_);
    const int sn = flip ? 27 : nin * 27;     // forward: w[n][c][k]; gradient: w[c][n][26 - k]
    const int sc = flip ? nout * 27 : 27;
    weights_bf16_kernel<<<(unsigned)((27LL * coutp * cinp + 255) / 256), 256, 0, st>>>(w, wb, nout, nin, coutp, cinp, sn, sc,
                                                                                      flip);
    const ConvOut o{y, nullptr, 0, 0, 0, 0, accumulate};
    return conv_packed(xp, wb, bias, o, nin, nout, d, h, w_, st);
}

namespace dvm_nn {

// ---------------------------------------------------------------------------- weight gradients
//
//   dw[co][ci][k] (+)= sum_v dy[co][v] x[ci][v + off(k)]
//
// GEMM view: M = (tap, input channel) rows in sub-blocks of 32 (sub-block sb = tap * cinp / 32 +
// channel chunk, four per 128-row tile), N = output channels (BN), K = voxels (chunks of 32 along
// x of one (z, y) row; x padded to a multiple of 32 with zeros).  The A rows of a sub-block are x
// shifted by the tap's offset: three BF16 copies of x (one per x offset dx = -1, 0, 1, already
// shifted along x, with a periodic one-row halo in y and z) make every box start at an x that is a
// multiple of 32; B is a BF16 copy of dy.  Every CTA sums its own range of K chunks (split K) into a
// partial [32 sb rows][coutp] block per sub-block; a second kernel adds the partials of the splits
// in split order (deterministic) into dw.

struct WgradGeom {
    int cin, cout, D, H, W, Wp;      // Wp: x extent padded to a multiple of 32
    int cinp, coutp;
    int nsb;                         // sub-blocks = 27 * cinp / 32
    int nchunks, chunks_per_split;   // K chunks (D * H * Wp / 32) and chunks per CTA
};

template <int BN>
__global__ void __launch_bounds__(kThreads) wgrad_umma_kernel(const __grid_constant__ CUtensorMap tmX,
                                                              const __grid_constant__ CUtensorMap tmG,
                                                              float* __restrict__ part, const WgradGeom g) {
    constexpr int kABytes = kBM * kBK * 2;            // four 32-row sub-blocks of 64-byte rows
    constexpr int kBBytes = BN * kBK * 2;
    constexpr int kStageBytes = kABytes + kBBytes;
    constexpr unsigned kTmemCols = BN < 32 ? 32u : (unsigned)BN;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sbase = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[kStages], empty[kStages], done;
    __shared__ unsigned s_tmem;
    __shared__ int s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mt = blockIdx.x, n0 = blockIdx.y * BN, split = blockIdx.z;
    const int c_begin = split * g.chunks_per_split;
    const int c_end = min(g.nchunks, c_begin + g.chunks_per_split);
    const int nsub = min(4, g.nsb - mt * 4);          // sub-blocks of this tile
    const int ncc = g.cinp / 32;
    const int xchunks = g.Wp / 32;

    if (nsub < 4) {   // rows of missing sub-blocks stay zero (their boxes are never loaded)
        for (int i = threadIdx.x * 16; i < kStages * kStageBytes; i += kThreads * 16)
            *reinterpret_cast<uint4*>(sbase + i) = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_d = s_tmem;
    const int niter = c_end - c_begin;
    const unsigned box_bytes = (unsigned)(nsub * 32 * kBK * 2 + kBBytes);

    if (warp == 0 && lane == 0) {
        for (int i = 0; i < niter; ++i) {
            const int s = i % kStages;
            if (i >= kStages && !mbar_wait(&empty[s], ((i / kStages) - 1) & 1)) {
                s_fail = 1;
                break;
            }
            const int ch = c_begin + i;                 // K chunk: 32 voxels of the (z, y) row
            const int x0 = (ch % xchunks) * 32;
            const int row = ch / xchunks;
            const int y = row % g.H, z = row / g.H;
            unsigned char* st = sbase + (size_t)s * kStageBytes;
            mbar_expect_tx(&full[s], box_bytes);
            for (int j = 0; j < nsub; ++j) {
                const int sb = mt * 4 + j;
                const int tap = sb / ncc, cc = sb - tap * ncc;
                const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
                tma_load_5d(st + j * 32 * kBK * 2, &tmX, x0, y + 1 + dy, z + 1 + dz, cc * 32, dx + 1, &full[s]);
            }
            tma_load_4d(st + kABytes, &tmG, x0, y, z, n0, &full[s]);
        }
    } else if (warp == 1 && lane == 0) {
        const unsigned idesc = idesc_bf16<BN>();
        for (int i = 0; i < niter; ++i) {
            const int s = i % kStages;
            if (!mbar_wait(&full[s], (i / kStages) & 1)) {
                s_fail = 1;
                break;
            }
            tc_fence_after();
            const unsigned char* st = sbase + (size_t)s * kStageBytes;
            const uint64_t ad = smem_desc_sw64(st), bd = smem_desc_sw64(st + kABytes);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
                umma_bf16(tmem_d, ad + 2 * kk, bd + 2 * kk, idesc, (i > 0 || kk > 0) ? 1 : 0);
            umma_commit(&empty[s]);
        }
        umma_commit(&done);
    }
    __syncwarp();
    const bool ok = mbar_wait(&done, 0);
    tc_fence_after();
    if (!ok || s_fail) {
        if (threadIdx.x == 0) atomicCAS(&g_conv_status, 0, -4);
    } else {
        // accumulator row r = (sub-block mt * 4 + r / 32, row r % 32), column j = output channel n0 + j
        const int r = warp * 32 + lane;
        const int sb = mt * 4 + r / 32;
#pragma unroll
        for (int c0 = 0; c0 < BN; c0 += 16) {
            unsigned a[16];
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                         "%13, %14, %15}, [%16];"
                         : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
                           "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]),
                           "=r"(a[14]), "=r"(a[15])
                         : "r"(tmem_d + ((unsigned)(32 * warp) << 16) + (unsigned)c0)
                         : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (sb < g.nsb) {
                float* d = part + (((size_t)split * g.nsb + sb) * 32 + (r & 31)) * g.coutp + n0 + c0;
#pragma unroll
                for (int j = 0; j < 16; ++j) d[j] = niter > 0 ? __uint_as_float(a[j]) : 0.f;
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(kTmemCols) : "memory");
}

// xs[dx + 1][c][pz][py][x] = bf16(x[c][pz - 1][py - 1][x + dx]) (periodic in every axis), zero for
// c >= cin or x >= W; one warp per (dx, c, pz, py) row, lanes along x
__global__ void __launch_bounds__(256) shift_bf16_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ xs,
                                                         int cin, int cinp, int D, int H, int W, int Wp) {
    const long long nrows = 3LL * cinp * (D + 2) * (H + 2);
    const long long row = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= nrows) return;
    const int lane = threadIdx.x & 31;
    const int py = (int)(row % (H + 2));
    const long long r2 = row / (H + 2);
    const int pz = (int)(r2 % (D + 2));
    const long long r3 = r2 / (D + 2);
    const int c = (int)(r3 % cinp);
    const int dx = (int)(r3 / cinp) - 1;
    const int sy = py == 0 ? H - 1 : (py == H + 1 ? 0 : py - 1);
    const int sz = pz == 0 ? D - 1 : (pz == D + 1 ? 0 : pz - 1);
    const float* src = x + (long long)c * D * H * W + ((long long)sz * H + sy) * W;
    __nv_bfloat16* dst = xs + row * Wp;
    for (int xx = lane; xx < Wp; xx += 32) {
        float val = 0.f;
        if (c < cin && xx < W) {
            int sx = xx + dx;
            sx = sx < 0 ? sx + W : (sx >= W ? sx - W : sx);
            val = src[sx];
        }
        dst[xx] = __float2bfloat16_rn(val);
    }
}

// gb[co][z][y][x] = bf16(dy[co][z][y][x]), zero for co >= cout or x >= W
__global__ void grad_bf16_kernel(const float* __restrict__ dy, __nv_bfloat16* __restrict__ gb, int cout, int coutp,
                                 int D, int H, int W, int Wp) {
    const long long total = (long long)coutp * D * H * Wp;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int xx = (int)(i % Wp);
    const long long rest = i / Wp;                      // (co, z, y)
    const long long row = rest % ((long long)D * H);
    const int co = (int)(rest / ((long long)D * H));
    float val = 0.f;
    if (co < cout && xx < W) val = dy[(long long)co * D * H * W + row * W + xx];
    gb[i] = __float2bfloat16_rn(val);
}

// dw[co][ci][k] (+)= sum over splits, in split order, of part[split][sb(k, ci)][ci % 32][co]
__global__ void wgrad_reduce_kernel(const float* __restrict__ part, float* __restrict__ dw, int cin, int cout,
                                    int cinp, int coutp, int nsb, int nsplit, int accumulate) {
    const long long total = (long long)cout * cin * 27;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int k = (int)(i % 27);
    const int ci = (int)((i / 27) % cin);
    const int co = (int)(i / (27LL * cin));
    const int sb = k * (cinp / 32) + ci / 32;
    const size_t off = ((size_t)sb * 32 + (ci & 31)) * coutp + co;
    const size_t stride = (size_t)nsb * 32 * coutp;
    float s = 0.f;
    for (int sp = 0; sp < nsplit; ++sp) s += part[off + (size_t)sp * stride];
    dw[i] = accumulate ? dw[i] + s : s;
}

constexpr int kWgradChunksPerSplit = 64;   // 2048 voxels of K per CTA

template <int BN>
cudaError_t launch_wgrad_bn(const CUtensorMap& tx, const CUtensorMap& tg, float* part, const WgradGeom& g,
                            int nsplit, cudaStream_t st) {
    constexpr int kStageBytes = kBM * kBK * 2 + BN * kBK * 2;
    const int smem = kStages * kStageBytes + 1024;
    auto kern = wgrad_umma_kernel<BN>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((g.nsb + 3) / 4), (unsigned)(g.coutp / BN), (unsigned)nsplit);
    kern<<<grid, kThreads, smem, st>>>(tx, tg, part, g);
    return cudaGetLastError();
}

WgradGeom wgrad_geom(int cin, int cout, int d, int h, int w) {
    WgradGeom g;
    g.cin = cin;
    g.cout = cout;
    g.D = d;
    g.H = h;
    g.W = w;
    g.Wp = (w + 31) / 32 * 32;
    g.cinp = (cin + 31) / 32 * 32;
    const int bn = bn_for(cout);
    g.coutp = (cout + bn - 1) / bn * bn;
    g.nsb = 27 * g.cinp / 32;
    g.nchunks = d * h * (g.Wp / 32);
    g.chunks_per_split = kWgradChunksPerSplit;
    return g;
}

}  // namespace dvm_nn

// Scratch bytes of one weight gradient: the three shifted BF16 copies of x, the BF16 copy of dy and
// the split partials, each 1 KB aligned.
long long wgrad_umma_scratch_bytes(int cin, int cout, int d, int h, int w) {
    using namespace dvm_nn;
    const WgradGeom g = wgrad_geom(cin, cout, d, h, w);
    const long long nsplit = (g.nchunks + g.chunks_per_split - 1) / g.chunks_per_split;
    return align1k(3LL * g.cinp * (d + 2) * (h + 2) * g.Wp * 2) + align1k((long long)g.coutp * d * h * g.Wp * 2) +
           align1k(nsplit * g.nsb * 32 * g.coutp * 4) + 1024;
}

// dw (+)= the weight gradient of y = conv(x, w) for the output gradient dy (see above); the bias
// gradient is not formed here.
cudaError_t wgrad_umma(const float* x, const float* dy, float* dw, int cin, int cout, int d, int h, int w, int accumulate,
                       void* scratch, long long scratch_bytes, cudaStream_t st) {
    using namespace dvm_nn;
    if (scratch_bytes < wgrad_umma_scratch_bytes(cin, cout, d, h, w)) return cudaErrorInvalidValue;
    EncodeFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    const WgradGeom g = wgrad_geom(cin, cout, d, h, w);
    const int bn = bn_for(cout);
    const int nsplit = (g.nchunks + g.chunks_per_split - 1) / g.chunks_per_split;
    const uintptr_t base = (reinterpret_cast<uintptr_t>(scratch) + 1023) & ~uintptr_t(1023);
    const long long xs_bytes = align1k(3LL * g.cinp * (d + 2) * (h + 2) * g.Wp * 2);
    const long long gb_bytes = align1k((long long)g.coutp * d * h * g.Wp * 2);
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(base);
    __nv_bfloat16* gb = reinterpret_cast<__nv_bfloat16*>(base + xs_bytes);
    float* part = reinterpret_cast<float*>(base + xs_bytes + gb_bytes);
    {
        const long long rows = 3LL * g.cinp * (d + 2) * (h + 2);
        shift_bf16_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, st>>>(x, xs, cin, g.cinp, d, h, w, g.Wp);
        const long long m = (long long)g.coutp * d * h * g.Wp;
        grad_bf16_kernel<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(dy, gb, cout, g.coutp, d, h, w, g.Wp);
    }
    CUtensorMap tx, tg;
    {
        const cuuint64_t dims[5] = {(cuuint64_t)g.Wp, (cuuint64_t)(h + 2), (cuuint64_t)(d + 2), (cuuint64_t)g.cinp, 3u};
        const cuuint64_t strides[4] = {(cuuint64_t)g.Wp * 2, (cuuint64_t)g.Wp * 2 * (h + 2),
                                       (cuuint64_t)g.Wp * 2 * (h + 2) * (d + 2),
                                       (cuuint64_t)g.Wp * 2 * (h + 2) * (d + 2) * g.cinp};
        const cuuint32_t box[5] = {32u, 1u, 1u, 32u, 1u};
        const cuuint32_t es[5] = {1u, 1u, 1u, 1u, 1u};
        if (enc(&tx, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, xs, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
            CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    {
        const cuuint64_t dims[4] = {(cuuint64_t)g.Wp, (cuuint64_t)h, (cuuint64_t)d, (cuuint64_t)g.coutp};
        const cuuint64_t strides[3] = {(cuuint64_t)g.Wp * 2, (cuuint64_t)g.Wp * 2 * h, (cuuint64_t)g.Wp * 2 * h * d};
        const cuuint32_t box[4] = {32u, 1u, 1u, (cuuint32_t)bn};
        const cuuint32_t es[4] = {1u, 1u, 1u, 1u};
        if (enc(&tg, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, gb, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
            CUDA_SUCCESS)
            return cudaErrorInvalidValue;
    }
    cudaError_t e;
    if (bn == 32) e = launch_wgrad_bn<32>(tx, tg, part, g, nsplit, st);
    else if (bn == 64) e = launch_wgrad_bn<64>(tx, tg, part, g, nsplit, st);
    else e = launch_wgrad_bn<128>(tx, tg, part, g, nsplit, st);
    if (e != cudaSuccess) return e;
    const long long total = (long long)cout * cin * 27;
    wgrad_reduce_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(part, dw, cin, cout, g.cinp, g.coutp, g.nsb,
                                                                         nsplit, accumulate);
    return cudaGetLastError();
}

namespace dvm_nn {

// ------------------------------------------------------- weight gradients of packed activations and gradients
//
// The same GEMM (M = (tap, input channel) in 32-row sub-blocks, N = output channels, K = voxels) straight from the
// channels-last forms: both operands then have K (voxels) as the strided dimension, which tcgen05.mma reads as
// MN-major tiles.  A sub-block is one TMA box of the packed layer input, 32 channels x a run of voxels shifted by the
// tap, a B block one box of the gradient (no halo, x padded with zeros to a multiple of 16, so that what the A box
// reads beyond a row's end counts for nothing): no shifted or transposed copies of either.
struct WgradPGeom {
    int D, H, W, bx, ry;             // a K chunk: bx voxels along x of ry rows (bx ry a multiple of 16)
    int nxc;                         // chunks along x
    int cinp, coutp;
    int nsb;                         // sub-blocks = 27 * cinp / 32
    int per_split;                   // (z, y) rows of a split
};

// shared-memory descriptor of an MN-major operand in the 64-byte swizzle: atoms of 32 elements x 8 rows of K; lbo is
// the distance between atoms along M or N, 512 bytes that between groups of eight K rows
__device__ __forceinline__ uint64_t smem_desc_mn64(const void* p, unsigned lbo) {
    const uint64_t addr = (smem_u32(p) >> 4) & 0x3FFFu;
    return addr | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}


template <int BN, int NST>
__global__ void __launch_bounds__(kThreads) wgrad_packed_kernel(const __grid_constant__ CUtensorMap tmX,
                                                                const __grid_constant__ CUtensorMap tmG,
                                                                float* __restrict__ part, const WgradPGeom g) {
    constexpr unsigned kTmemCols = BN < 32 ? 32u : (unsigned)BN;
    constexpr int NB = BN / 32;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sbase = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ __align__(8) uint64_t full[NST], empty[NST], done;
    __shared__ unsigned s_tmem;
    __shared__ int s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mt = blockIdx.x, n0 = blockIdx.y * BN, split = blockIdx.z;
    const int r_begin = split * g.per_split, r_end = min(g.D * g.H, r_begin + g.per_split);     // (z, y) rows
    const int nsub = min(4, g.nsb - mt * 4);
    const int ncc = g.cinp / 32;
    const unsigned blk = (unsigned)(g.bx * g.ry) * 64u;   // bytes of one 32-channel block of a chunk
    const unsigned stage = (4 + NB) * blk;
    if (nsub < 4) {   // rows of missing sub-blocks stay zero
        for (unsigned i = threadIdx.x * 16; i < NST * stage; i += kThreads * 16)
            *reinterpret_cast<uint4*>(sbase + i) = make_uint4(0u, 0u, 0u, 0u);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_d = s_tmem;
    // chunks in the order of the voxels: up to ry rows of one plane and of the split, bx voxels of each
    if (warp == 0 && lane == 0) {
        int i = 0, xc = 0;
        for (int r = r_begin; r < r_end; ++i) {
            const int s = i % NST;
            if (i >= NST && !mbar_wait(&empty[s], ((i / NST) - 1) & 1)) {
                s_fail = 1;
                break;
            }
            const int x0 = xc * g.bx;
            const int z = r / g.H, y0 = r - z * g.H;
            if (++xc == g.nxc) {
                xc = 0;
                r += min(g.ry, min(g.H - y0, r_end - r));
            }
            unsigned char* st = sbase + (size_t)s * stage;
            mbar_expect_tx(&full[s], (unsigned)(nsub + NB) * blk);
            for (int j = 0; j < nsub; ++j) {
                const int sb = mt * 4 + j;
                const int tap = sb / ncc, cc = sb - tap * ncc;
                const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
                tma_load_4d(st + j * blk, &tmX, cc * 32, x0 + 1 + dx, y0 + 1 + dy, z + 1 + dz, &full[s]);
            }
#pragma unroll
            for (int j = 0; j < NB; ++j) tma_load_4d(st + (4 + j) * blk, &tmG, n0 + 32 * j, x0, y0, z, &full[s]);
        }
    } else if (warp == 1 && lane == 0) {
        const unsigned idesc = idesc_bf16<BN>() | (1u << 15) | (1u << 16);     // A and B MN-major
        int i = 0, xc = 0;
        for (int r = r_begin; r < r_end; ++i) {
            const int s = i % NST;
            if (!mbar_wait(&full[s], (i / NST) & 1)) {
                s_fail = 1;
                break;
            }
            tc_fence_after();
            const int n = min(g.ry, min(g.H - r % g.H, r_end - r));   // rows of the box that belong to this split
            if (++xc == g.nxc) {
                xc = 0;
                r += n;
            }
            const unsigned char* st = sbase + (size_t)s * stage;
            const uint64_t ad = smem_desc_mn64(st, blk), bd = smem_desc_mn64(st + 4 * blk, blk);
            for (int k = 0; k < n * g.bx / 16; ++k)    // 16 voxels: 1024 bytes on
                umma_bf16(tmem_d, ad + 64 * k, bd + 64 * k, idesc, (i > 0 || k > 0) ? 1 : 0);
            umma_commit(&empty[s]);
        }
        umma_commit(&done);
    }
    __syncwarp();
    const bool ok = mbar_wait(&done, 0);
    tc_fence_after();
    if (!ok || s_fail) {
        if (threadIdx.x == 0) atomicCAS(&g_conv_status, 0, -4);
    } else {
        const int r = warp * 32 + lane;
        const int sb = mt * 4 + r / 32;
#pragma unroll
        for (int c0 = 0; c0 < BN; c0 += 16) {
            unsigned a[16];
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                         "%13, %14, %15}, [%16];"
                         : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
                           "=r"(a[7]), "=r"(a[8]), "=r"(a[9]), "=r"(a[10]), "=r"(a[11]), "=r"(a[12]), "=r"(a[13]),
                           "=r"(a[14]), "=r"(a[15])
                         : "r"(tmem_d + ((unsigned)(32 * warp) << 16) + (unsigned)c0)
                         : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (sb < g.nsb) {
                float4* d = reinterpret_cast<float4*>(part + (((size_t)split * g.nsb + sb) * 32 + (r & 31)) * g.coutp + n0 + c0);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    d[j] = make_float4(__uint_as_float(a[4 * j]), __uint_as_float(a[4 * j + 1]), __uint_as_float(a[4 * j + 2]),
                                       __uint_as_float(a[4 * j + 3]));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(kTmemCols) : "memory");
}

// dw[co][ci][k] += sum over splits, in split order, of part[split][sb(k, ci)][ci % 32][co]; packed channel c of the
// input is channel c (c < c0) or c - c0p + c0 (c >= c0p).  A block takes one input channel,
// 32 output channels and the nine taps of one z offset, a warp per tap: coalesced reads, runs of nine written.
// Bound by the latency of the chain over the splits, so that 32 of them are loaded at a time: 128 splits of 32 -> 32
// channels 13.5 -> 7 us, the 15 launches of a training step on 64^3 voxels 148 -> 99.
__global__ void __launch_bounds__(288) wgrad_packed_reduce_kernel(const float* __restrict__ part, float* __restrict__ dw, int cin,
                                                                  int cout, int c0, int c0p, int cinp, int coutp, int nsb, int nsplit) {
    __shared__ float t[32][9];
    const int cp = blockIdx.x, dz = blockIdx.y, co0 = blockIdx.z * 32;
    const int ci = cp < c0 ? cp : (cp >= c0p ? cp - c0p + c0 : -1);
    if (ci < 0 || ci >= cin) return;
    const int lane = threadIdx.x & 31, k9 = threadIdx.x >> 5;
    const int sb = (dz * 9 + k9) * (cinp / 32) + cp / 32;
    const float* p = part + ((size_t)sb * 32 + (cp & 31)) * coutp + co0 + lane;
    const size_t stride = (size_t)nsb * 32 * coutp;
    float s = 0.f;
    int sp = 0;
    for (; sp + 32 <= nsplit; sp += 32) {
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = p[(size_t)(sp + j) * stride];
#pragma unroll
        for (int j = 0; j < 32; ++j) s += v[j];
    }
#pragma unroll 4
    for (; sp < nsplit; ++sp) s += p[(size_t)sp * stride];
    t[lane][k9] = s;
    __syncthreads();
    const int co = co0 + threadIdx.x / 9, k = threadIdx.x % 9;
    if (co < cout) dw[((long long)co * cin + ci) * 27 + dz * 9 + k] += t[threadIdx.x / 9][k];
}

WgradPGeom wgrad_packed_geom(int cinp, int cout, int d, int h, int w) {
    WgradPGeom g;
    g.D = d;
    g.H = h;
    g.W = w;
    const int wp = (w + 15) / 16 * 16;
    g.nxc = (wp + 63) / 64;
    g.bx = ((wp + g.nxc - 1) / g.nxc + 15) / 16 * 16;
    g.ry = g.bx >= 64 ? 1 : (64 / g.bx < h ? 64 / g.bx : h);
    g.cinp = cinp;
    const int bn = bn_for(cout);
    g.coutp = (cout + bn - 1) / bn * bn;
    g.nsb = 27 * cinp / 32;
    // A split sums the rows that wgrad_umma's splits do (64 pieces of 32 voxels), in the same order: the two give the
    // same bits, except for 64 < w <= 96, where three pieces a row do not divide 64 and a split here has 21 whole rows.
    g.per_split = kWgradChunksPerSplit / ((w + 31) / 32);
    return g;
}

template <int BN, int NST>
cudaError_t launch_wgrad_packed_nst(const CUtensorMap& tx, const CUtensorMap& tg, float* part, const WgradPGeom& g, int nsplit,
                                    int smem, cudaStream_t st) {
    auto kern = wgrad_packed_kernel<BN, NST>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3((unsigned)((g.nsb + 3) / 4), (unsigned)(g.coutp / BN), (unsigned)nsplit), kThreads, smem, st>>>(tx, tg, part, g);
    return cudaGetLastError();
}

// A CTA's MMAs follow one another (one accumulator): it is CTAs per SM that fill the tensor core, so the ring is short.
// Two stages where that saves a wave of CTAs, else three.  64^3 voxels, 32 -> 32 channels (896 CTAs) with 4, 3, 2 stages:
// 83, 58, 64 us; 96 -> 32 (2688 CTAs): 242, 168, 132; 16^3, 384 -> 128 (324 CTAs): 52, 39, 27.
template <int BN>
cudaError_t launch_wgrad_packed(const CUtensorMap& tx, const CUtensorMap& tg, float* part, const WgradPGeom& g, int nsplit,
                                cudaStream_t st) {
    auto smem = [&](int nst) { return nst * (4 + BN / 32) * g.bx * g.ry * 64 + 1024; };
    const long long ctas = (long long)((g.nsb + 3) / 4) * (g.coutp / BN) * nsplit;
    auto waves = [&](int nst) {
        const long long slots = 152LL * (232448 / (smem(nst) + 1024));
        return (ctas + slots - 1) / slots;
    };
    if (waves(2) < waves(3)) return launch_wgrad_packed_nst<BN, 2>(tx, tg, part, g, nsplit, smem(2), st);
    return launch_wgrad_packed_nst<BN, 3>(tx, tg, part, g, nsplit, smem(3), st);
}

long long wgrad_packed_scratch_bytes(int cinp, int cout, int d, int h, int w) {
    const WgradPGeom g = wgrad_packed_geom(cinp, cout, d, h, w);
    return (long long)((d * h + g.per_split - 1) / g.per_split) * g.nsb * 32 * g.coutp * 4 + 1024;
}

// dw[cout][cin][27] += the weight gradient of a convolution with packed input xp (cinp channels: the first c0 of
// cin, the others from c0p on) and packed gradient gw ([d][h][w rounded up to 16][cout rounded up to 32])
cudaError_t wgrad_packed(const __nv_bfloat16* xp, const __nv_bfloat16* gw, float* dw, int cin, int c0, int c0p, int cinp, int cout, int d,
                         int h, int w, float* part, long long part_bytes, cudaStream_t st) {
    EncodeFn enc = encode_fn();
    if (!enc) return cudaErrorNotSupported;
    if (part_bytes < wgrad_packed_scratch_bytes(cinp, cout, d, h, w)) return cudaErrorInvalidValue;
    const WgradPGeom g = wgrad_packed_geom(cinp, cout, d, h, w);
    const int nsplit = (d * h + g.per_split - 1) / g.per_split;
    const int wp = (w + 15) / 16 * 16, coutg = (cout + 31) / 32 * 32;
    part = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(part) + 1023) & ~uintptr_t(1023));
    auto map = [&](CUtensorMap* m, const __nv_bfloat16* base, int c, int nx, int ny, int nz) {
        const cuuint64_t dims[4] = {(cuuint64_t)c, (cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)nz};
        const cuuint64_t strides[3] = {(cuuint64_t)c * 2, (cuuint64_t)c * 2 * nx, (cuuint64_t)c * 2 * nx * ny};
        const cuuint32_t box[4] = {32u, (cuuint32_t)g.bx, (cuuint32_t)g.ry, 1u};
        const cuuint32_t es[4] = {1u, 1u, 1u, 1u};
        return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(base), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    };
    CUtensorMap tx, tg;
    if (!map(&tx, xp, cinp, w + 2, h + 2, d + 2) || !map(&tg, gw, coutg, wp, h, d)) return cudaErrorInvalidValue;
    const int bn = bn_for(cout);
    cudaError_t e;
    if (bn == 32) e = launch_wgrad_packed<32>(tx, tg, part, g, nsplit, st);
    else if (bn == 64) e = launch_wgrad_packed<64>(tx, tg, part, g, nsplit, st);
    else e = launch_wgrad_packed<128>(tx, tg, part, g, nsplit, st);
    if (e != cudaSuccess) return e;
    wgrad_packed_reduce_kernel<<<dim3((unsigned)cinp, 3u, (unsigned)((cout + 31) / 32)), 288, 0, st>>>(part, dw, cin, cout, c0, c0p, cinp,
                                                                                                    g.coutp, g.nsb, nsplit);
    return cudaGetLastError();
}

cudaError_t pack_input(const float* x, __nv_bfloat16* xp, int c, int cp, int d, int h, int w, int pool, cudaStream_t st) {
    const dim3 grid = pad_grid(cp, d, h, w);
    if (pool) pad_bf16_kernel<true><<<grid, 256, 0, st>>>(x, xp, c, cp, d, h, w);
    else pad_bf16_kernel<false><<<grid, 256, 0, st>>>(x, xp, c, cp, d, h, w);
    return cudaGetLastError();
}

}  // namespace dvm_nn

// the device status word of the convolutions (nonzero after a bounded wait expired); cleared on read
int conv_umma_status(cudaStream_t st) {
    int v = 0;
    if (cudaStreamSynchronize(st) != cudaSuccess) return -3;
    if (cudaMemcpyFromSymbol(&v, dvm_nn::g_conv_status, sizeof(int)) != cudaSuccess) return -3;
    if (v) {
        const int zero = 0;
        cudaMemcpyToSymbol(dvm_nn::g_conv_status, &zero, sizeof(int));
    }
    return v;
}
