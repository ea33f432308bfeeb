// wsnet.cu -- the learned warm start: a 3D U-Net that maps the extruded
// skyrmion-tube ansatz (plus q0, Lz, W0) to the relaxed director field, with
// hand-written BF16 training and inference kernels (FP32 accumulation).
//
// Network (4 levels, widths 16/16/32/64, 394 419 parameters): two 3x3x3
// convolutions + ReLU per level, 2x2x2 mean pooling down, nearest x2 upsampling
// and channel concatenation up, a 1x1x1 head 16 -> 3 whose output corrects the
// ansatz, n = normalise(n_ansatz + delta).  Convolutions are cross-correlations,
// periodic in x and y and zero-padded in z.
//
// Layouts: activations are channels-last BF16 [batch][z][y][x][c]; gradients of
// pre-activations are channels-last BF16, of pooled and upsampled tensors FP32.  Parameters are one flat FP32 vector, layer
// by layer W[tap][cout][cin] (tap = 9 kz + 3 ky + kx) then bias[cout]; the head
// is W[3][16] then bias[3].
//
// Convolutions run on the tensor cores as implicit GEMMs (BF16 inputs, FP32
// accumulators):
//   forward       M = voxels (128 per step), N = cout, K = 27 taps x cin, on the
//                 5th-generation tensor cores (tcgen05.mma, accumulator in TMEM)
//   data grad     M = voxels, N = cin, K = 27 taps x cout (transposed weights),
//                 the same kernel
//   weight grad   M = cout, N = cin, K = voxels (all taps from one shared-memory
//                 halo tile, FP32 atomics across blocks), mma.sync.m16n8k16
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include "nh_internal.cuh"

namespace {

using bf16 = __nv_bfloat16;

// ------------------------------------------------------------------ architecture

struct LayerDesc {
    int cin, cout;
};
constexpr int kLayers = 14;
constexpr LayerDesc kConv[kLayers] = {{16, 16}, {16, 16}, {16, 16}, {16, 16}, {16, 32}, {32, 32}, {32, 64},
                                      {64, 64}, {96, 32}, {32, 32}, {48, 16}, {16, 16}, {32, 16}, {16, 16}};
enum { ENC1A, ENC1B, ENC2A, ENC2B, ENC3A, ENC3B, BOTA, BOTB, DEC3A, DEC3B, DEC2A, DEC2B, DEC1A, DEC1B };
constexpr int kHeadIn = 16, kHeadOut = 3, kInCh = 16;

int64_t layer_offset(int l)
{
    int64_t off = 0;
    for (int k = 0; k < l; ++k) off += 27LL * kConv[k].cin * kConv[k].cout + kConv[k].cout;
    return off;
}
int64_t head_offset() { return layer_offset(kLayers); }
int64_t total_params() { return head_offset() + kHeadIn * kHeadOut + kHeadOut; }

// ------------------------------------------------------------------ device helpers

__device__ __forceinline__ void mma16816(float c[4], const uint32_t a[4], const uint32_t b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}

struct Dims {
    int nx, ny, nz, nvox, batch;
};

// ------------------------------------------------------------------ convolution on tcgen05: forward and data gradient
//
// One CTA (four warps) computes 8 x 16 output voxels of a z plane x NB output
// channels per step and walks up a chunk of planes; each plane is the implicit
// GEMM D[128][NB] = sum over the 27 taps of A_t[128][K] W_t^T.  Planes of the
// input with a one-voxel halo in x and y (10 x 18 voxels) sit in a ring of four
// shared-memory slots in the tensor core's no-swizzle K-major layout, 16-byte
// channel groups of consecutive voxels next to each other: the eight voxels of
// an x run are a core matrix, so the A operand of *every* tap is the same plane
// read from a shifted start address (LBO = one channel-group plane, SBO = one
// row of ten voxels), and a plane is copied once instead of once per tap.
// (Copying each tap's rows took 339 us for a 16 -> 16 layer of 8 x 64 x 64 x 32
// voxels, bound by the copies and a barrier per three taps.)  The weights of all
// taps stay in shared memory for the CTA's life.  One thread issues a plane's 27
// K/16 MMAs (kind::f16, BF16 x BF16 -> FP32, M = 128, N = NB, K = 16) into one of
// two TMEM accumulators and commits them to its mbarrier; the copies of the plane
// after next and the epilogue of the plane before run meanwhile.  Every mbarrier
// wait is bounded: on expiry the kernel raises a.status, skips the epilogue,
// waits for its copies and frees its TMEM.
//
// Forward: input = the layer's sources, D + bias, ReLU, BF16 rows.  Data gradient
// (Flip): input = the pre-activation gradient, taps mirrored, transposed weights.
// Where the source is another convolution's output (mask), the epilogue makes that
// layer's pre-activation gradient at once -- masked by its ReLU, BF16 -- and its
// bias gradient, which spares the FP32 gradient's way through memory (a separate
// pass took 30 us a layer of 8 x 64 x 64 x 32 voxels); else FP32 rows go to dst1
// (channels below n1) and dst2.

struct ConvTc {
    const bf16* src1;
    int c1;
    const bf16* src2;  // concatenated after src1 (c2 = 0: none)
    int c2;
    int up1;           // src1 is held at half the resolution and read nearest (upsampling)
    const bf16* w;     // [27][n][c1 + c2]
    int n;             // output channels; blockIdx.y takes NB of them
    Dims d;
    int zc;            // planes per chunk
    const float* bias; // forward: [n]
    bf16* out;         // forward: [vox][n]
    const bf16* mask;  // data gradient: the source's activations [vox][n], or null
    bf16* gp;          // with mask: pre-activation gradient of the source's layer [vox][n]
    float* gb;         // with mask: its bias gradient [n] (accumulated)
    float* dst1;       // data gradient without mask: [vox][n1]
    int n1;
    float* dst2;       // data gradient without mask: [vox][n - n1]
    int* status;       // set to 1 when a bounded wait expires
};

constexpr int kTcM = 128;
constexpr int kTcThreads = 128;
constexpr int kTcX = 8, kTcY = 16;                                // output voxels of a plane step
constexpr int kTcHX = kTcX + 2, kTcHY = kTcY + 2, kTcHalo = kTcHX * kTcHY;
constexpr int kTcRing = 4;
inline size_t tc_smem(int K, int NB) { return (size_t)K * 2 * (kTcRing * kTcHalo + 27 * NB) + 64 + NB * sizeof(float); }
constexpr size_t kTcMaxSmem = 227 * 1024;

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor of the tensor core: no swizzle, start
// address, LBO and SBO in 16-byte units, descriptor version 1 (bits 46-48).
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
           ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: FP32 D (bits 4-5 = 1), BF16 A (7-9 = 1)
// and B (10-12 = 1), both K-major, N / 8 in bits 17-22, M / 16 in bits 24-28.
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity)
{
    for (int it = 0; it < (1 << 22); ++it) {
        uint32_t done;
        asm volatile(
            "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float v[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// g = 0 where the activation y (8 BF16 values) is not positive; and 8 FP32 values as BF16.
__device__ __forceinline__ void relu_mask(float g[8], const uint4 y)
{
    const __nv_bfloat162* yh = reinterpret_cast<const __nv_bfloat162*>(&y);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (!(__low2float(yh[k]) > 0.f)) g[2 * k] = 0.f;
        if (!(__high2float(yh[k]) > 0.f)) g[2 * k + 1] = 0.f;
    }
}
__device__ __forceinline__ uint4 pack8(const float g[8])
{
    return make_uint4(pack_bf16(g[0], g[1]), pack_bf16(g[2], g[3]), pack_bf16(g[4], g[5]), pack_bf16(g[6], g[7]));
}
__device__ __forceinline__ void unpack8(const uint4 y, float v[8])
{
    const __nv_bfloat162* yh = reinterpret_cast<const __nv_bfloat162*>(&y);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[2 * k] = __low2float(yh[k]);
        v[2 * k + 1] = __high2float(yh[k]);
    }
}

template <int NB, bool Flip>
__global__ void __launch_bounds__(kTcThreads) conv_tc_kernel(const ConvTc a)
{
    extern __shared__ __align__(128) unsigned char tc_smem_raw[];
    nh::step_kernel_enter();
    const int K = a.c1 + a.c2, kb = K / 8;  // 16-byte channel groups
    constexpr uint32_t kGroup = kTcHalo * 16;              // one channel group of a plane
    const uint32_t plane_bytes = (uint32_t)kb * kGroup;
    const uint32_t tap_bytes = (uint32_t)NB * K * 2;
    const uint32_t ring = smem_u32(tc_smem_raw), wbase = ring + kTcRing * plane_bytes;
    uint64_t* bars = reinterpret_cast<uint64_t*>(tc_smem_raw + kTcRing * plane_bytes + 27 * tap_bytes);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2);
    float* bshared = reinterpret_cast<float*>(bars + 8);  // bias gradient of the CTA's voxels (with mask)
    if (Flip && threadIdx.x < NB) bshared[threadIdx.x] = 0.f;
    constexpr uint32_t kCols = 2 * NB;  // two accumulators: 32 or 64 columns
    static_assert(NB == 16 || NB == 32, "TMEM columns are allocated in powers of two, at least 32");
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const Dims d = a.d;
    const int tx = (d.nx + kTcX - 1) / kTcX, ty = (d.ny + kTcY - 1) / kTcY, tz = (d.nz + a.zc - 1) / a.zc;
    int blk = blockIdx.x;
    const int x0 = (blk % tx) * kTcX;
    blk /= tx;
    const int y0 = (blk % ty) * kTcY;
    blk /= ty;
    const int z0 = (blk % tz) * a.zc, z1 = min(z0 + a.zc, d.nz), batch = blk / tz;
    const int n0 = blockIdx.y * NB;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "r"(kCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&bars[0])) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&bars[1])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }

    // a thread copies one channel group of every vstep-th voxel of a plane
    const int cq = tid % kb, vfirst = tid / kb, vstep = kTcThreads / kb;
    const bool loader = vfirst < vstep;
    const bool from1 = cq * 8 < a.c1;
    const bool up = from1 && a.up1;
    const bf16* lsrc = from1 ? a.src1 + cq * 8 : a.src2 + (cq * 8 - a.c1);
    const int lc = from1 ? a.c1 : a.c2;
    auto load_plane = [&](int z) {  // zero beyond the volume in z
        if (loader) {
            const bool zin = z >= 0 && z < d.nz;
            const uint32_t dst = ring + (uint32_t)(z & (kTcRing - 1)) * plane_bytes + (uint32_t)cq * kGroup;
            for (int v = vfirst; v < kTcHalo; v += vstep) {
                const int hy = v / kTcHX, hx = v - hy * kTcHX;
                int x = x0 - 1 + hx, y = y0 - 1 + hy;
                x = x < 0 ? x + d.nx : (x >= d.nx ? x - d.nx : x);
                y = y < 0 ? y + d.ny : (y >= d.ny ? y - d.ny : y);
                const bool ok = zin && x < d.nx && y < d.ny;  // beyond a ragged tile's halo: unused, zero
                const int s = up ? batch * (d.nvox >> 3) + (x >> 1) + (d.nx >> 1) * ((y >> 1) + (d.ny >> 1) * (z >> 1))
                                 : batch * d.nvox + x + d.nx * (y + d.ny * z);
                cp_async16(dst + (uint32_t)v * 16u, ok ? lsrc + (size_t)s * lc : lsrc, ok);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    for (int i = tid; i < 27 * NB * kb; i += kTcThreads) {
        const int q = i % kb, r = i / kb, n = r % NB, t = r / NB;
        cp_async16(wbase + (uint32_t)t * tap_bytes + (uint32_t)(n >> 3) * (uint32_t)(kb * 128) + (uint32_t)q * 128u +
                       (uint32_t)(n & 7) * 16u,
                   a.w + ((size_t)t * a.n + n0 + n) * K + q * 8, true);
    }
    for (int z = z0 - 1; z <= z0 + 1; ++z) load_plane(z);

    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tmem_slot;

    constexpr uint32_t idesc = umma_idesc_bf16(kTcM, NB);
    // row r of the accumulator is voxel (x0 + r % 8, y0 + r / 8) of the plane
    const int row = warp * 32 + lane;
    const int vx = x0 + (row & 7), vy = y0 + (row >> 3);
    const bool inside = vx < d.nx && vy < d.ny;
    float bsum[Flip ? NB : 1];  // bias gradient of this thread's voxels (with mask)
#pragma unroll
    for (int i = 0; i < (Flip ? NB : 1); ++i) bsum[i] = 0.f;
    auto epilogue = [&](int z) {
        const uint32_t acc0 = tmem + (uint32_t)(((z - z0) & 1) * NB) + ((uint32_t)(warp * 32) << 16);
        const size_t v = (size_t)batch * d.nvox + vx + (size_t)d.nx * (vy + (size_t)d.ny * z);
#pragma unroll
        for (int c0 = 0; c0 < NB; c0 += 16) {
            float acc[16];
            tmem_ld16(acc0 + (uint32_t)c0, acc);
            if (!inside) continue;
            if constexpr (!Flip) {
                uint32_t packed[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float b0 = __ldg(a.bias + n0 + c0 + 2 * i), b1 = __ldg(a.bias + n0 + c0 + 2 * i + 1);
                    packed[i] = pack_bf16(fmaxf(acc[2 * i] + b0, 0.f), fmaxf(acc[2 * i + 1] + b1, 0.f));
                }
                uint4* dst = reinterpret_cast<uint4*>(a.out + v * a.n + n0 + c0);
                dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
            } else if (a.mask != nullptr) {
                const uint4* m = reinterpret_cast<const uint4*>(a.mask + v * a.n + n0 + c0);
                uint4* dst = reinterpret_cast<uint4*>(a.gp + v * a.n + n0 + c0);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float* g = acc + 8 * h;
                    relu_mask(g, __ldg(m + h));
#pragma unroll
                    for (int i = 0; i < 8; ++i) bsum[c0 + 8 * h + i] += g[i];
                    dst[h] = pack8(g);
                }
            } else {
                const bool first = n0 + c0 < a.n1;
                float4* dst = reinterpret_cast<float4*>(first ? a.dst1 + v * a.n1 + n0 + c0
                                                              : a.dst2 + v * (a.n - a.n1) + (n0 + c0 - a.n1));
#pragma unroll
                for (int i = 0; i < 4; ++i) dst[i] = make_float4(acc[4 * i], acc[4 * i + 1], acc[4 * i + 2], acc[4 * i + 3]);
            }
        }
    };

    bool ok = true;
    for (int z = z0; z < z1; ++z) {
        const int k = z - z0;
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // the copies, to the tensor core's view
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");  // the epilogue's TMEM reads
        ok = __syncthreads_and(ok) != 0;
        if (!ok) break;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint64_t ad0 = umma_desc(0, kGroup, kTcHX * 16), bd0 = umma_desc(0, 128u, (uint32_t)kb * 128u);
            const uint32_t acc0 = tmem + (uint32_t)((k & 1) * NB);
            uint32_t acc = 0;
            for (int dz = 0; dz < 3; ++dz) {
                const int zp = Flip ? z + 1 - dz : z - 1 + dz;
                const uint32_t pa = (ring + (uint32_t)(zp & (kTcRing - 1)) * plane_bytes) >> 4;
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    const int off = Flip ? (2 - q / 3) * kTcHX + (2 - q % 3) : (q / 3) * kTcHX + q % 3;
                    const uint32_t wa = (wbase + (uint32_t)(dz * 9 + q) * tap_bytes) >> 4;
                    for (int j = 0; j < kb / 2; ++j) {
                        const uint64_t ad = ad0 | (uint64_t)(pa + off + (uint32_t)j * (2 * kGroup >> 4));
                        const uint64_t bd = bd0 | (uint64_t)(wa + (uint32_t)j * 16u);
                        asm volatile(
                            "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                            "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(acc0),
                            "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                            : "memory");
                        acc = 1;
                    }
                }
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                             smem_u32(&bars[k & 1]))
                         : "memory");
        }
        __syncwarp();
        // the MMAs of plane z - 1 are done: their lowest input plane's slot takes plane z + 2
        if (k > 0) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[(k - 1) & 1]), ((k - 1) >> 1) & 1)) != 0;
        if (ok && z + 1 < z1) load_plane(z + 2);
        if (ok && k > 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            epilogue(z - 1);
        }
    }
    if (ok) {
        const int k = z1 - 1 - z0;
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[k & 1]), (k >> 1) & 1)) != 0;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (ok) epilogue(z1 - 1);
    }
    if (!ok && lane == 0) atomicExch(a.status, 1);
    if constexpr (Flip) {
        if (a.mask != nullptr) {
            // halve the channels a lane holds as the lanes that add to it double: after the steps lane l has the
            // warp's sum of channel l mod NB (of NB 16, lanes l and l + 16 each half of it)
#pragma unroll
            for (int w = NB / 2; w > 0; w >>= 1) {
                const bool high = (lane & w) != 0;
#pragma unroll
                for (int i = 0; i < w; ++i) {
                    const float send = high ? bsum[i] : bsum[i + w], keep = high ? bsum[i + w] : bsum[i];
                    bsum[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
                }
            }
            atomicAdd(&bshared[lane & (NB - 1)], bsum[0]);
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if constexpr (Flip)
        if (a.mask != nullptr && tid < NB) atomicAdd(a.gb + n0 + tid, bshared[tid]);
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols) : "memory");
    }
}

// Launch over every plane tile of the level.  NB = 32 where two such weight
// sets fit an SM (K <= 32), else 16: more CTAs on the coarse levels, whose wide
// layers have few voxels.  Planes per chunk: the CTAs run in waves of as many as
// an SM holds (shared memory, TMEM columns), and a chunk loads two planes beyond
// its own; the split with the least waves x (planes + 2).  (8 planes of
// 8 x 64 x 64 x 32 voxels made 1024 CTAs of which 912 are resident.)
template <bool Flip>
cudaError_t launch_conv_tc(ConvTc a, cudaStream_t st)
{
    static bool attr_set = false;  // the opt-in to more than 48 KB of shared memory, once per process
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(conv_tc_kernel<16, Flip>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kTcMaxSmem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(conv_tc_kernel<32, Flip>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcMaxSmem);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    const int K = a.c1 + a.c2;
    const int NB = a.n % 32 == 0 && K <= 32 ? 32 : 16;
    if (K % 16 || a.n % 16 || a.c1 % 8 || tc_smem(K, NB) > kTcMaxSmem) return cudaErrorInvalidValue;
    const int cols = ((a.d.nx + kTcX - 1) / kTcX) * ((a.d.ny + kTcY - 1) / kTcY) * a.d.batch;
    const int resident = 152 * std::min((int)(kTcMaxSmem / (tc_smem(K, NB) + 1024)), 512 / (2 * NB));
    int64_t best = -1;
    for (int n = 1; n <= a.d.nz; ++n) {
        const int zc = (a.d.nz + n - 1) / n;
        const int64_t blocks = (int64_t)cols * ((a.d.nz + zc - 1) / zc) * (a.n / NB);
        const int64_t cost = (blocks + resident - 1) / resident * (zc + 2);
        if (best < 0 || cost < best) {
            best = cost;
            a.zc = zc;
        }
    }
    const dim3 grid(cols * ((a.d.nz + a.zc - 1) / a.zc), a.n / NB);
    if (NB == 32)
        nh::launch_step_kernel(conv_tc_kernel<32, Flip>, grid, kTcThreads, tc_smem(K, NB), st, a);
    else
        nh::launch_step_kernel(conv_tc_kernel<16, Flip>, grid, kTcThreads, tc_smem(K, NB), st, a);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ convolution: weight gradient

struct ConvBwdW {
    const bf16* gp;     // [vox][cout] gradient of the pre-activation (ReLU mask applied), BF16
    const bf16* src1;   // [vox][c1]
    int c1;
    const bf16* src2;   // [vox][c2]
    int c2;
    int cout;
    int up1;            // src1 is held at half the resolution and read nearest (upsampling)
    float* gw;          // [27][cout][cin] (accumulated)
    Dims d;
    int tiles;          // voxel tiles of the level
};

// A block owns 16 output x 16 input channels (blockIdx.y) of all 27 taps and
// walks 8 x 8 x 4 voxel tiles (blockIdx.x, grid stride).  A tile's gradient rows
// and its activation rows with a one-voxel halo are copied into shared memory
// once (cp.async, the next tile in flight) and serve all 27 taps: reading the
// activations again for every tap made this 2291 us for a 16 -> 16 layer of
// 8 x 64 x 64 x 32 voxels.  Warp w takes the nine taps of dz = w % 3 - 1 and half
// w / 3 of the tile's voxels: per 16 voxels (two x runs of eight) one transposed
// ldmatrix of the gradient is multiplied with nine of the shifted activations;
// the 9 x 16 x 16 sums stay in registers (72 a thread) until the block's last
// tile.  Rows are 32 bytes; their two 16-byte halves are swapped on every other
// group of four voxels of a run, so that the eight rows of an ldmatrix hit
// distinct banks at any x shift.
constexpr int kWTx = 8, kWTy = 8, kWTz = 4, kWVox = kWTx * kWTy * kWTz;
constexpr int kWHx = kWTx + 2, kWHy = kWTy + 2, kWHz = kWTz + 2, kWHalo = kWHx * kWHy * kWHz;
constexpr int kWThreads = 192;
constexpr int kWStage = (kWVox + kWHalo) * 32;  // bytes: gradient rows, then activation rows
constexpr int kWSmem = 2 * kWStage;
constexpr int kWBlocksPerSM = 3;

__device__ __forceinline__ void ldm_x4_trans(uint32_t addr, uint32_t r[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

__global__ void __launch_bounds__(kWThreads, kWBlocksPerSM) conv_bwd_w_kernel(const ConvBwdW a)
{
    extern __shared__ __align__(128) unsigned char w_smem[];
    nh::step_kernel_enter();
    const uint32_t smem0 = smem_u32(w_smem);
    const int cin = a.c1 + a.c2;
    const int nci = cin / 16;
    const int co0 = ((int)blockIdx.y / nci) * 16, ci0 = ((int)blockIdx.y % nci) * 16;
    const bool first = ci0 < a.c1;
    const bf16* xs = first ? a.src1 + ci0 : a.src2 + (ci0 - a.c1);
    const int xc = first ? a.c1 : a.c2;
    const bool up = first && a.up1;
    const Dims d = a.d;
    const int tx = (d.nx + kWTx - 1) / kWTx, ty = (d.ny + kWTy - 1) / kWTy, tz = (d.nz + kWTz - 1) / kWTz;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // copies of one tile into stage s; rows outside the volume (and the
    // gradient of voxels beyond a ragged tile's end) are zero
    auto load_tile = [&](int t, int s) {
        const int x0 = (t % tx) * kWTx;
        int r = t / tx;
        const int y0 = (r % ty) * kWTy;
        r /= ty;
        const int z0 = (r % tz) * kWTz, batch = r / tz, vb = batch * d.nvox;
        const uint32_t G = smem0 + (uint32_t)s * kWStage, X = G + kWVox * 32;
        for (int i = tid; i < kWVox * 2; i += kWThreads) {
            const int c = i & 1, v = i >> 1;
            const int x = x0 + v % kWTx, y = y0 + (v / kWTx) % kWTy, z = z0 + v / (kWTx * kWTy);
            const bool ok = x < d.nx && y < d.ny && z < d.nz;
            const bf16* src = ok ? a.gp + (size_t)(vb + x + d.nx * (y + d.ny * z)) * a.cout + co0 + 8 * c : a.gp;
            cp_async16(G + v * 32 + ((c ^ ((v >> 2) & 1)) << 4), src, ok);
        }
        for (int i = tid; i < kWHalo * 2; i += kWThreads) {
            const int c = i & 1, v = i >> 1;
            const int hx = v % kWHx, hy = (v / kWHx) % kWHy, hz = v / (kWHx * kWHy);
            int x = x0 - 1 + hx, y = y0 - 1 + hy;
            const int z = z0 - 1 + hz;
            x = x < 0 ? x + d.nx : (x >= d.nx ? x - d.nx : x);
            y = y < 0 ? y + d.ny : (y >= d.ny ? y - d.ny : y);
            const bool ok = x < d.nx && y < d.ny && z >= 0 && z < d.nz;
            const int sv = up ? batch * (d.nvox >> 3) + (x >> 1) + (d.nx >> 1) * ((y >> 1) + (d.ny >> 1) * (z >> 1))
                              : vb + x + d.nx * (y + d.ny * z);
            const bf16* src = ok ? xs + (size_t)sv * xc + 8 * c : xs;
            cp_async16(X + v * 32 + ((c ^ ((hx >> 2) & 1)) << 4), src, ok);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    const int dz = warp % 3, half = warp / 3;
    const int mi = lane >> 3, r8 = lane & 7;
    // A[co][v] = G[v][co]: matrices (v 0-7, co 0-7), (v 0-7, co 8-15), (v 8-15, co 0-7), (v 8-15, co 8-15)
    const uint32_t laneA = (uint32_t)(((mi >> 1) * 8 + r8) * 32 + (((mi & 1) ^ ((r8 >> 2) & 1)) << 4));
    // B[v][ci] = X[v + tap][ci]: (v 0-7, ci 0-7), (v 8-15, ci 0-7), (v 0-7, ci 8-15), (v 8-15, ci 8-15)
    uint32_t laneB[3];
#pragma unroll
    for (int dx = 0; dx < 3; ++dx)
        laneB[dx] = (uint32_t)((mi & 1) * (kWHx * 32) + (r8 + dx) * 32 + (((mi >> 1) ^ (((r8 + dx) >> 2) & 1)) << 4));
    float acc[9][2][4];
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
        for (int h = 0; h < 2; ++h) acc[q][h][0] = acc[q][h][1] = acc[q][h][2] = acc[q][h][3] = 0.f;

    int t = blockIdx.x;
    if (t < a.tiles) load_tile(t, 0);
    for (int s = 0; t < a.tiles; t += gridDim.x, s ^= 1) {
        if (t + (int)gridDim.x < a.tiles) {
            load_tile(t + gridDim.x, s ^ 1);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        const uint32_t G = smem0 + (uint32_t)s * kWStage, X = G + kWVox * 32;
#pragma unroll 2
        for (int k = 0; k < 8; ++k) {  // 16 voxels: rows y = 2 j, 2 j + 1 of layer z
            const int z = 2 * half + (k >> 2), j = k & 3;
            uint32_t fa[4];
            ldm_x4_trans(G + laneA + (uint32_t)((z * kWTy + 2 * j) * kWTx * 32), fa);
            const uint32_t xb = X + (uint32_t)(((z + dz) * kWHy + 2 * j) * (kWHx * 32));
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                uint32_t fb[4];
                ldm_x4_trans(xb + laneB[q % 3] + (uint32_t)(q / 3) * (kWHx * 32), fb);
                mma16816(acc[q][0], fa, fb);
                mma16816(acc[q][1], fa, fb + 2);
            }
        }
        __syncthreads();
    }

    // the two voxel halves meet in shared memory, then one add per value and block
    float* red = reinterpret_cast<float*>(w_smem) + (size_t)dz * 72 * 32 + lane;
    if (half == 1) {
#pragma unroll
        for (int q = 0; q < 9; ++q)
#pragma unroll
            for (int i = 0; i < 8; ++i) red[(q * 8 + i) * 32] = acc[q][i >> 2][i & 3];
    }
    __syncthreads();
    if (half == 1) return;
    const int g = lane >> 2, c2 = 2 * (lane & 3);
    const bool vec = (reinterpret_cast<uintptr_t>(a.gw) & 7) == 0;
#pragma unroll
    for (int q = 0; q < 9; ++q)
#pragma unroll
        for (int i = 0; i < 8; i += 2) {  // i: n half (4), row half (2)
            const float v0 = acc[q][i >> 2][i & 3] + red[(q * 8 + i) * 32];
            const float v1 = acc[q][i >> 2][(i & 3) + 1] + red[(q * 8 + i + 1) * 32];
            float* dst = a.gw + (size_t)((dz * 9 + q) * a.cout + co0 + g + ((i & 2) ? 8 : 0)) * cin + ci0 + (i >> 2) * 8 + c2;
            if (vec) {
                atomicAdd(reinterpret_cast<float2*>(dst), make_float2(v0, v1));
            } else {
                atomicAdd(dst, v0);
                atomicAdd(dst + 1, v1);
            }
        }
}

// ------------------------------------------------------------------ pooling / upsampling
//
// All of these move 8-channel groups (16 bytes of BF16, 32 of FP32): a thread per
// group, so that a warp reads and writes whole lines.

// dst (coarse) = mean of the 2x2x2 children in src (fine), channels-last, C channels
__global__ void pool_fwd_kernel(const bf16* __restrict__ src, bf16* __restrict__ dst, Dims fine, int C)
{
    nh::step_kernel_enter();
    const int cx = fine.nx / 2, cy = fine.ny / 2, cz = fine.nz / 2, cvox = cx * cy * cz, cg = C / 8;
    const int total = cvox * fine.batch * cg;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int v = i / cg, q = i - v * cg;
        const int b = v / cvox, r = v - b * cvox;
        const int x = r % cx, y = (r / cx) % cy, z = r / (cx * cy);
        float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int fx = 2 * x + (k & 1), fy = 2 * y + ((k >> 1) & 1), fz = 2 * z + (k >> 2);
            float c[8];
            unpack8(__ldg(reinterpret_cast<const uint4*>(src) + (size_t)(b * fine.nvox + fx + fine.nx * (fy + fine.ny * fz)) * cg + q), c);
#pragma unroll
            for (int j = 0; j < 8; ++j) s[j] += c[j];
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) s[j] *= 0.125f;
        reinterpret_cast<uint4*>(dst)[i] = pack8(s);
    }
}

// A pre-activation gradient from the gradient g of an activation group: masked
// by the ReLU of act, BF16 into gp, and summed into the thread's bias sums.
__device__ __forceinline__ void prep_group(float g[8], const bf16* act, bf16* gp, int64_t i, float bias[8])
{
    relu_mask(g, __ldg(reinterpret_cast<const uint4*>(act) + i));
    reinterpret_cast<uint4*>(gp)[i] = pack8(g);
#pragma unroll
    for (int k = 0; k < 8; ++k) bias[k] += g[k];
}
// The block's bias sums into gb: a thread's group q is fixed (the grid stride is
// a multiple of C / 8, and so are a warp's 32 threads), so the lanes of a group
// add by shuffles, the warps in shared memory, and the block with one atomic per
// channel.
__device__ __forceinline__ void bias_out(const float bias[8], int q, int C, float* gb)
{
    __shared__ float bsum[64];
    for (int k = threadIdx.x; k < C; k += blockDim.x) bsum[k] = 0.f;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        float v = bias[k];
        for (int o = 16; o >= C / 8; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) < C / 8) atomicAdd(&bsum[q * 8 + k], v);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < C; k += blockDim.x) atomicAdd(&gb[k], bsum[k]);
}

__device__ __forceinline__ void ld8(const float* p, int64_t i, float v[8])
{
    const float4 a = __ldg(reinterpret_cast<const float4*>(p) + 2 * i), b = __ldg(reinterpret_cast<const float4*>(p) + 2 * i + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// Pre-activation gradient of the layer that a pooling and a skip connection read:
// the skip's gradient plus an eighth of the pooled one's.
__global__ void __launch_bounds__(256) pool_bwd_kernel(const float* __restrict__ gpool, const float* __restrict__ gskip,
                                                       const bf16* __restrict__ act, bf16* __restrict__ gp, float* gb,
                                                       Dims fine, int C)
{
    nh::step_kernel_enter();
    const int cx = fine.nx / 2, cy = fine.ny / 2, cg = C / 8;
    const int total = fine.nvox * fine.batch * cg, first = blockIdx.x * blockDim.x + threadIdx.x;
    float bias[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int i = first; i < total; i += gridDim.x * blockDim.x) {
        const int v = i / cg, q = i - v * cg;
        const int b = v / fine.nvox, r = v - b * fine.nvox;
        const int x = r % fine.nx, y = (r / fine.nx) % fine.ny, z = r / (fine.nx * fine.ny);
        const int64_t cv = (int64_t)b * (fine.nvox / 8) + x / 2 + cx * (y / 2 + cy * (z / 2));
        float g[8], c[8];
        ld8(gskip, i, g);
        ld8(gpool, cv * cg + q, c);
#pragma unroll
        for (int k = 0; k < 8; ++k) g[k] += 0.125f * c[k];
        prep_group(g, act, gp, i, bias);
    }
    bias_out(bias, first % cg, C, gb);
}

// Pre-activation gradient of the layer that an upsampling reads: the sum over the 8 children.
__global__ void __launch_bounds__(256) up_bwd_kernel(const float* __restrict__ gup, const bf16* __restrict__ act,
                                                     bf16* __restrict__ gp, float* gb, Dims fine, int C)
{
    nh::step_kernel_enter();
    const int cx = fine.nx / 2, cy = fine.ny / 2, cz = fine.nz / 2, cvox = cx * cy * cz, cg = C / 8;
    const int total = cvox * fine.batch * cg, first = blockIdx.x * blockDim.x + threadIdx.x;
    float bias[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int i = first; i < total; i += gridDim.x * blockDim.x) {
        const int v = i / cg, q = i - v * cg;
        const int b = v / cvox, r = v - b * cvox;
        const int x = r % cx, y = (r / cx) % cy, z = r / (cx * cy);
        float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int fx = 2 * x + (k & 1), fy = 2 * y + ((k >> 1) & 1), fz = 2 * z + (k >> 2);
            float c[8];
            ld8(gup, (int64_t)(b * fine.nvox + fx + fine.nx * (fy + fine.ny * fz)) * cg + q, c);
#pragma unroll
            for (int j = 0; j < 8; ++j) g[j] += c[j];
        }
        prep_group(g, act, gp, i, bias);
    }
    bias_out(bias, first % cg, C, gb);
}

// ------------------------------------------------------------------ input, head, loss, optimiser

// x[v][0..2] = n_ansatz, x[v][3] = q0 Lz / 2 pi, [4] = Lz / 32, [5] = W0 / 1e-3, rest 0.
__global__ void input_kernel(const float* __restrict__ n, const float* __restrict__ scal, bf16* __restrict__ x, Dims d)
{
    nh::step_kernel_enter();
    const int total = d.nvox * d.batch;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < total; v += gridDim.x * blockDim.x) {
        const int b = v / d.nvox, r = v - b * d.nvox;
        const float* nb = n + (size_t)b * 3 * d.nvox;
        const float q0 = scal[3 * b], lz = scal[3 * b + 1], w0 = scal[3 * b + 2];
        const float vals[8] = {nb[r], nb[d.nvox + r], nb[2 * d.nvox + r], q0 * lz / 6.283185307179586f, lz / 32.f,
                               w0 / 1e-3f, 0.f, 0.f};
        uint4* dst = reinterpret_cast<uint4*>(x + (size_t)v * kInCh);
        dst[0] = pack8(vals);
        dst[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// Head (1x1x1 conv 16 -> 3), residual on the ansatz, normalisation.  Train: the
// loss mean |n - target|^2, the gradients of W_head and b_head, and the last
// convolution's pre-activation gradient (ReLU mask of d1, BF16) and bias gradient.
template <bool Train>
__global__ void __launch_bounds__(256) head_kernel(const bf16* __restrict__ d1, const float* __restrict__ n_ans,
                                                   const float* __restrict__ params_head, float* __restrict__ n_out,
                                                   const float* __restrict__ target, bf16* __restrict__ gp,
                                                   float* __restrict__ gb, float* __restrict__ g_head,
                                                   float* __restrict__ loss, Dims d)
{
    nh::step_kernel_enter();
    constexpr int kW = kHeadOut * kHeadIn, kSums = kW + kHeadOut + 1 + kHeadIn;  // W, b, loss, bias of the last conv
    __shared__ float sh[kW + kHeadOut];
    __shared__ float red[kSums][8];
    for (int k = threadIdx.x; k < kW + kHeadOut; k += blockDim.x) sh[k] = params_head[k];
    __syncthreads();
    const int total = d.nvox * d.batch;
    const float inv_total = 1.f / (float)total;
    float gacc[Train ? kSums : 1];
#pragma unroll
    for (int k = 0; k < (Train ? kSums : 1); ++k) gacc[k] = 0.f;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < total; v += gridDim.x * blockDim.x) {
        const int b = v / d.nvox, r = v - b * d.nvox;
        const size_t o0 = (size_t)b * 3 * d.nvox + r;
        float h[kHeadIn];
        const uint4* row = reinterpret_cast<const uint4*>(d1 + (size_t)v * kHeadIn);
        unpack8(__ldg(row), h);
        unpack8(__ldg(row + 1), h + 8);
        float vv[3];
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            float s = sh[kW + o];
#pragma unroll
            for (int c = 0; c < kHeadIn; ++c) s += sh[o * kHeadIn + c] * h[c];
            vv[o] = n_ans[o0 + (size_t)o * d.nvox] + s;
        }
        const float len = sqrtf(vv[0] * vv[0] + vv[1] * vv[1] + vv[2] * vv[2]);
        const float nn[3] = {vv[0] / len, vv[1] / len, vv[2] / len};
        if (n_out)
#pragma unroll
            for (int o = 0; o < 3; ++o) n_out[o0 + (size_t)o * d.nvox] = nn[o];
        if constexpr (Train) {
            float gn[3], dot = 0.f, l = 0.f;
#pragma unroll
            for (int o = 0; o < 3; ++o) {
                const float diff = nn[o] - target[o0 + (size_t)o * d.nvox];
                l += diff * diff;
                gn[o] = 2.f * diff * inv_total;
                dot += gn[o] * nn[o];
            }
            gacc[kW + kHeadOut] += l * inv_total;
            float gd[3];
#pragma unroll
            for (int o = 0; o < 3; ++o) gd[o] = (gn[o] - dot * nn[o]) / len;  // d/dv of v/|v|
            float g[kHeadIn];
#pragma unroll
            for (int c = 0; c < kHeadIn; ++c) {
                float s = 0.f;
#pragma unroll
                for (int o = 0; o < 3; ++o) {
                    s += sh[o * kHeadIn + c] * gd[o];
                    gacc[o * kHeadIn + c] += gd[o] * h[c];
                }
                g[c] = h[c] > 0.f ? s : 0.f;
                gacc[kW + kHeadOut + 1 + c] += g[c];
            }
#pragma unroll
            for (int o = 0; o < 3; ++o) gacc[kW + o] += gd[o];
            uint4* dst = reinterpret_cast<uint4*>(gp + (size_t)v * kHeadIn);
            dst[0] = pack8(g);
            dst[1] = pack8(g + 8);
        }
    }
    if constexpr (Train) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < kSums; ++k) {
            float s = gacc[k];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) red[k][warp] = s;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < kSums; k += blockDim.x) {
            float s = 0.f;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[k][w];
            if (k < kW + kHeadOut)
                atomicAdd(&g_head[k], s);
            else if (k == kW + kHeadOut)
                atomicAdd(loss, s);
            else
                atomicAdd(&gb[k - (kW + kHeadOut + 1)], s);
        }
    }
}

__global__ void bf16_to_f32_kernel(const bf16* __restrict__ a, float* __restrict__ out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __bfloat162float(a[i]);
}

// BF16 copies of all parameters, and of the convolution weights transposed,
// wt[l][tap][ci][co] = w[l][tap][co][ci], in one launch (one per layer took 45 us).
struct ParamTable {
    int begin[kLayers + 1];  // first parameter of each layer, and of the head
    int cin[kLayers], cout[kLayers];
    bf16* wt[kLayers];
};
__global__ void params_kernel(const float* __restrict__ p, bf16* __restrict__ w, const ParamTable t, int n)
{
    nh::step_kernel_enter();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const bf16 v = __float2bfloat16_rn(p[i]);
        w[i] = v;
        int l = 0;
        while (l < kLayers && i >= t.begin[l + 1]) ++l;
        if (l == kLayers) continue;
        const int k = i - t.begin[l], cc = t.cin[l] * t.cout[l];
        if (k >= 27 * cc) continue;  // bias
        const int tap = k / cc, r = k - tap * cc, co = r / t.cin[l], ci = r - co * t.cin[l];
        t.wt[l][tap * cc + ci * t.cout[l] + co] = v;
    }
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2)
{
    nh::step_kernel_enter();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

inline int grid_for(int64_t n, int threads = 256)
{
    int64_t b = (n + threads - 1) / threads;
    return (int)(b > 4096 ? 4096 : b);
}

}  // namespace

// ------------------------------------------------------------------ network runner

struct nh_unet {
    Dims lv[4];           // level dims (fine to coarse)
    int batch;
    char* ws = nullptr;
    size_t ws_bytes = 0;
    size_t need = 0;
    // offsets into the workspace
    size_t wbf, wt[kLayers], x, act[kLayers], pool_[3], grad, grad_skip[3], gp[2], status;
    std::string err;
};

namespace {

int unet_fail(nh_unet* u, int code, const std::string& m)
{
    if (u) u->err = m;
    nh::set_global_error(m);
    return code;
}

size_t al(size_t v) { return (v + 255) / 256 * 256; }

void plan(nh_unet* u)
{
    size_t off = 0;
    auto take = [&](size_t b) {
        size_t o = off;
        off += al(b);
        return o;
    };
    const int64_t P = total_params();
    u->wbf = take(P * sizeof(bf16));
    for (int l = 0; l < kLayers; ++l) u->wt[l] = take(27 * (size_t)kConv[l].cin * kConv[l].cout * sizeof(bf16));
    const size_t V0 = (size_t)u->lv[0].nvox * u->batch;
    u->x = take(V0 * kInCh * sizeof(bf16));
    const int level_of[kLayers] = {0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0};
    for (int l = 0; l < kLayers; ++l)
        u->act[l] = take((size_t)u->lv[level_of[l]].nvox * u->batch * kConv[l].cout * sizeof(bf16));
    // pooled inputs of levels 1..3
    const int pool_c[3] = {16, 16, 32};
    for (int k = 0; k < 3; ++k) u->pool_[k] = take((size_t)u->lv[k + 1].nvox * u->batch * pool_c[k] * sizeof(bf16));
    // FP32 gradient of a tensor that a pooling or an upsampling produced (at most 16 channels of level 0, 32 of
    // level 1, 64 of level 2), the three skip gradients (e1, e2, e3), and two pre-activation gradients
    u->grad = take(V0 * 16 * sizeof(float));
    const int skip_c[3] = {16, 16, 32};
    for (int k = 0; k < 3; ++k) u->grad_skip[k] = take((size_t)u->lv[k].nvox * u->batch * skip_c[k] * sizeof(float));
    for (int k = 0; k < 2; ++k) u->gp[k] = take(V0 * 16 * sizeof(bf16));  // level 0 has the largest output
    u->status = take(sizeof(int));  // raised by an expired wait of the tensor-core convolution
    u->need = off;
}

template <typename T>
T* P(nh_unet* u, size_t off)
{
    return reinterpret_cast<T*>(u->ws + off);
}

// Forward conv layer l; up1: source 1 is the coarser level's output, read upsampled.
cudaError_t conv_fwd(nh_unet* u, int l, int level, const bf16* s1, int c1, const bf16* s2, int c2, bool up1,
                     const float* params, cudaStream_t st)
{
    ConvTc a{};
    a.src1 = s1;
    a.c1 = c1;
    a.src2 = s2;
    a.c2 = c2;
    a.up1 = up1;
    a.w = P<bf16>(u, u->wbf) + layer_offset(l);
    a.n = kConv[l].cout;
    a.bias = params + layer_offset(l) + 27LL * kConv[l].cin * kConv[l].cout;
    a.out = P<bf16>(u, u->act[l]);
    a.d = u->lv[level];
    a.status = P<int>(u, u->status);
    return launch_conv_tc<false>(a, st);
}

// Backward of conv layer l from its pre-activation gradient gp: weight gradient
// into grad, then the data gradient: of a single source that is layer `below`
// its pre-activation gradient into gp_below (and its bias gradient into grad),
// else (below < 0) FP32 into dst1 (c1 channels) and dst2 (c2); none with both null.
cudaError_t conv_bwd(nh_unet* u, int l, int level, const bf16* gp, const bf16* s1, int c1, const bf16* s2, int c2, bool up1,
                     int below, bf16* gp_below, float* dst1, float* dst2, float* grad, cudaStream_t st)
{
    const Dims d = u->lv[level];
    const int cout = kConv[l].cout, cin = kConv[l].cin;
    ConvBwdW w;
    w.gp = gp;
    w.src1 = s1;
    w.c1 = c1;
    w.src2 = s2;
    w.c2 = c2;
    w.cout = cout;
    w.up1 = up1;
    w.gw = grad + layer_offset(l);
    w.d = d;
    w.tiles = ((d.nx + kWTx - 1) / kWTx) * ((d.ny + kWTy - 1) / kWTy) * ((d.nz + kWTz - 1) / kWTz) * d.batch;
    static bool attr_set = false;  // the opt-in to more than 48 KB of shared memory, once per process
    if (!attr_set) {
        cudaError_t e = cudaFuncSetAttribute(conv_bwd_w_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWSmem);
        if (e != cudaSuccess) return e;
        attr_set = true;
    }
    // one wave of resident blocks over the channel pairs; each walks its share of the tiles
    const int pairs = (cin / 16) * (cout / 16);
    dim3 grid(std::min(w.tiles, std::max(1, kWBlocksPerSM * 152 / pairs)), pairs);
    nh::launch_step_kernel(conv_bwd_w_kernel, grid, kWThreads, kWSmem, st, w);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || (gp_below == nullptr && dst1 == nullptr)) return e;
    ConvTc b{};
    b.src1 = gp;
    b.c1 = cout;
    b.w = P<bf16>(u, u->wt[l]);
    b.n = cin;
    b.d = d;
    if (below >= 0) {
        b.mask = P<bf16>(u, u->act[below]);
        b.gp = gp_below;
        b.gb = grad + layer_offset(below) + 27LL * kConv[below].cin * kConv[below].cout;
    }
    b.dst1 = dst1;
    b.n1 = c1;
    b.dst2 = dst2;
    b.status = P<int>(u, u->status);
    return launch_conv_tc<true>(b, st);
}

// Grid of the group kernels: a stride that is a multiple of C / 8 (1, 2, 4 or 8).
inline int group_grid(int64_t groups) { return (int)std::min<int64_t>(8 * 152, (groups + 255) / 256); }

}  // namespace

#define UNET_CUDA(u, ...)                                                                      \
    do {                                                                                       \
        cudaError_t e_ = (__VA_ARGS__);                                                        \
        if (e_ != cudaSuccess) return unet_fail((u), NH_ECUDA, std::string(#__VA_ARGS__) + ": " + cudaGetErrorString(e_)); \
    } while (0)

extern "C" {

int64_t nh_unet_param_count(void) { return total_params(); }

int nh_unet_create(int batch, int nx, int ny, int nz, nh_unet** out)
{
    if (!out) return unet_fail(nullptr, NH_EINVAL, "out is NULL");
    *out = nullptr;
    if (batch < 1 || nx < 16 || ny < 16 || nz < 8 || nx % 8 || ny % 8 || nz % 8)
        return unet_fail(nullptr, NH_EINVAL, "batch >= 1; nx, ny multiples of 8 and >= 16; nz a multiple of 8");
    if ((int64_t)nx * ny * nz * batch * 96 > 2000000000LL) return unet_fail(nullptr, NH_EINVAL, "problem too large");
    nh_unet* u = new (std::nothrow) nh_unet();
    if (!u) return unet_fail(nullptr, NH_ENOMEM, "host allocation failed");
    u->batch = batch;
    for (int k = 0; k < 4; ++k) {
        const int s = 1 << k;
        u->lv[k] = Dims{nx / s, ny / s, nz / s, (nx / s) * (ny / s) * (nz / s), batch};
    }
    if ((u->lv[3].nvox * batch) % 16) {
        delete u;
        return unet_fail(nullptr, NH_EINVAL, "the coarsest level must hold a multiple of 16 voxels");
    }
    plan(u);
    *out = u;
    return NH_OK;
}

int nh_unet_workspace_bytes(const nh_unet* u, size_t* bytes)
{
    if (!u || !bytes) return unet_fail(nullptr, NH_EINVAL, "NULL argument");
    *bytes = u->need;
    return NH_OK;
}

int nh_unet_bind(nh_unet* u, void* ws, size_t bytes)
{
    if (!u || !ws) return unet_fail(u, NH_EINVAL, "NULL argument");
    if (reinterpret_cast<uintptr_t>(ws) % 256) return unet_fail(u, NH_EINVAL, "workspace must be 256-byte aligned");
    if (bytes < u->need) return unet_fail(u, NH_ENOMEM, "workspace too small: need " + std::to_string(u->need));
    u->ws = static_cast<char*>(ws);
    u->ws_bytes = bytes;
    UNET_CUDA(u, cudaMemset(u->ws + u->status, 0, sizeof(int)));
    return NH_OK;
}

int nh_unet_status(nh_unet* u, void* stream)
{
    if (!u || !u->ws) return unet_fail(u, NH_EINVAL, "unbound network");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    int flag = 0;
    UNET_CUDA(u, cudaMemcpyAsync(&flag, u->ws + u->status, sizeof(int), cudaMemcpyDeviceToHost, st));
    UNET_CUDA(u, cudaStreamSynchronize(st));
    if (flag) {
        UNET_CUDA(u, cudaMemsetAsync(u->ws + u->status, 0, sizeof(int), st));
        return unet_fail(u, NH_ETIMEOUT, "a tensor-core convolution gave up waiting for its MMAs");
    }
    return NH_OK;
}

int nh_unet_set_params(nh_unet* u, const float* params, void* stream)
{
    if (!u || !u->ws || !params) return unet_fail(u, NH_EINVAL, "unbound network or NULL params");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int n = (int)total_params();
    ParamTable t;
    for (int l = 0; l < kLayers; ++l) {
        t.begin[l] = (int)layer_offset(l);
        t.cin[l] = kConv[l].cin;
        t.cout[l] = kConv[l].cout;
        t.wt[l] = P<bf16>(u, u->wt[l]);
    }
    t.begin[kLayers] = (int)head_offset();
    nh::launch_step_kernel(params_kernel, grid_for(n), 256, 0, st, params, P<bf16>(u, u->wbf), t, n);
    UNET_CUDA(u, cudaGetLastError());
    return NH_OK;
}

int nh_unet_forward(nh_unet* u, const float* params, const float* n_ansatz, const float* scalars, float* n_out,
                    void* stream)
{
    if (!u || !u->ws || !params || !n_ansatz || !scalars) return unet_fail(u, NH_EINVAL, "NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const Dims d0 = u->lv[0];
    nh::launch_step_kernel(input_kernel, grid_for((int64_t)d0.nvox * d0.batch), 256, 0, st, n_ansatz, scalars,
                           P<bf16>(u, u->x), d0);
    UNET_CUDA(u, cudaGetLastError());
    auto act = [&](int l) { return P<bf16>(u, u->act[l]); };
    auto pool = [&](int k) { return P<bf16>(u, u->pool_[k]); };
    UNET_CUDA(u, conv_fwd(u, ENC1A, 0, P<bf16>(u, u->x), 16, nullptr, 0, false, params, st));
    UNET_CUDA(u, conv_fwd(u, ENC1B, 0, act(ENC1A), 16, nullptr, 0, false, params, st));
    nh::launch_step_kernel(pool_fwd_kernel, group_grid((int64_t)u->lv[1].nvox * u->batch * 2), 256, 0, st, act(ENC1B), pool(0),
                           u->lv[0], 16);
    UNET_CUDA(u, conv_fwd(u, ENC2A, 1, pool(0), 16, nullptr, 0, false, params, st));
    UNET_CUDA(u, conv_fwd(u, ENC2B, 1, act(ENC2A), 16, nullptr, 0, false, params, st));
    nh::launch_step_kernel(pool_fwd_kernel, group_grid((int64_t)u->lv[2].nvox * u->batch * 2), 256, 0, st, act(ENC2B), pool(1),
                           u->lv[1], 16);
    UNET_CUDA(u, conv_fwd(u, ENC3A, 2, pool(1), 16, nullptr, 0, false, params, st));
    UNET_CUDA(u, conv_fwd(u, ENC3B, 2, act(ENC3A), 32, nullptr, 0, false, params, st));
    nh::launch_step_kernel(pool_fwd_kernel, group_grid((int64_t)u->lv[3].nvox * u->batch * 4), 256, 0, st, act(ENC3B), pool(2),
                           u->lv[2], 32);
    UNET_CUDA(u, conv_fwd(u, BOTA, 3, pool(2), 32, nullptr, 0, false, params, st));
    UNET_CUDA(u, conv_fwd(u, BOTB, 3, act(BOTA), 64, nullptr, 0, false, params, st));
    UNET_CUDA(u, conv_fwd(u, DEC3A, 2, act(BOTB), 64, act(ENC3B), 32, true, params, st));
    UNET_CUDA(u, conv_fwd(u, DEC3B, 2, act(DEC3A), 32, nullptr, 0, false, params, st));
    UNET_CUDA(u, conv_fwd(u, DEC2A, 1, act(DEC3B), 32, act(ENC2B), 16, true, params, st));
    UNET_CUDA(u, conv_fwd(u, DEC2B, 1, act(DEC2A), 16, nullptr, 0, false, params, st));
    UNET_CUDA(u, conv_fwd(u, DEC1A, 0, act(DEC2B), 16, act(ENC1B), 16, true, params, st));
    UNET_CUDA(u, conv_fwd(u, DEC1B, 0, act(DEC1A), 16, nullptr, 0, false, params, st));
    nh::launch_step_kernel(head_kernel<false>, grid_for((int64_t)d0.nvox * d0.batch), 256, 0, st, act(DEC1B), n_ansatz,
                           params + head_offset(), n_out, nullptr, nullptr, nullptr, nullptr, nullptr, d0);
    UNET_CUDA(u, cudaGetLastError());
    return NH_OK;
}

int nh_unet_backward(nh_unet* u, const float* params, const float* n_ansatz, const float* target, float* grad,
                     float* loss, void* stream)
{
    if (!u || !u->ws || !params || !n_ansatz || !target || !grad || !loss)
        return unet_fail(u, NH_EINVAL, "NULL argument");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const Dims d0 = u->lv[0];
    UNET_CUDA(u, cudaMemsetAsync(grad, 0, total_params() * sizeof(float), st));
    UNET_CUDA(u, cudaMemsetAsync(loss, 0, sizeof(float), st));
    auto act = [&](int l) { return P<bf16>(u, u->act[l]); };
    auto pool = [&](int k) { return P<bf16>(u, u->pool_[k]); };
    float* g = P<float>(u, u->grad);
    float* gskip[3] = {P<float>(u, u->grad_skip[0]), P<float>(u, u->grad_skip[1]), P<float>(u, u->grad_skip[2])};
    bf16 *gpa = P<bf16>(u, u->gp[0]), *gpb = P<bf16>(u, u->gp[1]);
    auto gbias = [&](int l) { return grad + layer_offset(l) + 27LL * kConv[l].cin * kConv[l].cout; };
    // layer l read by an upsampling to level `fine`, or by a pooling from level `fine` and a skip connection
    auto up_bwd = [&](int l, int fine) {
        const int C = kConv[l].cout;
        nh::launch_step_kernel(up_bwd_kernel, group_grid((int64_t)u->lv[fine + 1].nvox * u->batch * (C / 8)), 256, 0, st, g,
                               act(l), gpa, gbias(l), u->lv[fine], C);
        return cudaGetLastError();
    };
    auto pool_bwd = [&](int l, int fine) {
        const int C = kConv[l].cout;
        nh::launch_step_kernel(pool_bwd_kernel, group_grid((int64_t)u->lv[fine].nvox * u->batch * (C / 8)), 256, 0, st, g,
                               gskip[fine], act(l), gpa, gbias(l), u->lv[fine], C);
        return cudaGetLastError();
    };
    nh::launch_step_kernel(head_kernel<true>, std::min(4 * 152, grid_for((int64_t)d0.nvox * d0.batch)), 256, 0, st,
                           act(DEC1B), n_ansatz, params + head_offset(), nullptr, target, gpa, gbias(DEC1B),
                           grad + head_offset(), loss, d0);
    UNET_CUDA(u, cudaGetLastError());
    // decoder: of each level the second convolution, then the first, whose sources are the upsampled level
    // below and the encoder's skip connection
    UNET_CUDA(u, conv_bwd(u, DEC1B, 0, gpa, act(DEC1A), 16, nullptr, 0, false, DEC1A, gpb, nullptr, nullptr, grad, st));
    UNET_CUDA(u, conv_bwd(u, DEC1A, 0, gpb, act(DEC2B), 16, act(ENC1B), 16, true, -1, nullptr, g, gskip[0], grad, st));
    UNET_CUDA(u, up_bwd(DEC2B, 0));
    UNET_CUDA(u, conv_bwd(u, DEC2B, 1, gpa, act(DEC2A), 16, nullptr, 0, false, DEC2A, gpb, nullptr, nullptr, grad, st));
    UNET_CUDA(u, conv_bwd(u, DEC2A, 1, gpb, act(DEC3B), 32, act(ENC2B), 16, true, -1, nullptr, g, gskip[1], grad, st));
    UNET_CUDA(u, up_bwd(DEC3B, 1));
    UNET_CUDA(u, conv_bwd(u, DEC3B, 2, gpa, act(DEC3A), 32, nullptr, 0, false, DEC3A, gpb, nullptr, nullptr, grad, st));
    UNET_CUDA(u, conv_bwd(u, DEC3A, 2, gpb, act(BOTB), 64, act(ENC3B), 32, true, -1, nullptr, g, gskip[2], grad, st));
    UNET_CUDA(u, up_bwd(BOTB, 2));
    // bottleneck
    UNET_CUDA(u, conv_bwd(u, BOTB, 3, gpa, act(BOTA), 64, nullptr, 0, false, BOTA, gpb, nullptr, nullptr, grad, st));
    UNET_CUDA(u, conv_bwd(u, BOTA, 3, gpb, pool(2), 32, nullptr, 0, false, -1, nullptr, g, nullptr, grad, st));
    // encoder: each level's output feeds the pooling and the skip connection
    UNET_CUDA(u, pool_bwd(ENC3B, 2));
    UNET_CUDA(u, conv_bwd(u, ENC3B, 2, gpa, act(ENC3A), 32, nullptr, 0, false, ENC3A, gpb, nullptr, nullptr, grad, st));
    UNET_CUDA(u, conv_bwd(u, ENC3A, 2, gpb, pool(1), 16, nullptr, 0, false, -1, nullptr, g, nullptr, grad, st));
    UNET_CUDA(u, pool_bwd(ENC2B, 1));
    UNET_CUDA(u, conv_bwd(u, ENC2B, 1, gpa, act(ENC2A), 16, nullptr, 0, false, ENC2A, gpb, nullptr, nullptr, grad, st));
    UNET_CUDA(u, conv_bwd(u, ENC2A, 1, gpb, pool(0), 16, nullptr, 0, false, -1, nullptr, g, nullptr, grad, st));
    UNET_CUDA(u, pool_bwd(ENC1B, 0));
    UNET_CUDA(u, conv_bwd(u, ENC1B, 0, gpa, act(ENC1A), 16, nullptr, 0, false, ENC1A, gpb, nullptr, nullptr, grad, st));
    // (the input needs no gradient)
    UNET_CUDA(u, conv_bwd(u, ENC1A, 0, gpb, P<bf16>(u, u->x), 16, nullptr, 0, false, -1, nullptr, nullptr, nullptr, grad, st));
    return NH_OK;
}

int nh_unet_activation(nh_unet* u, int layer, float* out, void* stream)
{
    if (!u || !u->ws || !out || layer < 0 || layer >= kLayers) return unet_fail(u, NH_EINVAL, "bad arguments");
    const int level_of[kLayers] = {0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0};
    const int64_t n = (int64_t)u->lv[level_of[layer]].nvox * u->batch * kConv[layer].cout;
    bf16_to_f32_kernel<<<grid_for(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(P<bf16>(u, u->act[layer]), out, n);
    UNET_CUDA(u, cudaGetLastError());
    return NH_OK;
}

int nh_unet_adam(float* params, const float* grad, float* m, float* v, int64_t count, int step, float lr, void* stream)
{
    if (!params || !grad || !m || !v || count < 1 || step < 1) return unet_fail(nullptr, NH_EINVAL, "bad Adam arguments");
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    nh::launch_step_kernel(adam_kernel, grid_for(count), 256, 0, static_cast<cudaStream_t>(stream), params, grad, m, v,
                           count, lr, b1, b2, 1e-8f, c1, c2);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return unet_fail(nullptr, NH_ECUDA, std::string("adam: ") + cudaGetErrorString(e));
    return NH_OK;
}

void nh_unet_destroy(nh_unet* u) { delete u; }

}  // extern "C"
