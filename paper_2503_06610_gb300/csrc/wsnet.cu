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
// One CTA (five warps) computes 8 x 16 voxels x NB output channels of a chunk of
// z planes.  It walks along the *input* planes: a plane with a one-voxel halo in x
// and y (10 x 18 voxels) is copied once into a ring of shared-memory slots, in
// the tensor core's no-swizzle K-major layout with 16-byte channel groups of
// consecutive voxels next to each other.  The eight voxels of an x run are a core
// matrix, so the A operand of each of the nine (dy, dx) taps is the same plane
// read from a shifted start address (LBO = one channel-group plane, SBO = one row
// of ten voxels).  An input plane is a term of the three output planes next to it:
// their accumulators are neighbours on a strip of 128 TMEM columns, and the three
// dz taps' weights are stacked to 3 NB rows of B, so that one MMA (M = 128,
// N = 3 NB, K = 16) serves all three.  At N = 16 an MMA is bound by reading A from
// shared memory, whatever N is up to 48.  (16 -> 16 layer of 8 x 64 x 64 x 32
// voxels, caches cold: 339 us with each tap's rows copied, 41 us with one MMA per
// tap, 28 us so.)  Where the window of three runs past the strip's end it is
// issued in two parts; the accumulator that enters the window is cleared by its
// first MMA, and the two that lie outside the chunk are not read.
// The weights of all taps stay in shared memory for the CTA's life.  The fifth
// warp issues a plane's MMAs and commits them to an mbarrier; the other four copy
// the planes to come and write the output plane that the previous input plane
// completed meanwhile.  What bounds the kernel is the issuing warp's instructions
// (predicating the MMAs off changes nothing, leaving out copies or epilogue
// neither), so K is a template argument and the descriptors are constants added to
// two bases: eight cells' forward pass 281 us with K at run time, 242 us so.
// Every mbarrier wait is bounded: on expiry the kernel raises a.status, skips the
// epilogue, waits (again with a limit) for its copies and MMAs and frees its TMEM.
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
    const bf16* w;     // the weights' image (tc_weight_index)
    int n;             // output channels; blockIdx.y takes NB of them
    Dims d;
    int zc;            // planes per chunk
    int ring;          // input planes held in shared memory, 2 ... kTcMaxRing
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
constexpr int kTcCopy = 128;     // threads of the four warps that copy planes and run the epilogue
constexpr int kTcThreads = 160;  // and a warp that issues the MMAs
constexpr int kTcX = 8, kTcY = 16;                                // output voxels of a plane step
constexpr int kTcHX = kTcX + 2, kTcHY = kTcY + 2, kTcHalo = kTcHX * kTcHY;
constexpr int kTcMaxRing = 5;      // input planes held: one in use, the others being copied
constexpr uint32_t kTcCols = 128;  // TMEM columns of a CTA: a strip of 128 / NB accumulators
// Ring, weights, voxel offsets, barriers, bias.  At least 46 KB, so that an SM takes at most the four CTAs whose
// 512 columns it has.
inline size_t tc_smem(int K, int NB, int ring)
{
    const size_t b = (size_t)K * 2 * (ring * kTcHalo + 27 * NB) + 2 * kTcHalo * sizeof(int) + 64 + NB * sizeof(float);
    return std::max<size_t>(b, 46 * 1024);
}
constexpr size_t kTcMaxSmem = 227 * 1024, kTcSmSmem = 228 * 1024;  // of a block, of an SM

// Output channels of a CTA: 32 where two such weight sets fit an SM, else 16 (more CTAs on the coarse levels, whose
// wide layers have few voxels).
__host__ __device__ constexpr int tc_nb(int n, int K) { return n % 32 == 0 && K <= 32 ? 32 : 16; }

// Where w[tap][row][k] (n rows of K) stands in the image that the CTAs copy: per group of NB rows the B operands of
// the nine (dy, dx) taps as they lie in shared memory, 3 NB rows each (dz tap 2, then 1, then 0, for the
// output planes that an input plane is the last, second and first term of), rows of eight and 16-byte groups of k as the tensor core's core matrices.  A CTA's part
// is contiguous, one bulk copy: copied and arranged by each CTA's threads, the weights took 92 us of the 366 us of
// the fourteen layers' forward pass of eight cells of 64 x 64 x 32, most of it in layers of few CTAs.
__device__ __forceinline__ int tc_weight_index(int n, int K, int tap, int row, int k)
{
    const int NB = tc_nb(n, K), r = (2 - tap / 9) * NB + row % NB;
    return row / NB * (27 * NB * K) + ((tap % 9 * (3 * NB / 8) + r / 8) * (K / 8) + k / 8) * 64 + r % 8 * 8 + k % 8;
}

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

template <int NB, bool Flip, int K>
__global__ void __launch_bounds__(kTcThreads, NB == 32 && Flip ? 3 : 4) conv_tc_kernel(const ConvTc a)
{
    extern __shared__ __align__(128) unsigned char tc_smem_raw[];
    constexpr int kb = K / 8;  // 16-byte channel groups
    constexpr uint32_t kGroup = kTcHalo * 16;              // one channel group of a plane
    constexpr uint32_t plane_bytes = (uint32_t)kb * kGroup;
    constexpr uint32_t tap_bytes = 3u * NB * K * 2;  // of a (dy, dx) tap
    const uint32_t ring = smem_u32(tc_smem_raw), wbase = ring + (uint32_t)a.ring * plane_bytes;
    int* voxel = reinterpret_cast<int*>(tc_smem_raw + (uint32_t)a.ring * plane_bytes + 9 * tap_bytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(voxel + 2 * kTcHalo);
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 5);
    float* bshared = reinterpret_cast<float*>(bars + 8);  // bias gradient of the CTA's voxels (with mask)
    if (Flip && threadIdx.x < NB) bshared[threadIdx.x] = 0.f;
    constexpr int kSlots = kTcCols / NB;
    static_assert(NB == 16 || NB == 32, "3 NB is a valid N, and the strip holds the window of three and one being read");
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
                     "r"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    // bars[0], [1]: the MMAs of an even or odd input plane are done; bars[2], [3]: its copies are; bars[4]: the weights are here
    if (tid == 0) {
#pragma unroll
        for (int i = 0; i < 5; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(&bars[i])), "r"(i == 2 || i == 3 ? kTcCopy : 1)
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }

    // a thread copies one channel group of every vstep-th voxel of a plane
    const int cq = tid % kb, vfirst = tid / kb, vstep = kTcCopy / kb;
    const bool loader = tid < kTcCopy && vfirst < vstep;
    const bool from1 = cq * 8 < a.c1;
    const bool up = from1 && a.up1;
    const bf16* lsrc = from1 ? a.src1 + cq * 8 : a.src2 + (cq * 8 - a.c1);
    const int lc = from1 ? a.c1 : a.c2;
    // where a plane's voxels lie in a z layer of the source, and in one of half the resolution
    for (int v = tid; v < kTcHalo; v += kTcThreads) {
        const int hy = v / kTcHX, hx = v - hy * kTcHX;
        int x = x0 - 1 + hx, y = y0 - 1 + hy;
        x = x < 0 ? x + d.nx : (x >= d.nx ? x - d.nx : x);
        y = y < 0 ? y + d.ny : (y >= d.ny ? y - d.ny : y);
        const bool ok = x < d.nx && y < d.ny;  // beyond a ragged tile's halo: unused, zero
        voxel[v] = ok ? x + d.nx * y : -1;
        voxel[kTcHalo + v] = ok ? (x >> 1) + (d.nx >> 1) * (y >> 1) : -1;
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    nh::step_kernel_enter();  // nothing above reads or writes global memory
    if (tid == kTcCopy) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(&bars[4])), "r"(9 * tap_bytes)
                     : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(wbase),
                     "l"(a.w + (size_t)blockIdx.y * (27 * NB * K)), "r"(9 * tap_bytes), "r"(smem_u32(&bars[4]))
                     : "memory");
    }
    const int* lvox = voxel + (up ? kTcHalo : 0);
    int lslot = 0;
    // the input planes upwards from z0 - 1, for the mirrored taps of the data gradient downwards from z1: either way
    // an output plane's terms come in the order of the taps
    auto plane = [&](int w) { return Flip ? z1 - w : z0 - 1 + w; };
    auto load_plane = [&](int w) {  // input plane w, zero beyond the volume in z; nothing beyond the chunk's
        if (loader && w < z1 - z0 + 2) {
            const int z = plane(w);
            const bool zin = z >= 0 && z < d.nz;
            const uint32_t dst = ring + (uint32_t)lslot * plane_bytes + (uint32_t)cq * kGroup;
            const int first = up ? batch * (d.nvox >> 3) + (d.nx >> 1) * (d.ny >> 1) * (z >> 1) : batch * d.nvox + d.nx * d.ny * z;
            for (int v = vfirst; v < kTcHalo; v += vstep) {
                const int o = lvox[v];
                const bool ok = zin && o >= 0;
                cp_async16(dst + (uint32_t)v * 16u, ok ? lsrc + (size_t)(first + o) * lc : lsrc, ok);
            }
        }
        if (++lslot == a.ring) lslot = 0;
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    const int steps = z1 - z0 + 2;  // input planes z0 - 1 ... z1
    if (tid < kTcCopy)
        for (int w = 0; w < a.ring - 1; ++w) load_plane(w);

    // row r of the accumulator is voxel (x0 + r % 8, y0 + r / 8) of the plane
    const int row = warp * 32 + lane;
    const int vx = x0 + (row & 7), vy = y0 + (row >> 3);
    const bool inside = vx < d.nx && vy < d.ny;
    float bsum[Flip ? NB : 1];  // bias gradient of this thread's voxels (with mask)
#pragma unroll
    for (int i = 0; i < (Flip ? NB : 1); ++i) bsum[i] = 0.f;
    // the epilogue's operands, on their way while the tensor core works: the bias, or the next plane's ReLU mask
    float bias[Flip ? 1 : NB];
    uint4 mask[Flip ? NB / 8 : 1];
    if constexpr (!Flip) {
#pragma unroll
        for (int i = 0; i < NB; ++i) bias[i] = __ldg(a.bias + n0 + i);
    }
    auto load_mask = [&](int k) {
        if constexpr (Flip)
            if (a.mask != nullptr && inside && k < z1 - z0) {
                const int z = plane(k + 1);
                const size_t v = (size_t)batch * d.nvox + vx + (size_t)d.nx * (vy + (size_t)d.ny * z);
#pragma unroll
                for (int h = 0; h < NB / 8; ++h) mask[h] = __ldg(reinterpret_cast<const uint4*>(a.mask + v * a.n + n0) + h);
            }
    };
    load_mask(0);
    auto epilogue = [&](int k) {  // the k-th output plane
        const int z = plane(k + 1);
        const uint32_t acc0 = tmem + (uint32_t)((k + 2) % kSlots * NB) + ((uint32_t)(warp * 32) << 16);
        const size_t v = (size_t)batch * d.nvox + vx + (size_t)d.nx * (vy + (size_t)d.ny * z);
#pragma unroll
        for (int c0 = 0; c0 < NB; c0 += 16) {
            float acc[16];
            tmem_ld16(acc0 + (uint32_t)c0, acc);
            if (!inside) continue;
            if constexpr (!Flip) {
                uint32_t packed[8];
#pragma unroll
                for (int i = 0; i < 8; ++i)
                    packed[i] = pack_bf16(fmaxf(acc[2 * i] + bias[c0 + 2 * i], 0.f),
                                          fmaxf(acc[2 * i + 1] + bias[c0 + 2 * i + 1], 0.f));
                uint4* dst = reinterpret_cast<uint4*>(a.out + v * a.n + n0 + c0);
                dst[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
                dst[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
            } else if (a.mask != nullptr) {
                uint4* dst = reinterpret_cast<uint4*>(a.gp + v * a.n + n0 + c0);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float* g = acc + 8 * h;
                    relu_mask(g, mask[c0 / 8 + h]);
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
        load_mask(k + 1);
    };

    bool ok = true;
    if (warp == kTcCopy / 32) {
        // The warp runs as one, its first lane's instructions taking effect: descriptors stay in uniform registers.
        const uint32_t lead = lane == 0;
        const uint64_t ad0 = umma_desc(0, kGroup, kTcHX * 16), bd0 = umma_desc(0, 128u, (uint32_t)kb * 128u);
        ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[4]), 0)) != 0;
        int issued = 0;  // input planes whose MMAs are under way or done
        // accumulators w, w + 1, w + 2 of the strip: output planes number w - 2, w - 1 and w of the chunk
        for (int w = 0, slot = 0; w < steps && ok; ++w, slot = slot + 1 == a.ring ? 0 : slot + 1) {
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[2 + (w & 1)]), (w >> 1) & 1)) != 0;
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t pa = (ring + (uint32_t)slot * plane_bytes) >> 4;
            const int s = w % kSlots;
            // rows o ... o + count - 1 of the stacked weights into the accumulators from slot t on
            auto mma = [&](int q, int j, int o, int count, int t, uint32_t acc) {
                const int off = Flip ? (2 - q / 3) * kTcHX + (2 - q % 3) : (q / 3) * kTcHX + q % 3;
                const uint64_t ad = ad0 | (uint64_t)(pa + off + (uint32_t)j * (2 * kGroup >> 4));
                const uint64_t bd = bd0 | (uint64_t)(((wbase + (uint32_t)q * tap_bytes) >> 4) +
                                                     (uint32_t)o * (uint32_t)(NB * kb) + (uint32_t)j * 16u);
                asm volatile(
                    "{\n.reg .pred p, l;\nsetp.ne.b32 p, %4, 0;\nsetp.ne.b32 l, %5, 0;\n"
                    "@l tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + (uint32_t)(t * NB)),
                    "l"(ad), "l"(bd), "r"(umma_idesc_bf16(kTcM, count * NB)), "r"(acc), "r"(lead)
                    : "memory");
            };
            const int head = min(3, kSlots - s);  // accumulators of the window before the strip's end
            if (head == 1) {
                mma(0, 0, 0, 1, s, 1);
                mma(0, 0, 1, 1, 0, 1);
            } else {
                mma(0, 0, 0, 2, s, 1);
            }
            mma(0, 0, 2, 1, (s + 2) % kSlots, 0);
            auto rest = [&](auto&& f) {
#pragma unroll
                for (int i = 1; i < 9 * (kb / 2); ++i) f(i / (kb / 2), i % (kb / 2));
            };
            if (head == 3)
                rest([&](int q, int j) { mma(q, j, 0, 3, s, 1); });
            else
                rest([&](int q, int j) {
                    mma(q, j, 0, head, s, 1);
                    mma(q, j, head, 3 - head, 0, 1);
                });
            asm volatile("{\n.reg .pred l;\nsetp.ne.b32 l, %1, 0;\n"
                         "@l tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(
                             smem_u32(&bars[w & 1])), "r"(lead)
                         : "memory");
            __syncwarp();
            issued = w + 1;
        }
        if (!ok) {  // nothing of this CTA's may be under way when it leaves: the weights' copy, the last plane's MMAs
            mbar_wait(smem_u32(&bars[4]), 0);
            if (issued > 0) mbar_wait(smem_u32(&bars[(issued - 1) & 1]), ((issued - 1) >> 1) & 1);
        }
    } else {
        for (int w = 0; w < steps && ok; ++w) {
            if (a.ring == 5)
                asm volatile("cp.async.wait_group 3;\n" ::: "memory");
            else if (a.ring == 4)
                asm volatile("cp.async.wait_group 2;\n" ::: "memory");
            else if (a.ring == 3)
                asm volatile("cp.async.wait_group 1;\n" ::: "memory");
            else
                asm volatile("cp.async.wait_group 0;\n" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // the copies, to the tensor core's view
            asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");  // the epilogue's TMEM reads
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(&bars[2 + (w & 1)])) : "memory");
            // the MMAs of the plane before are done: its slot takes the next to come, and its lowest output is complete
            if (w > 0) ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[(w - 1) & 1]), ((w - 1) >> 1) & 1)) != 0;
            if (ok) load_plane(w + a.ring - 1);
            if (ok && w > 2) {
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                epilogue(w - 3);
            }
        }
        if (ok) {
            const int k = steps - 1;
            ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars[k & 1]), (k >> 1) & 1)) != 0;
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            if (ok) epilogue(steps - 3);
        }
    }
    if (!ok && lane == 0) atomicExch(a.status, 1);
    if constexpr (Flip) {
        if (a.mask != nullptr && tid < kTcCopy) {
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
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTcCols) : "memory");
    }
}

// Launch over every plane tile of the level.  Planes per chunk and of the ring: the
// CTAs run in waves of as many as an SM holds (shared memory, TMEM columns,
// registers), and a chunk loads two planes beyond its own; the pair with the least
// waves x (planes + 2).  (8 x 64 x 64 x 32 voxels at K = 32: three planes held, three
// CTAs an SM and two waves of 11 planes 66 us, two held, four an SM and one wave of
// 16 planes 55 us, both with K at run time.)
template <bool Flip, int K, int NB>
cudaError_t launch_conv_tc(ConvTc a, cudaStream_t st)
{
    static nh::OncePerDevice once;  // the opt-in to more than 48 KB of shared memory
    const cudaError_t e = nh::once_per_device(once, [] {
        return cudaFuncSetAttribute(conv_tc_kernel<NB, Flip, K>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kTcMaxSmem);
    });
    if (e != cudaSuccess) return e;
    if (a.n % NB || a.c1 % 8) return cudaErrorInvalidValue;
    const int cols = ((a.d.nx + kTcX - 1) / kTcX) * ((a.d.ny + kTcY - 1) / kTcY) * a.d.batch;
    int64_t best = -1;
    for (int ring = 2; ring <= kTcMaxRing && tc_smem(K, NB, ring) <= kTcMaxSmem; ++ring) {
        const int per_sm = std::min((int)(kTcSmSmem / (tc_smem(K, NB, ring) + 1024)), NB == 32 && Flip ? 3 : 4);
        for (int n = 1; n <= a.d.nz; ++n) {
            const int zc = (a.d.nz + n - 1) / n;
            const int64_t blocks = (int64_t)cols * ((a.d.nz + zc - 1) / zc) * (a.n / NB);
            const int64_t cost = (blocks + 152 * per_sm - 1) / (152 * per_sm) * (zc + 2);
            if (best >= 0 && (cost > best || (cost == best && ring == a.ring))) continue;
            best = cost;
            a.zc = zc;
            a.ring = ring;
        }
    }
    const dim3 grid(cols * ((a.d.nz + a.zc - 1) / a.zc), a.n / NB);
    nh::launch_step_kernel(conv_tc_kernel<NB, Flip, K>, grid, kTcThreads, tc_smem(K, NB, a.ring), st, a);
    return cudaGetLastError();
}

// The depths K and widths that the network's layers have, forward and (Flip) backward.
template <bool Flip>
cudaError_t launch_conv_tc(const ConvTc& a, cudaStream_t st)
{
    const int K = a.c1 + a.c2, NB = tc_nb(a.n, K);
    if (K == 16) return NB == 32 ? launch_conv_tc<Flip, 16, 32>(a, st) : launch_conv_tc<Flip, 16, 16>(a, st);
    if (K == 32) return NB == 32 ? launch_conv_tc<Flip, 32, 32>(a, st) : launch_conv_tc<Flip, 32, 16>(a, st);
    if (K == 64) return launch_conv_tc<Flip, 64, 16>(a, st);
    if constexpr (!Flip) {  // concatenated sources
        if (K == 48) return launch_conv_tc<Flip, 48, 16>(a, st);
        if (K == 96) return launch_conv_tc<Flip, 96, 16>(a, st);
    }
    return cudaErrorInvalidValue;
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
// ldmatrix of the gradient is multiplied with nine of the shifted activations,
// whose pairs of rows serve all three dy (five ldmatrix per dx and layer instead of
// twelve); the 9 x 16 x 16 sums stay in registers (72 a thread) until the block's
// last tile.  Two blocks an SM of 164 registers: 36 us for that layer with an
// ldmatrix per tap and three blocks of 96 registers, with spills if those kept the
// rows; with caches cold 58 us then and 45 us now.  Rows are 32 bytes; their two 16-byte halves are swapped on every other
// group of four voxels of a run, so that the eight rows of an ldmatrix hit
// distinct banks at any x shift.
constexpr int kWTx = 8, kWTy = 8, kWTz = 4, kWVox = kWTx * kWTy * kWTz;
constexpr int kWHx = kWTx + 2, kWHy = kWTy + 2, kWHz = kWTz + 2, kWHalo = kWHx * kWHy * kWHz;
constexpr int kWThreads = 192;
constexpr int kWStage = (kWVox + kWHalo) * 32;  // bytes: gradient rows, then activation rows
constexpr int kWSmem = 2 * kWStage;
constexpr int kWBlocksPerSM = 2;
static_assert(kWHx * kWHy * 2 == kWThreads + 8 && 8 * kWHz <= kWThreads, "the halo's copies");

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

    // tile t and its successors t + gridDim.x, ...: x, y, z, batch advance with carries
    int t = blockIdx.x, bx = t % tx, by = t / tx % ty, bz = t / (tx * ty) % tz, bb = t / (tx * ty * tz);
    const int G = gridDim.x, sx = G % tx, sy = G / tx % ty, sz = G / (tx * ty) % tz, sb = G / (tx * ty * tz);
    // Copies of the current tile into stage s; rows outside the volume (and the gradient of voxels beyond a ragged
    // tile's end) are zero.  A thread copies one half row of the halo's 10 x 10 columns in all its layers (the last
    // eight of the 200 half rows go to 48 threads, a layer each), so that a column's wrapped address is found once.
    const int h2 = kWThreads + (tid & 7);
    auto load_halo = [&](uint32_t X, int h, int z0, int lo, int hi) {
        const int c = h & 1, hy = (h >> 1) / kWHx, hx = (h >> 1) - hy * kWHx;
        int x = bx * kWTx - 1 + hx, y = by * kWTy - 1 + hy;
        x = x < 0 ? x + d.nx : (x >= d.nx ? x - d.nx : x);
        y = y < 0 ? y + d.ny : (y >= d.ny ? y - d.ny : y);
        const bool xyok = x < d.nx && y < d.ny;
        const int shift = up ? 1 : 0, layer = (d.nx >> shift) * (d.ny >> shift);
        const bf16* col = xs + (size_t)(bb * (up ? d.nvox >> 3 : d.nvox) + (x >> shift) + (d.nx >> shift) * (y >> shift)) * xc + 8 * c;
        const uint32_t dst = X + (uint32_t)(h >> 1) * 32u + (uint32_t)((c ^ ((hx >> 2) & 1)) << 4);
#pragma unroll
        for (int hz = lo; hz < hi; ++hz) {
            const int z = z0 - 1 + hz;
            const bool ok = xyok && z >= 0 && z < d.nz;
            cp_async16(dst + (uint32_t)hz * (kWHx * kWHy * 32), ok ? col + (size_t)(layer * (z >> shift)) * xc : xs, ok);
        }
    };
    auto load_tile = [&](int s) {
        const int x0 = bx * kWTx, y0 = by * kWTy, z0 = bz * kWTz, vb = bb * d.nvox;
        const uint32_t G = smem0 + (uint32_t)s * kWStage, X = G + kWVox * 32;
        for (int i = tid; i < kWVox * 2; i += kWThreads) {
            const int c = i & 1, v = i >> 1;
            const int x = x0 + v % kWTx, y = y0 + (v / kWTx) % kWTy, z = z0 + v / (kWTx * kWTy);
            const bool ok = x < d.nx && y < d.ny && z < d.nz;
            const bf16* src = ok ? a.gp + (size_t)(vb + x + d.nx * (y + d.ny * z)) * a.cout + co0 + 8 * c : a.gp;
            cp_async16(G + v * 32 + ((c ^ ((v >> 2) & 1)) << 4), src, ok);
        }
        load_halo(X, tid, z0, 0, kWHz);
        if (tid < 8 * kWHz) load_halo(X, h2, z0, tid >> 3, (tid >> 3) + 1);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        bx += sx;
        by += sy + (bx >= tx);
        bx -= bx >= tx ? tx : 0;
        bz += sz + (by >= ty);
        by -= by >= ty ? ty : 0;
        bb += sb + (bz >= tz);
        bz -= bz >= tz ? tz : 0;
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

    if (t < a.tiles) load_tile(0);
    for (int s = 0; t < a.tiles; t += gridDim.x, s ^= 1) {
        if (t + (int)gridDim.x < a.tiles) {
            load_tile(s ^ 1);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        const uint32_t G = smem0 + (uint32_t)s * kWStage, X = G + kWVox * 32;
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
            // a tile's sums by themselves: the tensor core's additions do not round to nearest, and a chain of them
            // through all of a block's tiles is off by as many units in the last place
            float part[3][2][4] = {};
#pragma unroll
            for (int z = 0; z < 2; ++z) {
                const uint32_t xb = X + laneB[dx] + (uint32_t)((2 * half + z + dz) * kWHy * (kWHx * 32));
                uint32_t fa[4][4];  // 16 voxels: rows y = 2 j, 2 j + 1
#pragma unroll
                for (int j = 0; j < 4; ++j) ldm_x4_trans(G + laneA + (uint32_t)(((2 * half + z) * kWTy + 2 * j) * kWTx * 32), fa[j]);
                uint32_t lo[4], hi[4];  // halo rows 2 j, 2 j + 1 and the two above
                ldm_x4_trans(xb, lo);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    ldm_x4_trans(xb + (uint32_t)((2 * j + 2) * (kWHx * 32)), hi);
                    const uint32_t b0[2] = {lo[1], hi[0]}, b1[2] = {lo[3], hi[2]};
                    mma16816(part[0][0], fa[j], lo);
                    mma16816(part[0][1], fa[j], lo + 2);
                    mma16816(part[1][0], fa[j], b0);
                    mma16816(part[1][1], fa[j], b1);
                    mma16816(part[2][0], fa[j], hi);
                    mma16816(part[2][1], fa[j], hi + 2);
#pragma unroll
                    for (int i = 0; i < 4; ++i) lo[i] = hi[i];
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[3 * q + dx][i >> 2][i & 3] += part[q][i >> 2][i & 3];
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

// Head (1x1x1 conv 16 -> 3), residual on the ansatz, normalisation.
__global__ void __launch_bounds__(256) head_kernel(const bf16* __restrict__ d1, const float* __restrict__ n_ans,
                                                   const float* __restrict__ params_head, float* __restrict__ n_out, Dims d)
{
    nh::step_kernel_enter();
    constexpr int kW = kHeadOut * kHeadIn;
    __shared__ float sh[kW + kHeadOut];
    for (int k = threadIdx.x; k < kW + kHeadOut; k += blockDim.x) sh[k] = params_head[k];
    __syncthreads();
    const int total = d.nvox * d.batch;
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
#pragma unroll
        for (int o = 0; o < 3; ++o)
            if (n_out) n_out[o0 + (size_t)o * d.nvox] = vv[o] / len;
    }
}

// The head again with the loss mean |n - target|^2, the gradients of W_head and
// b_head, and the last convolution's pre-activation gradient (ReLU mask of d1,
// BF16) and bias gradient.  Two lanes share a voxel, eight channels each, and
// pass on their halves of the three dot products: a lane keeps 36 running sums
// where a thread per voxel kept 68, which held an SM to one block of 164
// registers (58 us at 8 x 64 x 64 x 32 voxels, waiting for memory; now 35 us).
__global__ void __launch_bounds__(256, 2) head_bwd_kernel(const bf16* __restrict__ d1, const float* __restrict__ n_ans,
                                                          const float* __restrict__ params_head,
                                                          const float* __restrict__ target, bf16* __restrict__ gp,
                                                          float* __restrict__ gb, float* __restrict__ g_head,
                                                          float* __restrict__ loss, Dims d)
{
    nh::step_kernel_enter();
    constexpr int kW = kHeadOut * kHeadIn;
    // a lane's sums: W[3][8], bias of its eight channels, b_head[3], loss (of both lanes of a voxel: halved)
    constexpr int kSums = kHeadOut * 8 + 8 + kHeadOut + 1;
    __shared__ float red[2][kSums][8];
    const int half = threadIdx.x & 1;
    float w[kHeadOut][8], b3[kHeadOut];
#pragma unroll
    for (int o = 0; o < kHeadOut; ++o) {
#pragma unroll
        for (int c = 0; c < 8; ++c) w[o][c] = params_head[o * kHeadIn + half * 8 + c];
        b3[o] = params_head[kW + o];
    }
    const int total = d.nvox * d.batch;
    const float inv_total = 1.f / (float)total;
    float sum[kSums];
#pragma unroll
    for (int k = 0; k < kSums; ++k) sum[k] = 0.f;
    const int stride = (gridDim.x * blockDim.x) >> 1;
    // the voxel count (of 16 x 16 x 8 at least, in eights) and the stride are multiples of 16: a warp stays together
    for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 1; v < total; v += stride) {
        const int b = v / d.nvox, r = v - b * d.nvox;
        const size_t o0 = (size_t)b * 3 * d.nvox + r;
        float h[8];
        unpack8(__ldg(reinterpret_cast<const uint4*>(d1 + (size_t)v * kHeadIn) + half), h);
        float vv[3], tg[3];
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            vv[o] = __ldg(n_ans + o0 + (size_t)o * d.nvox);
            tg[o] = __ldg(target + o0 + (size_t)o * d.nvox);
        }
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            // b + the sixteen products one after another, as the forward head adds them: where n_ansatz and the
            // correction nearly cancel, another order would move n
            float s = b3[o];
#pragma unroll
            for (int c = 0; c < 8; ++c) s += w[o][c] * h[c];
            s = __shfl_xor_sync(0xffffffffu, s, 1);  // of the upper lane: the lower one's sum
#pragma unroll
            for (int c = 0; c < 8; ++c) s += w[o][c] * h[c];
            vv[o] += __shfl_sync(0xffffffffu, s, threadIdx.x | 1);
        }
        const float len = sqrtf(vv[0] * vv[0] + vv[1] * vv[1] + vv[2] * vv[2]);
        float gn[3], nn[3], dot = 0.f, l = 0.f;
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            nn[o] = vv[o] / len;
            const float diff = nn[o] - tg[o];
            l += diff * diff;
            gn[o] = 2.f * diff * inv_total;
            dot += gn[o] * nn[o];
        }
        sum[kSums - 1] += l * inv_total;
        float g[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) g[c] = 0.f;
#pragma unroll
        for (int o = 0; o < 3; ++o) {
            const float gd = (gn[o] - dot * nn[o]) / len;  // d/dv of v/|v|
            sum[32 + o] += gd;
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                g[c] += w[o][c] * gd;
                sum[o * 8 + c] += gd * h[c];
            }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            g[c] = h[c] > 0.f ? g[c] : 0.f;
            sum[24 + c] += g[c];
        }
        reinterpret_cast<uint4*>(gp + (size_t)v * kHeadIn)[half] = pack8(g);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kSums; ++k) {
        float s = sum[k];
        for (int o = 16; o > 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane < 2) red[lane][k][warp] = s;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * kSums; i += blockDim.x) {
        const int hh = i / kSums, k = i - hh * kSums;
        if (hh == 1 && k >= 32) continue;  // both lanes have these
        float s = 0.f;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += red[hh][k][q];
        if (k < 24)
            atomicAdd(&g_head[(k >> 3) * kHeadIn + hh * 8 + (k & 7)], s);
        else if (k < 32)
            atomicAdd(&gb[hh * 8 + k - 24], s);
        else if (k < 35)
            atomicAdd(&g_head[kW + k - 32], s);
        else
            atomicAdd(loss, s);
    }
}

__global__ void bf16_to_f32_kernel(const bf16* __restrict__ a, float* __restrict__ out, int64_t n)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __bfloat162float(a[i]);
}

// BF16 weights of all convolutions as the forward pass's and the data gradient's
// images, in one launch (one per layer took 45 us).
struct ParamTable {
    int begin[kLayers + 1];  // first parameter of each layer, and of the head
    int cin[kLayers], cout[kLayers];
    bf16 *w[kLayers], *wt[kLayers];
};
__global__ void params_kernel(const float* __restrict__ p, const ParamTable t)
{
    nh::step_kernel_enter();
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < t.begin[kLayers]; i += gridDim.x * blockDim.x) {
        int l = 0;
        while (i >= t.begin[l + 1]) ++l;
        const int cin = t.cin[l], cout = t.cout[l], k = i - t.begin[l], cc = cin * cout;
        if (k >= 27 * cc) continue;  // bias
        const int tap = k / cc, r = k - tap * cc, co = r / cin, ci = r - co * cin;
        const bf16 v = __float2bfloat16_rn(p[i]);
        t.w[l][tc_weight_index(cout, cin, tap, co, ci)] = v;
        t.wt[l][tc_weight_index(cin, cout, tap, ci, co)] = v;
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
    size_t w[kLayers], wt[kLayers], x, act[kLayers], pool_[3], grad, grad_skip[3], gp[2], status;
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
    for (int l = 0; l < kLayers; ++l) {
        u->w[l] = take(27 * (size_t)kConv[l].cin * kConv[l].cout * sizeof(bf16));
        u->wt[l] = take(27 * (size_t)kConv[l].cin * kConv[l].cout * sizeof(bf16));
    }
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
    a.w = P<bf16>(u, u->w[l]);
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
    static nh::OncePerDevice once;  // the opt-in to more than 48 KB of shared memory
    cudaError_t e = nh::once_per_device(
        once, [] { return cudaFuncSetAttribute(conv_bwd_w_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWSmem); });
    if (e != cudaSuccess) return e;
    // one wave of resident blocks over the channel pairs; each walks its share of the tiles
    const int pairs = (cin / 16) * (cout / 16);
    dim3 grid(std::min(w.tiles, std::max(1, kWBlocksPerSM * 152 / pairs)), pairs);
    nh::launch_step_kernel(conv_bwd_w_kernel, grid, kWThreads, kWSmem, st, w);
    e = cudaGetLastError();
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
    ParamTable t;
    for (int l = 0; l < kLayers; ++l) {
        t.begin[l] = (int)layer_offset(l);
        t.cin[l] = kConv[l].cin;
        t.cout[l] = kConv[l].cout;
        t.w[l] = P<bf16>(u, u->w[l]);
        t.wt[l] = P<bf16>(u, u->wt[l]);
    }
    t.begin[kLayers] = (int)head_offset();
    nh::launch_step_kernel(params_kernel, grid_for(head_offset()), 256, 0, st, params, t);
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
    nh::launch_step_kernel(head_kernel, grid_for((int64_t)d0.nvox * d0.batch), 256, 0, st, act(DEC1B), n_ansatz,
                           params + head_offset(), n_out, d0);
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
    nh::launch_step_kernel(head_bwd_kernel, std::min(2 * 152, grid_for((int64_t)d0.nvox * d0.batch * 2)), 256, 0, st,
                           act(DEC1B), n_ansatz, params + head_offset(), target, gpa, gbias(DEC1B),
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
