// Learned warm start for the Poisson solve: a 3D convolutional network
// (3^3 kernels, channels 2 -> 16 -> 16 -> 16 -> 1, ReLU between layers,
// linear output) mapping the step's change of the Poisson source and the
// previous potential to the change of the potential.  The solver then runs to
// its usual residual from the improved start, so only iterations are saved.
//
// Layout: activations node-major, 16 channels contiguous (NDHWC) in BF16;
// parameters as one FP32 vector, per layer W[co][ci][k] then b[co] with
// k = (dz+1)*9 + (dy+1)*3 + (dx+1); periodic wrap on periodic axes, zeros
// beyond closed ones.
//
// The two 16 -> 16 layers (about 93 % of the arithmetic) are implicit GEMMs
// on the tensor cores, K = 27 offsets x 16 input channels, BF16 operands,
// FP32 accumulation: by default on tcgen05 (128 nodes per block, the
// accumulator in tensor memory, operands staged in shared memory), or with
// the warp-level mma.sync m16n8k16 (16 nodes per warp); the data gradient of
// those layers is the same kernel with flipped offsets and transposed
// channels.  The 2 -> 16 and 16 -> 1 layers, the weight
// gradients (per-block partial sums reduced in a fixed order) and Adam run on
// the CUDA cores in FP32.
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <memory>
#include <type_traits>
#include <vector>

#include <new>
#include <utility>

#include "ekl_kernels.cuh"

struct ekl_handle {
    ekl::Ctx c;
};

namespace {

using namespace ekl;

constexpr int K27 = 27;
constexpr int NT = 256;   // threads per block of the CUDA-core kernels
// parameter offsets
constexpr int OW1 = 0, OB1 = OW1 + 16 * 2 * 27, OW2 = OB1 + 16, OB2 = OW2 + 16 * 16 * 27,
              OW3 = OB2 + 16, OB3 = OW3 + 16 * 16 * 27, OW4 = OB3 + 16, OB4 = OW4 + 16 * 27,
              NPARAM = OB4 + 1;
static_assert(NPARAM == EKL_NET_PARAMS, "parameter count");

struct NetGrid {
    int nx, ny, nz;
    int per[3];
    int N;      // nodes of one sample
    int total;  // nodes of all samples of the pass (ns N): node n belongs to sample n / N
};

// neighbour of node (x,y,z) at offset k; -1 beyond a closed face
__device__ __forceinline__ int nbr_off(const NetGrid &g, int x, int y, int z, int k)
{
    int dx = k % 3 - 1, dy = (k / 3) % 3 - 1, dz = k / 9 - 1;
    int X = x + dx, Y = y + dy, Z = z + dz;
    if (X < 0 || X >= g.nx) {
        if (!g.per[0]) return -1;
        X = X < 0 ? X + g.nx : X - g.nx;
    }
    if (Y < 0 || Y >= g.ny) {
        if (!g.per[1]) return -1;
        Y = Y < 0 ? Y + g.ny : Y - g.ny;
    }
    if (Z < 0 || Z >= g.nz) {
        if (!g.per[2]) return -1;
        Z = Z < 0 ? Z + g.nz : Z - g.nz;
    }
    return X + g.nx * (Y + g.ny * Z);
}

__device__ __forceinline__ void xyz_of(const NetGrid &g, int n, int &x, int &y, int &z)
{
    int r = n / g.nx;
    x = n - r * g.nx;
    z = r / g.ny;
    y = r - z * g.ny;
}

// coordinates of node n of a pass over several samples; returns the first
// node of its sample
__device__ __forceinline__ int sample_xyz(const NetGrid &g, int n, int &x, int &y, int &z)
{
    const int base = (n / g.N) * g.N;
    xyz_of(g, n - base, x, y, z);
    return base;
}

// Network input of the samples of a pass: sample s is x + 2 N smp[s] (smp
// null: the samples in order), two channels of N nodes.
struct NetInput {
    const float *x;
    const int *smp;
};
__device__ __forceinline__ const float *sample_x(const NetGrid &g, const NetInput &in, int s)
{
    return in.x + 2 * (size_t)g.N * (in.smp ? in.smp[s] : s);
}

// ---------------------------------------------------------------- layer 1
// act1[n][co] = relu(b1[co] + sum_k sum_ci W1[co][ci][k] x[ci][n + off_k])
__global__ void __launch_bounds__(NT) l1_fwd(NetGrid g, NetInput in, const float *__restrict__ w,
                                             __nv_bfloat16 *__restrict__ act)
{
    // weights as [offset and channel][16 outputs]: one 16-byte load per four outputs
    __shared__ __align__(16) float sw[16 * 2 * 27 + 16];
    for (int t = threadIdx.x; t < 16 * 54; t += blockDim.x) {
        const int c = t / 54, r = t - 54 * c, ci = r / 27, k = r - 27 * ci;
        sw[(2 * k + ci) * 16 + c] = w[OW1 + t];
    }
    if (threadIdx.x < 16) sw[16 * 54 + threadIdx.x] = w[OB1 + threadIdx.x];
    __syncthreads();
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= g.total) return;
    int X, Y, Z;
    const float *x = sample_x(g, in, sample_xyz(g, n, X, Y, Z) / g.N);
    float acc[16];
#pragma unroll
    for (int c = 0; c < 16; c++) acc[c] = sw[16 * 54 + c];
#pragma unroll 3
    for (int k = 0; k < K27; k++) {
        const int j = nbr_off(g, X, Y, Z, k);
        if (j < 0) continue;
        const float x0 = x[j], x1 = x[g.N + j];
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
            const float4 w0 = *(const float4 *)(sw + 32 * k + c), w1 = *(const float4 *)(sw + 32 * k + 16 + c);
            acc[c] += w0.x * x0 + w1.x * x1;
            acc[c + 1] += w0.y * x0 + w1.y * x1;
            acc[c + 2] += w0.z * x0 + w1.z * x1;
            acc[c + 3] += w0.w * x0 + w1.w * x1;
        }
    }
    for (int c = 0; c < 16; c += 2) {
        __nv_bfloat162 v = __floats2bfloat162_rn(fmaxf(acc[c], 0.f), fmaxf(acc[c + 1], 0.f));
        *(__nv_bfloat162 *)(act + (size_t)n * 16 + c) = v;
    }
}

// ---------------------------------------------------------------- 16 -> 16 on tensor cores
__device__ __forceinline__ void mma_bf16(float d[4], const uint32_t a[4], const uint32_t b[2])
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// out[n][co] = act?(bias[co] + sum_k sum_ci Wt[k][co][ci] in[n + off_k][ci]); flip = use -off_k.
// Wt is BF16 [27][16 co][16 ci] (ci contiguous).  One warp: 16 consecutive nodes.
template <bool RELU, bool OUT_F32>
__global__ void __launch_bounds__(256) conv16_mma(NetGrid g, const __nv_bfloat16 *__restrict__ in,
                                                  const __nv_bfloat16 *__restrict__ Wt,
                                                  const float *__restrict__ bias, int flip, void *out,
                                                  const __nv_bfloat16 *__restrict__ relu_mask_src)
{
    __shared__ uint32_t sW[27 * 16 * 8];  // [k][co][ci pair]
    for (int t = threadIdx.x; t < 27 * 16 * 8; t += blockDim.x) sW[t] = ((const uint32_t *)Wt)[t];
    __syncthreads();
    const int lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
    const int warp_global = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int n0 = warp_global * 16;
    if (n0 >= g.total) return;
    const int na = n0 + gid, nb = n0 + gid + 8;
    int xa, ya, za, xb, yb, zb;
    const int basea = sample_xyz(g, na < g.total ? na : 0, xa, ya, za);
    const int baseb = sample_xyz(g, nb < g.total ? nb : 0, xb, yb, zb);
    float d[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    const uint32_t *in32 = (const uint32_t *)in;
    for (int k = 0; k < K27; k++) {
        const int kk = flip ? 26 - k : k;
        const int ja = na < g.total ? nbr_off(g, xa, ya, za, kk) : -1;
        const int jb = nb < g.total ? nbr_off(g, xb, yb, zb, kk) : -1;
        const uint32_t *pa = in32 + (size_t)(basea + ja) * 8, *pb = in32 + (size_t)(baseb + jb) * 8;
        uint32_t a[4];
        a[0] = ja >= 0 ? pa[tig] : 0u;
        a[1] = jb >= 0 ? pb[tig] : 0u;
        a[2] = ja >= 0 ? pa[tig + 4] : 0u;
        a[3] = jb >= 0 ? pb[tig + 4] : 0u;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int co = h * 8 + gid;
            uint32_t b[2] = {sW[(k * 16 + co) * 8 + tig], sW[(k * 16 + co) * 8 + tig + 4]};
            mma_bf16(d[h], a, b);
        }
    }
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int co = h * 8 + 2 * tig;
        float v[4] = {d[h][0], d[h][1], d[h][2], d[h][3]};
        if (bias) {
            v[0] += bias[co];
            v[1] += bias[co + 1];
            v[2] += bias[co];
            v[3] += bias[co + 1];
        }
        if (RELU)
            for (int q = 0; q < 4; q++) v[q] = fmaxf(v[q], 0.f);
        // gradient through the ReLU of the layer that produced `relu_mask_src`
        if (relu_mask_src) {
            if (na < g.total) {
                if (!(__bfloat162float(relu_mask_src[(size_t)na * 16 + co]) > 0.f)) v[0] = 0.f;
                if (!(__bfloat162float(relu_mask_src[(size_t)na * 16 + co + 1]) > 0.f)) v[1] = 0.f;
            }
            if (nb < g.total) {
                if (!(__bfloat162float(relu_mask_src[(size_t)nb * 16 + co]) > 0.f)) v[2] = 0.f;
                if (!(__bfloat162float(relu_mask_src[(size_t)nb * 16 + co + 1]) > 0.f)) v[3] = 0.f;
            }
        }
        if (OUT_F32) {
            float *o = (float *)out;
            if (na < g.total) { o[(size_t)na * 16 + co] = v[0]; o[(size_t)na * 16 + co + 1] = v[1]; }
            if (nb < g.total) { o[(size_t)nb * 16 + co] = v[2]; o[(size_t)nb * 16 + co + 1] = v[3]; }
        } else {
            __nv_bfloat16 *o = (__nv_bfloat16 *)out;
            if (na < g.total) *(__nv_bfloat162 *)(o + (size_t)na * 16 + co) = __floats2bfloat162_rn(v[0], v[1]);
            if (nb < g.total) *(__nv_bfloat162 *)(o + (size_t)nb * 16 + co) = __floats2bfloat162_rn(v[2], v[3]);
        }
    }
}

// ---------------------------------------------------------------- tiles
// The layers that read hidden activations work on tiles of tx x ty nodes and
// TL_Z planes, staged with a one-node halo in shared memory as one list of
// rows (x fastest, then y, then z; W = tx + 2 rows per line, H = ty + 2 lines
// per plane; zero rows beyond closed faces).  In that list the neighbour at
// offset (dx, dy, dz) of row p is row p + dx + W dy + W H dz for every p, so
// a layer's 27 shifted operands are the same rows from 27 starting points.  A
// plane's outputs are the TC_M rows from its first node on; tx and ty are
// chosen so that these hold all of them (rows that fall on the halo are
// computed and dropped).  The eight channels of each half of a row have
// their own plane of 16-byte rows.
constexpr int TC_M = 128;
constexpr int TL_Z = 2;
constexpr int TL_T = 256;   // threads of a block: one per output row of the planes
constexpr int TL_U = 4;     // rows a thread has in flight while staging
struct NetTile {
    int tx, ty, W, H;       // nodes per tile along x and y, padded extents
    int ntx, nty, ntz;      // tiles per sample
    int rows;               // staged rows, with the slack the last plane's shifted operands reach
};
__host__ inline int split_even(int n, int most) { return (n + (n + most - 1) / most - 1) / ((n + most - 1) / most); }
__host__ inline NetTile make_tile(const NetGrid &g)
{
    NetTile T;
    T.tx = split_even(g.nx, 30);
    T.W = T.tx + 2;
    T.ty = split_even(g.ny, (TC_M - T.tx) / T.W + 1);
    T.H = T.ty + 2;
    T.ntx = (g.nx + T.tx - 1) / T.tx;
    T.nty = (g.ny + T.ty - 1) / T.ty;
    T.ntz = (g.nz + TL_Z - 1) / TL_Z;
    T.rows = T.W * T.H * (TL_Z + 2) + TC_M;
    return T;
}
struct TilePos {
    int x0, y0, z0, base;   // first node of the tile and of its sample
};
__device__ __forceinline__ TilePos tile_pos(const NetGrid &g, const NetTile &T, int blk)
{
    TilePos P;
    int t = blk / T.ntx;
    P.x0 = (blk - t * T.ntx) * T.tx;
    int u = t / T.nty;
    P.y0 = (t - u * T.nty) * T.ty;
    const int s = u / T.ntz;
    P.z0 = (u - s * T.ntz) * TL_Z;
    P.base = s * g.N;
    return P;
}
// rows of the tile and its halo into sA (two planes of T.rows 16-byte rows);
// the slack rows are zeroed
__device__ __forceinline__ void tile_stage(const NetGrid &g, const NetTile &T, const TilePos &P,
                                           const __nv_bfloat16 *__restrict__ in, uint4 *sA)
{
    const int WH = T.W * T.H, real = WH * (TL_Z + 2);
    for (int p0 = threadIdx.x; p0 < T.rows; p0 += TL_U * TL_T) {
        uint4 v[TL_U][2];
#pragma unroll
        for (int u = 0; u < TL_U; u++) {
            const int p = p0 + u * TL_T;
            v[u][0] = v[u][1] = make_uint4(0u, 0u, 0u, 0u);
            if (p >= real) continue;
            const int lz = p / WH, r = p - lz * WH, ly = r / T.W, lx = r - ly * T.W;
            int X = P.x0 + lx - 1, Y = P.y0 + ly - 1, Z = P.z0 + lz - 1;
            // rows past a ragged tile's last neighbour are never used
            bool ok = X <= g.nx && Y <= g.ny && Z <= g.nz;
            if (X < 0 || X >= g.nx) {
                ok = ok && g.per[0];
                X = X < 0 ? X + g.nx : X - g.nx;
            }
            if (Y < 0 || Y >= g.ny) {
                ok = ok && g.per[1];
                Y = Y < 0 ? Y + g.ny : Y - g.ny;
            }
            if (Z < 0 || Z >= g.nz) {
                ok = ok && g.per[2];
                Z = Z < 0 ? Z + g.nz : Z - g.nz;
            }
            if (ok) {
                const uint4 *src = (const uint4 *)(in + (size_t)(P.base + X + g.nx * (Y + g.ny * Z)) * 16);
                v[u][0] = __ldg(src);
                v[u][1] = __ldg(src + 1);
            }
        }
#pragma unroll
        for (int u = 0; u < TL_U; u++) {
            const int p = p0 + u * TL_T;
            if (p >= T.rows) continue;
            sA[p] = v[u][0];
            sA[T.rows + p] = v[u][1];
        }
    }
}
// node of output row r (0 .. TC_M - 1) of the tile's plane lz, -1 on halo rows and past the grid
__device__ __forceinline__ int tile_node(const NetGrid &g, const NetTile &T, const TilePos &P, int r, int lz)
{
    const int q = r + 1, ly = q / T.W, lx = q - ly * T.W - 1;  // row r is (lx, ly) + the first node
    const int X = P.x0 + lx, Y = P.y0 + ly, Z = P.z0 + lz;
    if (lx < 0 || lx >= T.tx || ly >= T.ty || X >= g.nx || Y >= g.ny || Z >= g.nz) return -1;
    return P.base + X + g.nx * (Y + g.ny * Z);
}

// ---------------------------------------------------------------- 16 -> 16 on tcgen05
// The same layer as an implicit GEMM on the fifth-generation tensor cores:
// per plane of a tile M = 128 rows, N = 16 output channels, and K = 27 offsets
// x 16 input channels as 27 MMAs of K = 16 (one per offset), BF16 operands
// from shared memory, FP32 accumulation in tensor memory.
//   * A (per offset): the tile's rows from the plane's first node plus the
//     offset's shift, K-major without swizzle: core matrices of 8 rows x 16
//     bytes are 128 contiguous bytes (SBO), the K-halves lie a plane apart
//     (LBO), and the start address (16-byte units) carries the shift, so no
//     operand is staged twice;
//   * B (per offset): W[co][ci], 16 x 16 BF16, row-group g and K-half h at
//     byte g * 256 + h * 128;
//   * D: TMEM lanes = rows, 16 columns per plane; warp w reads lanes
//     32w..32w+31 back with tcgen05.ld (32x32b, 16 columns).
// One thread issues the MMAs of all planes and commits them to an mbarrier;
// the wait is bounded (on giving up the block raises tc_status and skips the
// epilogue), and the block frees its tensor memory on every path.
// What bounds it: staging.  With a copy of the rows per offset (27 x 4 KB a
// block, one block per SM) a 65 536-node layer took 45 us, now 11 us.
constexpr int TC_B_BYTES = 16 * 32;             // one offset's B tile
constexpr int TC_COLS = TL_Z * 16;              // TMEM columns (a power of two, at least 32)

__device__ int tc_status;  // nonzero after a bounded wait gave up

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: no swizzle, K-major core matrices
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// instruction descriptor: D FP32, A and B BF16, both K-major, N = 16, M = 128
constexpr uint32_t TC_IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((16u >> 3) << 17) | ((128u >> 4) << 24);

// byte offset of element (row, k) (k < 16) in a no-swizzle K-major tile
__device__ __forceinline__ int tc_off(int row, int k) { return (row >> 3) * 256 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2; }

// wait (bounded, about a second at most) for phase 0 of the mbarrier
__device__ __forceinline__ uint32_t tc_wait(uint64_t *mbar)
{
    uint32_t done = 0;
    for (int it = 0; it < (1 << 20) && !done; it++) {
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_u32(mbar)));
    }
    return done;
}

// at most 42 560 bytes (tiles of 30 x 4 nodes): with the kernels' static shared
// memory still within the 48 KB of any launch
inline size_t tc_smem(const NetTile &T) { return (size_t)T.rows * 32 + K27 * TC_B_BYTES + 64; }

template <bool RELU>
__global__ void __launch_bounds__(TL_T) conv16_tc(NetGrid g, NetTile T, const __nv_bfloat16 *__restrict__ in,
                                                  const __nv_bfloat16 *__restrict__ Wt,
                                                  const float *__restrict__ bias, int flip,
                                                  __nv_bfloat16 *__restrict__ out,
                                                  const __nv_bfloat16 *__restrict__ relu_mask_src)
{
    extern __shared__ __align__(1024) uint8_t tc_sm[];
    uint8_t *sB = tc_sm;                              // [27][TC_B_BYTES]
    uint64_t *mbar = (uint64_t *)(sB + K27 * TC_B_BYTES);
    uint32_t *tmem_slot = (uint32_t *)(mbar + 1);
    uint4 *sA = (uint4 *)(sB + K27 * TC_B_BYTES + 64);  // [2][T.rows]
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "n"(TC_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(mbar)));
    }
    for (int t = tid; t < K27 * 16 * 2; t += TL_T) {
        const int k = t >> 5, co = (t >> 1) & 15, h = t & 1;
        const uint4 v = *(const uint4 *)(Wt + ((size_t)k * 16 + co) * 16 + 8 * h);
        *(uint4 *)(sB + k * TC_B_BYTES + tc_off(co, 8 * h)) = v;
    }
    const TilePos P = tile_pos(g, T, blockIdx.x);
    tile_stage(g, T, P, in, sA);
    // make the generic-proxy writes visible to the tensor cores' async proxy
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    if (tid == 0) {
        const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
        const int WH = T.W * T.H;
        for (int z = 0; z < TL_Z; z++) {
            const int first = 1 + T.W + WH * (z + 1);  // the plane's first node
            for (int k = 0; k < K27; k++) {
                const int kk = flip ? 26 - k : k;
                const int row = first + (kk % 3 - 1) + T.W * ((kk / 3) % 3 - 1) + WH * (kk / 9 - 1);
                const uint64_t ad = tc_desc(a0 + 16u * (uint32_t)row, 16u * (uint32_t)T.rows, 128);
                const uint64_t bd = tc_desc(b0 + k * TC_B_BYTES, 128, 256);
                const uint32_t acc = k > 0;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + 16u * (uint32_t)z),
                    "l"(ad), "l"(bd), "r"(TC_IDESC), "r"(acc));
            }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
            smem_u32(mbar)));
    }
    // bounded wait for the MMAs (phase 0 of the mbarrier)
    uint32_t done = tc_wait(mbar);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (!done) {
        // give up: raise the status, wait once more (bounded) for the MMAs
        // still in flight, then free the tensor memory below
        if (lane == 0) atomicExch(&tc_status, 1);
        done = tc_wait(mbar);
    } else {
        // warps 0-3 read the first plane's columns, warps 4-7 the second's
        // (a warp reaches the 32 lanes of its number modulo 4)
        static_assert(TL_T == TL_Z * TC_M, "one warp group per plane");
        const int z = warp >> 2;
        uint32_t d[16];
        const uint32_t taddr = tmem + 16u * (uint32_t)z + ((uint32_t)((warp & 3) * 32) << 16);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
            "%14, %15}, [%16];\n"
            : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3]), "=r"(d[4]), "=r"(d[5]), "=r"(d[6]), "=r"(d[7]),
              "=r"(d[8]), "=r"(d[9]), "=r"(d[10]), "=r"(d[11]), "=r"(d[12]), "=r"(d[13]), "=r"(d[14]), "=r"(d[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        const int n = tile_node(g, T, P, tid & (TC_M - 1), z);
        if (n >= 0) {
            uint4 m[2];
            if (relu_mask_src) {
                m[0] = __ldg((const uint4 *)(relu_mask_src + (size_t)n * 16));
                m[1] = __ldg((const uint4 *)(relu_mask_src + (size_t)n * 16) + 1);
            }
            const __nv_bfloat16 *mv = (const __nv_bfloat16 *)m;
            float v[16];
#pragma unroll
            for (int co = 0; co < 16; co++) {
                v[co] = __uint_as_float(d[co]) + (bias ? bias[co] : 0.f);
                if (RELU) v[co] = fmaxf(v[co], 0.f);
                // gradient through the ReLU of the layer that produced relu_mask_src
                if (relu_mask_src && !(__bfloat162float(mv[co]) > 0.f)) v[co] = 0.f;
            }
            __align__(16) __nv_bfloat162 o[8];
#pragma unroll
            for (int c = 0; c < 8; c++) o[c] = __floats2bfloat162_rn(v[2 * c], v[2 * c + 1]);
            uint4 *dst = (uint4 *)(out + (size_t)n * 16);
            dst[0] = ((const uint4 *)o)[0];
            dst[1] = ((const uint4 *)o)[1];
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "n"(TC_COLS));
}

// which kernel runs the 16 -> 16 layers: 1 = tcgen05 (default), 0 = mma.sync
int g_tensor_path = 1;

template <bool RELU>
void conv16(const NetGrid &g, const __nv_bfloat16 *in, const __nv_bfloat16 *Wt, const float *bias, int flip,
            __nv_bfloat16 *out, const __nv_bfloat16 *relu_mask_src, cudaStream_t s)
{
    if (g_tensor_path) {
        const NetTile T = make_tile(g);
        const int blocks = T.ntx * T.nty * T.ntz * (g.total / g.N);
        conv16_tc<RELU><<<blocks, TL_T, tc_smem(T), s>>>(g, T, in, Wt, bias, flip, out, relu_mask_src);
    } else {
        conv16_mma<RELU, false><<<(g.total + 127) / 128, 256, 0, s>>>(g, in, Wt, bias, flip, out, relu_mask_src);
    }
}

// BF16 B-operand tables of the two 16->16 layers: forward Wt[k][co][ci] =
// W[co][ci][k]; data gradient Wb[k][ci][co] = W[co][ci][k] (used with flipped
// offsets).
__global__ void prep_w16(const float *__restrict__ w, __nv_bfloat16 *__restrict__ W2f, __nv_bfloat16 *__restrict__ W2b,
                         __nv_bfloat16 *__restrict__ W3f, __nv_bfloat16 *__restrict__ W3b)
{
    int t = blockIdx.x * blockDim.x + threadIdx.x;
    const bool third = t >= 27 * 256;
    if (third) t -= 27 * 256;
    if (t >= 27 * 256) return;
    const int k = t / 256, r = t % 256, co = r / 16, ci = r % 16;
    const __nv_bfloat16 v = __float2bfloat16_rn(w[(third ? OW3 : OW2) + (co * 16 + ci) * 27 + k]);
    (third ? W3f : W2f)[(k * 16 + co) * 16 + ci] = v;
    (third ? W3b : W2b)[(k * 16 + ci) * 16 + co] = v;
}

// ---------------------------------------------------------------- layer 4
// y[n] = b4 + sum_k sum_ci W4[ci][k] act[n + off_k][ci] in FP32, one thread
// per row of a staged tile's plane (27 row reads of 32 bytes each: from
// shared memory, not from L1 with the neighbours' indices worked out per
// offset: 11 us for 65 536 nodes against 23)
__global__ void __launch_bounds__(TL_T) l4_fwd(NetGrid g, NetTile T, const __nv_bfloat16 *__restrict__ act,
                                               const float *__restrict__ w, float *__restrict__ y)
{
    extern __shared__ __align__(1024) uint8_t tc_sm[];
    float *sw = (float *)tc_sm;                              // [offset][channel], then the bias
    uint4 *sA = (uint4 *)(tc_sm + K27 * TC_B_BYTES + 64);    // as in conv16_tc
    int finite = 1;
    for (int t = threadIdx.x; t < 16 * 27; t += blockDim.x) {
        const float v = w[OW4 + t];
        sw[(t % 27) * 16 + t / 27] = v;
        finite &= isfinite(v);
    }
    if (threadIdx.x == 0) sw[16 * 27] = w[OB4];
    const TilePos P = tile_pos(g, T, blockIdx.x);
    tile_stage(g, T, P, act, sA);
    finite = __syncthreads_and(finite);
    const int WH = T.W * T.H;
    const int z = threadIdx.x / TC_M, r = threadIdx.x & (TC_M - 1);
    const int n = tile_node(g, T, P, r, z);
    if (n < 0) return;
    const int first = 1 + T.W + WH * (z + 1) + r;
    auto add = [&](float &acc, int k) {
        const int row = first + (k % 3 - 1) + T.W * ((k / 3) % 3 - 1) + WH * (k / 9 - 1);
        const uint4 v[2] = {sA[row], sA[T.rows + row]};
        const __nv_bfloat162 *a = (const __nv_bfloat162 *)v;
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const float2 f = __bfloat1622float2(a[c]);
            acc += sw[16 * k + 2 * c] * f.x + sw[16 * k + 2 * c + 1] * f.y;
        }
    };
    float acc = sw[16 * 27];
    if (finite) {
#pragma unroll 3
        for (int k = 0; k < K27; k++) add(acc, k);
    } else {
        // zero rows beyond closed faces times a weight that has overflowed
        // would be NaN: only neighbours on the grid take part
        int X, Y, Z;
        xyz_of(g, n - P.base, X, Y, Z);
#pragma unroll 1
        for (int k = 0; k < K27; k++)
            if (nbr_off(g, X, Y, Z, k) >= 0) add(acc, k);
    }
    y[n] = acc;
}

// loss gradient g = 2 (y - t) / cnt on masked nodes (target of sample s:
// t + N smp[s]); per-block loss partials
__global__ void __launch_bounds__(NT) loss_grad_k(NetGrid gr, const float *y, const float *t, const int *smp,
                                                  const uint8_t *mask, float inv_cnt, float *g, double *part)
{
    __shared__ double sh[NT / 32];
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    float l = 0.f;
    if (n < gr.total) {
        const int s = n / gr.N, i = n - s * gr.N;
        float d = (mask == nullptr || mask[i]) ? y[n] - t[(size_t)gr.N * (smp ? smp[s] : s) + i] : 0.f;
        g[n] = 2.f * d * inv_cnt;
        l = d * d;
    }
    double s = block_sum((double)l, sh);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// loss[0] (+)= scale * (sum of the block partials, in a fixed order)
__global__ void __launch_bounds__(NT) loss_sum_k(const double *part, int n, double scale, int add, double *loss)
{
    __shared__ double sh[NT / 32];
    double v = 0.0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) v += part[k];
    const double t = block_sum(v, sh);
    if (threadIdx.x == 0) *loss = (add ? *loss : 0.0) + scale * t;
}

// d_act3[m][ci] = relu'(act3) * sum_k W4[ci][k] g[m - off_k]  (BF16 out)
__global__ void __launch_bounds__(NT) l4_bwd_data(NetGrid g, const float *__restrict__ gy, const float *__restrict__ w,
                                                  const __nv_bfloat16 *__restrict__ act3, __nv_bfloat16 *__restrict__ dz)
{
    __shared__ __align__(16) float sw[16 * 27];  // [offset][channel]
    for (int t = threadIdx.x; t < 16 * 27; t += blockDim.x) sw[(t % 27) * 16 + t / 27] = w[OW4 + t];
    __syncthreads();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= g.total) return;
    int X, Y, Z;
    const int base = sample_xyz(g, m, X, Y, Z);
    float acc[16];
#pragma unroll
    for (int c = 0; c < 16; c++) acc[c] = 0.f;
#pragma unroll 3
    for (int k = 0; k < K27; k++) {
        const int j = nbr_off(g, X, Y, Z, 26 - k);  // m - off_k
        if (j < 0) continue;
        const float gv = gy[base + j];
#pragma unroll
        for (int c = 0; c < 16; c += 4) {
            const float4 w4 = *(const float4 *)(sw + 16 * k + c);
            acc[c] += w4.x * gv;
            acc[c + 1] += w4.y * gv;
            acc[c + 2] += w4.z * gv;
            acc[c + 3] += w4.w * gv;
        }
    }
    for (int c = 0; c < 16; c += 2) {
        float v0 = __bfloat162float(act3[(size_t)m * 16 + c]) > 0.f ? acc[c] : 0.f;
        float v1 = __bfloat162float(act3[(size_t)m * 16 + c + 1]) > 0.f ? acc[c + 1] : 0.f;
        *(__nv_bfloat162 *)(dz + (size_t)m * 16 + c) = __floats2bfloat162_rn(v0, v1);
    }
}

// ---------------------------------------------------------------- weight gradients
// dW[co][ci][k] = sum_n dz[n][co] a[ci][n + off_k], db[co] = sum_n dz[n][co],
// with a BF16 node-major [n][16] (CI = 16) or the FP32 network input (CI = 2),
// dz BF16 [n][16] (CO = 16) or FP32 [n] (CO = 1).  FP32 sums in a fixed
// order: WG_CH consecutive nodes of a sample in one FMA chain, the chains of
// a block's WG_NODES nodes added in order, one partial per block, the
// partials of a sample added in order (grad_reduce), then the samples.
//
// A block stages the 27 neighbour rows of WG_CH nodes as FP32 in shared
// memory (16 bytes of BF16 channels per load, the next chunk's loads in
// flight under this chunk's arithmetic), and a thread keeps 4 x 4 outputs (4
// output by 4 input channels of one offset), so two 16-byte shared loads feed
// 16 FMAs.  What bounds it: latency, the chain of a block's 32 chunks (staging,
// barrier, arithmetic) with one block of 14 warps on an SM.  Eight samples of
// 8192 nodes are 128 blocks and take 66 us for a 16 -> 16 layer (issue slots 51 %
// busy, FMA pipe 28 %; its 6928 FMAs a node alone would take 11 us), 45 us for the
// last layer and 47 us for the first; fewer samples take no less.  The form before
// gathered one value per thread with its index arithmetic and two scalar shared
// loads per FMA: 710 us per 16 -> 16 layer and sample.
constexpr int WG_CH = 16;
constexpr int WG_NODES = 512;
constexpr int WG_T = 448;

template <int CI, int CO> constexpr int wg_smem() { return 2 * WG_CH * (27 * CI + CO) * (int)sizeof(float); }

template <int CI, int CO>
__global__ void __launch_bounds__(WG_T) wgrad_k(NetGrid g, NetInput in, const __nv_bfloat16 *__restrict__ a,
                                                const void *__restrict__ dz, float *__restrict__ part)
{
    constexpr int NW = CO * CI * 27 + CO;
    constexpr int VC = CI == 16 ? 8 : 1;                 // channels per staged load
    constexpr int PER = 27 * CI / VC;                    // loads per node (54)
    constexpr int LOADS = (WG_CH * PER + WG_T - 1) / WG_T;
    constexpr int TI = CI == 16 ? 4 : 1, TO = CO == 16 ? 4 : 1;  // outputs per thread
    constexpr int JI = 27 * CI / TI, JO = CO / TO;       // thread grid
    static_assert(JI * JO + CO <= WG_T, "threads");
    // double-buffered chunks (57 KB for a 16 -> 16 layer: dynamic)
    extern __shared__ __align__(1024) uint8_t tc_sm[];
    float(*sa)[WG_CH][27 * CI] = (float(*)[WG_CH][27 * CI])tc_sm;
    float(*sd)[WG_CH][CO] = (float(*)[WG_CH][CO])(tc_sm + 2 * sizeof(float) * WG_CH * 27 * CI);
    const int per_sample = (g.N + WG_NODES - 1) / WG_NODES;
    const int s = blockIdx.x / per_sample, base = (blockIdx.x - s * per_sample) * WG_NODES;
    const float *x = CI == 16 ? nullptr : sample_x(g, in, s);
    const int tid = threadIdx.x;
    // this thread's staged loads: node nn of the chunk, offset k, channels
    int nn_[LOADS], k_[LOADS], c_[LOADS];
#pragma unroll
    for (int l = 0; l < LOADS; l++) {
        const int it = tid + l * WG_T;
        nn_[l] = it < WG_CH * PER ? it / PER : -1;
        const int r = it - (it / PER) * PER;
        k_[l] = CI == 16 ? r >> 1 : r % 27;
        c_[l] = CI == 16 ? 8 * (r & 1) : r / 27;
    }
    uint4 va[LOADS];
    float vx[LOADS], vd1 = 0.f;
    uint4 vd = make_uint4(0u, 0u, 0u, 0u);
    auto load = [&](int chunk) {
#pragma unroll
        for (int l = 0; l < LOADS; l++) {
            va[l] = make_uint4(0u, 0u, 0u, 0u);
            vx[l] = 0.f;
            const int n = base + chunk + nn_[l];
            if (nn_[l] < 0 || n >= g.N) continue;
            int X, Y, Z;
            xyz_of(g, n, X, Y, Z);
            const int j = nbr_off(g, X, Y, Z, k_[l]);
            if (j < 0) continue;
            if constexpr (CI == 16)
                va[l] = __ldg((const uint4 *)(a + ((size_t)s * g.N + j) * 16 + c_[l]));
            else
                vx[l] = __ldg(x + (size_t)c_[l] * g.N + j);
        }
        if (tid < WG_CH * (CO == 16 ? 2 : 1)) {
            const int n = base + chunk + (CO == 16 ? tid >> 1 : tid);
            vd = make_uint4(0u, 0u, 0u, 0u);
            vd1 = 0.f;
            if (n < g.N) {
                if constexpr (CO == 16)
                    vd = __ldg((const uint4 *)((const __nv_bfloat16 *)dz + ((size_t)s * g.N + n) * 16 + 8 * (tid & 1)));
                else
                    vd1 = __ldg((const float *)dz + (size_t)s * g.N + n);
            }
        }
    };
    auto unpack = [](const uint4 &v, float *dst) {
        const __nv_bfloat162 *p = (const __nv_bfloat162 *)&v;
        const float2 f0 = __bfloat1622float2(p[0]), f1 = __bfloat1622float2(p[1]), f2 = __bfloat1622float2(p[2]),
                     f3 = __bfloat1622float2(p[3]);
        ((float4 *)dst)[0] = make_float4(f0.x, f0.y, f1.x, f1.y);
        ((float4 *)dst)[1] = make_float4(f2.x, f2.y, f3.x, f3.y);
    };
    auto store = [&](int buf) {
#pragma unroll
        for (int l = 0; l < LOADS; l++) {
            if (nn_[l] < 0) continue;
            float *dst = &sa[buf][nn_[l]][k_[l] * CI + c_[l]];
            if constexpr (CI == 16) unpack(va[l], dst);
            else *dst = vx[l];
        }
        if constexpr (CO == 16) {
            if (tid < 2 * WG_CH) unpack(vd, &sd[buf][tid >> 1][8 * (tid & 1)]);
        } else {
            if (tid < WG_CH) sd[buf][tid][0] = vd1;
        }
    };
    const int ji = tid % JI, jo = tid / JI;
    const bool mine = tid < JI * JO, bias = tid >= JI * JO && tid < JI * JO + CO;
    float acc[TO][TI], accb = 0.f;
#pragma unroll
    for (int o = 0; o < TO; o++)
#pragma unroll
        for (int i = 0; i < TI; i++) acc[o][i] = 0.f;
    load(0);
    store(0);
    __syncthreads();
    const int nodes = min(WG_NODES, g.N - base);
    int buf = 0;
    for (int chunk = 0; chunk < nodes; chunk += WG_CH, buf ^= 1) {
        const bool more = chunk + WG_CH < nodes;
        if (more) load(chunk + WG_CH);
        if (mine) {
            float t[TO][TI];
#pragma unroll
            for (int o = 0; o < TO; o++)
#pragma unroll
                for (int i = 0; i < TI; i++) t[o][i] = 0.f;
#pragma unroll
            for (int nn = 0; nn < WG_CH; nn++) {
                float av[TI], dv[TO];
                if constexpr (TI == 4) *(float4 *)av = *(const float4 *)&sa[buf][nn][4 * ji];
                else av[0] = sa[buf][nn][ji];
                if constexpr (TO == 4) *(float4 *)dv = *(const float4 *)&sd[buf][nn][4 * jo];
                else dv[0] = sd[buf][nn][0];
#pragma unroll
                for (int o = 0; o < TO; o++)
#pragma unroll
                    for (int i = 0; i < TI; i++) t[o][i] += dv[o] * av[i];
            }
#pragma unroll
            for (int o = 0; o < TO; o++)
#pragma unroll
                for (int i = 0; i < TI; i++) acc[o][i] += t[o][i];
        } else if (bias) {
            float t = 0.f;
#pragma unroll
            for (int nn = 0; nn < WG_CH; nn++) t += sd[buf][nn][tid - JI * JO];
            accb += t;
        }
        if (more) store(buf ^ 1);
        __syncthreads();
    }
    float *P = part + (size_t)blockIdx.x * NW;
    if (mine) {
#pragma unroll
        for (int o = 0; o < TO; o++)
#pragma unroll
            for (int i = 0; i < TI; i++) {
                const int q = TI * ji + i, k = q / CI, ci = q - k * CI;
                P[((TO * jo + o) * CI + ci) * 27 + k] = acc[o][i];
            }
    } else if (bias) {
        P[CO * CI * 27 + tid - JI * JO] = accb;
    }
}

// grad[i] (+)= sum over samples of (sum over the sample's blocks, in order, of
// part[b][i - first parameter of its layer]), for the parameters first .. end - 1
__global__ void __launch_bounds__(64) grad_reduce(const float *part1, const float *part2, const float *part3,
                                                  const float *part4, int per_sample, int ns, int add, float *grad,
                                                  int first, int end)
{
    const int i = first + blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= end) return;
    const float *p;
    int nw, o;
    if (i < OW2) { p = part1; nw = OW2 - OW1; o = OW1; }
    else if (i < OW3) { p = part2; nw = OW3 - OW2; o = OW2; }
    else if (i < OW4) { p = part3; nw = OW4 - OW3; o = OW3; }
    else { p = part4; nw = NPARAM - OW4; o = OW4; }
    p += i - o;
    float t = add ? grad[i] : 0.f;
    for (int s = 0; s < ns; s++) {
        float v = 0.f;
#pragma unroll 16
        for (int b = 0; b < per_sample; b++) v += __ldg(p + (size_t)(s * per_sample + b) * nw);
        t += v;
    }
    grad[i] = t;
}

// Adam (Kingma & Ba) on the FP32 master parameters
__global__ void adam_k(int n, float *w, const float *g, float *m, float *v, float lr, float b1, float b2, float eps,
                       float c1, float c2)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float gi = g[i];
    m[i] = b1 * m[i] + (1.f - b1) * gi;
    v[i] = b2 * v[i] + (1.f - b2) * gi * gi;
    w[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
}

// ---------------------------------------------------------------- host side
// Device buffers of one network pass over up to cap nodes (samples x nodes),
// carved out of one allocation.
struct NetWork {
    NetGrid g;
    float *x = nullptr;         // [2][N]: the in-step warm start's input
    __nv_bfloat16 *a1 = nullptr, *a2 = nullptr, *a3 = nullptr, *dz = nullptr, *dz2 = nullptr;
    float *y = nullptr, *gy = nullptr;
    float *w = nullptr, *grad = nullptr;
    __nv_bfloat16 *W2f = nullptr, *W2b = nullptr, *W3f = nullptr, *W3b = nullptr;
    float *part[4] = {};        // weight-gradient partials per layer
    double *lpart = nullptr;
    void *arena = nullptr;
};

int cuda_err(cudaError_t e) { return e == cudaSuccess ? EKL_OK : EKL_ERR_CUDA; }

// the weight-gradient kernels that need more than 48 KB, before every call that trains
cudaError_t wgrad_opt_in()
{
    static_assert(wg_smem<2, 16>() <= SMEM_DEFAULT, "needs no opt-in");
    const cudaError_t e = smem_opt_in((const void *)wgrad_k<16, 1>, wg_smem<16, 1>());
    return e == cudaSuccess ? smem_opt_in((const void *)wgrad_k<16, 16>, wg_smem<16, 16>()) : e;
}

constexpr int LAYER_PARAMS[4] = {OW2 - OW1, OW3 - OW2, OW4 - OW3, NPARAM - OW4};

// What a pass needs buffers for: the in-step network and ekl_net_eval read one
// input and give its output; training keeps the partials of all layers for one
// reduction, or (TRAIN_TIGHT) reduces layer by layer through one buffer, so that
// a pass over one sample needs no more than a layer's partials at a time.
enum NetUse { NET_EVAL, NET_TRAIN, NET_TRAIN_TIGHT };

// The buffers for passes over `samples` samples of W.g (and `input`: one sample's
// input at W.x) out of `base`; returns their bytes (base null: only that).
size_t work_layout(NetWork &W, NetUse use, int samples, bool input, char *base)
{
    size_t off = 0;
    auto carve = [&](auto *&p, size_t bytes) {
        p = base ? (std::remove_reference_t<decltype(p)>)(base + off) : nullptr;
        off += (bytes + 255) & ~(size_t)255;
    };
    const size_t n = (size_t)samples * W.g.N;
    if (input) carve(W.x, 2 * (size_t)W.g.N * 4);
    carve(W.a1, n * 32);
    carve(W.a2, n * 32);
    carve(W.a3, n * 32);
    carve(W.y, n * 4);
    carve(W.w, NPARAM * 4);
    carve(W.W2f, 27 * 512);
    carve(W.W2b, 27 * 512);
    carve(W.W3f, 27 * 512);
    carve(W.W3b, 27 * 512);
    if (use == NET_EVAL) return off;
    carve(W.dz, n * 32);
    carve(W.dz2, n * 32);
    carve(W.gy, n * 4);
    carve(W.grad, NPARAM * 4);
    carve(W.lpart, ((n + NT - 1) / NT) * sizeof(double));
    const size_t nb = (size_t)samples * ((W.g.N + WG_NODES - 1) / WG_NODES);
    if (use == NET_TRAIN_TIGHT) {
        carve(W.part[0], nb * *std::max_element(LAYER_PARAMS, LAYER_PARAMS + 4) * 4);
        for (int l = 1; l < 4; l++) W.part[l] = W.part[0];
    } else {
        for (int l = 0; l < 4; l++) carve(W.part[l], nb * LAYER_PARAMS[l] * 4);
    }
    return off;
}

// the same, allocated, with `extra` bytes more (256-byte aligned) at *extra_out
int work_alloc(NetWork &W, NetUse use, int samples, bool input, size_t extra = 0, char **extra_out = nullptr)
{
    const size_t bytes = work_layout(W, use, samples, input, nullptr);
    if (cudaMalloc(&W.arena, bytes + extra) != cudaSuccess) {
        cudaGetLastError();
        W.arena = nullptr;
        return EKL_ERR_ALLOC;
    }
    work_layout(W, use, samples, input, (char *)W.arena);
    if (extra_out) *extra_out = (char *)W.arena + bytes;
    return EKL_OK;
}

void work_free(NetWork &W)
{
    cudaFree(W.arena);
    W = NetWork();
}

// BF16 copies of the 16 -> 16 layers' parameters in W.w
void net_prepare(NetWork &W, cudaStream_t s)
{
    prep_w16<<<54, 256, 0, s>>>(W.w, W.W2f, W.W2b, W.W3f, W.W3b);
}

// forward pass over ns samples of `in` with the parameters in W.w (prepared);
// output in W.y
void net_forward(NetWork &W, const NetInput &in, int ns, cudaStream_t s)
{
    NetGrid &g = W.g;
    g.total = ns * g.N;
    const int bn = (g.total + NT - 1) / NT;
    l1_fwd<<<bn, NT, 0, s>>>(g, in, W.w, W.a1);
    conv16<true>(g, W.a1, W.W2f, W.w + OB2, 0, W.a2, nullptr, s);
    conv16<true>(g, W.a2, W.W3f, W.w + OB3, 0, W.a3, nullptr, s);
    const NetTile T = make_tile(g);
    l4_fwd<<<T.ntx * T.nty * T.ntz * ns, TL_T, tc_smem(T), s>>>(g, T, W.a3, W.w, W.y);
}

template <int CI, int CO>
void wgrad(const NetGrid &g, const NetInput &in, const __nv_bfloat16 *a, const void *dz, float *part, cudaStream_t s)
{
    const int blocks = (g.N + WG_NODES - 1) / WG_NODES * (g.total / g.N);
    wgrad_k<CI, CO><<<blocks, WG_T, wg_smem<CI, CO>(), s>>>(g, in, a, dz, part);
}

// gradient of the loss over the ns samples of the last forward pass, into (or
// added to) W.grad; *loss (device) (+)= loss_scale times their summed squared
// error
void net_backward(NetWork &W, const NetInput &in, int ns, const float *d_t, const uint8_t *d_mask, float inv_cnt,
                  bool add, double loss_scale, double *d_loss, cudaStream_t s)
{
    const NetGrid &g = W.g;
    const int bn = (g.total + NT - 1) / NT;
    const int per = (g.N + WG_NODES - 1) / WG_NODES;
    const bool tight = W.part[0] == W.part[1];
    auto reduce = [&](int first, int end) {
        grad_reduce<<<(end - first + 63) / 64, 64, 0, s>>>(W.part[0], W.part[1], W.part[2], W.part[3], per, ns,
                                                          add ? 1 : 0, W.grad, first, end);
    };
    loss_grad_k<<<bn, NT, 0, s>>>(g, W.y, d_t, in.smp, d_mask, inv_cnt, W.gy, W.lpart);
    loss_sum_k<<<1, NT, 0, s>>>(W.lpart, bn, loss_scale, add ? 1 : 0, d_loss);
    wgrad<16, 1>(g, in, W.a3, W.gy, W.part[3], s);
    if (tight) reduce(OW4, NPARAM);
    l4_bwd_data<<<bn, NT, 0, s>>>(g, W.gy, W.w, W.a3, W.dz);
    // dz holds d z3 (through relu of a3)
    wgrad<16, 16>(g, in, W.a2, W.dz, W.part[2], s);
    if (tight) reduce(OW3, OW4);
    conv16<false>(g, W.dz, W.W3b, nullptr, 1, W.dz2, W.a2, s);
    wgrad<16, 16>(g, in, W.a1, W.dz2, W.part[1], s);
    if (tight) reduce(OW2, OW3);
    conv16<false>(g, W.dz2, W.W2b, nullptr, 1, W.dz, W.a1, s);
    wgrad<2, 16>(g, in, nullptr, W.dz, W.part[0], s);
    if (tight) reduce(OW1, OW2);
    else reduce(0, NPARAM);
}

// Extents that the kernels' 32-bit node ids (up to 2 N, the second input
// channel) and the splits into tiles can take: none empty, at most 2^30 nodes.
// False with the message set otherwise.
bool grid_ok(const int32_t dims[3])
{
    long long n = 1;
    for (int a = 0; a < 3; a++) {
        if (dims[a] < 1) {
            set_last_error("every extent must be >= 1");
            return false;
        }
        n *= dims[a];
        if (n > (1ll << 30)) {
            set_last_error("grid too large for 32-bit node ids");
            return false;
        }
    }
    return true;
}

NetGrid make_grid(const int32_t dims[3], const int32_t periodic[3])
{
    NetGrid g;
    g.nx = dims[0];
    g.ny = dims[1];
    g.nz = dims[2];
    for (int a = 0; a < 3; a++) g.per[a] = periodic ? (periodic[a] ? 1 : 0) : 0;
    g.N = g.nx * g.ny * g.nz;
    g.total = g.N;
    return g;
}

// ---------------------------------------------------------------- in-step warm start
struct WarmStart {
    NetWork W;               // on the lattice (level 0) or on cubes of 2^level nodes
    float s_db = 1.f, s_phi = 1.f, s_out = 1.f;
    int enabled = 0;
    int have_prev = 0;
    int level = 0;
    NetGrid fine;            // the lattice
    float *bprev = nullptr, *bcur = nullptr, *phiprev = nullptr;
    float *dbf = nullptr, *phf = nullptr;  // level > 0: the lattice's inputs before restriction
    double *mean = nullptr;
    int collect = 0, crop = 0, ncrops = 0;
    float *crops = nullptr;  // [cap][3][crop^3]: dB, phi_prev, dphi
    long long cap = 0, used = 0;
    uint64_t seed = 0;
};

__global__ void mean_k(const double *part, int n, double nfl, double *mean)
{
    __shared__ double sh[32];
    double v = 0.0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) v += part[k];
    double t = block_sum(v, sh);
    if (threadIdx.x == 0) *mean = nfl > 0 ? t / nfl : 0.0;
}

// network inputs on the lattice: x0 = s_db (b(t) - b(t-1)), x1 = s_phi phi(t-1);
// b = 4 pi l_B (rho - mean)
template <typename R, typename PhiT>
__global__ void ws_inputs(int N, const uint32_t *mask, const R *rho, const double *mean, double c4, const PhiT *phi,
                          const float *bprev, int have_prev, float s_db, float s_phi, float *x0, float *x1,
                          float *bcur, float *phiprev)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    const bool solid = mask[n] & SOLID_BIT;
    float b = solid ? 0.f : (float)(c4 * ((double)rho[n] - *mean));
    float p;
    if constexpr (((PhiT)0.5) != 0) p = (float)phi[n];
    else p = ll_to_float(phi[n]) * (float)PHI_INV;
    if (solid) p = 0.f;
    bcur[n] = b;
    if (phiprev) phiprev[n] = p;
    x0[n] = solid ? 0.f : s_db * (b - (have_prev ? bprev[n] : b));
    x1[n] = s_phi * p;
}

// The network on a coarse level: cell (X, Y, Z) of level L covers the cube
// of 2^L nodes starting at 2^L (X, Y, Z).  Inputs: x0 = s_db times the sum of
// the change of the source over the cube (the source a coarse Poisson
// operator sees), x1 = s_phi times the mean of phi(t-1) over its fluid nodes.
__global__ void ws_restrict(NetGrid f, NetGrid c, int L, const uint32_t *mask, const float *db, const float *ph,
                            float s_db, float s_phi, float *x)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= c.N) return;
    int X, Y, Z;
    xyz_of(c, I, X, Y, Z);
    const int B = 1 << L;
    double sd = 0.0, sp = 0.0;
    int cnt = 0;
    for (int dz = 0; dz < B; dz++)
        for (int dy = 0; dy < B; dy++)
            for (int dx = 0; dx < B; dx++) {
                const int n = (X * B + dx) + f.nx * ((Y * B + dy) + f.ny * (Z * B + dz));
                if (mask[n] & SOLID_BIT) continue;
                sd += (double)db[n];
                sp += (double)ph[n];
                cnt++;
            }
    x[I] = (float)(s_db * sd);
    x[c.N + I] = cnt ? (float)(s_phi * (sp / cnt)) : 0.f;
}

// mean over the fluid nodes of each cube of phi(t) - phi(t-1): the training
// target of the coarse network
template <typename PhiT>
__global__ void ws_coarse_target(NetGrid f, NetGrid c, int L, const uint32_t *mask, const PhiT *phi,
                                 const float *phiprev, float *out)
{
    const int I = blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= c.N) return;
    int X, Y, Z;
    xyz_of(c, I, X, Y, Z);
    const int B = 1 << L;
    double s = 0.0;
    int cnt = 0;
    for (int dz = 0; dz < B; dz++)
        for (int dy = 0; dy < B; dy++)
            for (int dx = 0; dx < B; dx++) {
                const int n = (X * B + dx) + f.nx * ((Y * B + dy) + f.ny * (Z * B + dz));
                if (mask[n] & SOLID_BIT) continue;
                float pn;
                if constexpr (((PhiT)0.5) != 0) pn = (float)phi[n];
                else pn = ll_to_float(phi[n]) * (float)PHI_INV;
                s += (double)(pn - phiprev[n]);
                cnt++;
            }
    out[I] = cnt ? (float)(s / cnt) : 0.f;
}

// phi += s_out y(cube of the node) on the fluid nodes (piecewise-constant
// prolongation of the coarse network's output)
template <typename PhiT>
__global__ void ws_apply_coarse(NetGrid f, NetGrid c, int L, const uint32_t *mask, const float *y, float s_out,
                                PhiT *phi)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= f.N || (mask[n] & SOLID_BIT)) return;
    int x, yy, z;
    xyz_of(f, n, x, yy, z);
    const float d = s_out * y[(x >> L) + c.nx * ((yy >> L) + c.ny * (z >> L))];
    if constexpr (((PhiT)0.5) != 0) phi[n] += (double)d;
    else phi[n] += float_to_ll(d * (float)PHI_SCALE);
}

template <typename PhiT>
__global__ void ws_apply(int N, const uint32_t *mask, const float *y, float s_out, PhiT *phi)
{
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N || (mask[n] & SOLID_BIT)) return;
    const float d = s_out * y[n];
    if constexpr (((PhiT)0.5) != 0) phi[n] += (double)d;
    else phi[n] += float_to_ll(d * (float)PHI_SCALE);
}

// training crops centred on beads (seeded jitter): inputs and the change of
// the converged potential
template <typename PhiT>
__global__ void ws_crops(NetGrid g, const float *x, const float *phiprev, const PhiT *phi, const double *Rb,
                         int nb, int crop, int ncrops, long long step, uint64_t seed, float *out)
{
    const int j = blockIdx.x;
    const int c3 = crop * crop * crop;
    const int b = (int)((step * ncrops + j) % nb);
    uint32_t ctr[4] = {(uint32_t)j, 3u << 24, (uint32_t)step, (uint32_t)((uint64_t)step >> 32)};
    philox4x32_10(ctr, (uint32_t)seed, (uint32_t)(seed >> 32));
    int o[3];
    for (int a = 0; a < 3; a++) {
        int jit = (int)(ctr[a] % 5u) - 2;
        o[a] = (int)floor(Rb[3 * b + a]) + jit - crop / 2;
    }
    for (int t = threadIdx.x; t < c3; t += blockDim.x) {
        int cx = t % crop, cy = (t / crop) % crop, cz = t / (crop * crop);
        int q[3] = {o[0] + cx, o[1] + cy, o[2] + cz};
        const int dims[3] = {g.nx, g.ny, g.nz};
        bool in = true;
        for (int a = 0; a < 3; a++) {
            if (q[a] < 0 || q[a] >= dims[a]) {
                if (g.per[a]) q[a] = ((q[a] % dims[a]) + dims[a]) % dims[a];
                else in = false;
            }
        }
        float v0 = 0.f, v1 = 0.f, v2 = 0.f;
        if (in) {
            int n = q[0] + g.nx * (q[1] + g.ny * q[2]);
            v0 = x[n];
            v1 = x[g.N + n];
            float pn;
            if constexpr (((PhiT)0.5) != 0) pn = (float)phi[n];
            else pn = ll_to_float(phi[n]) * (float)PHI_INV;
            v2 = (v1 == 0.f && phiprev[n] == 0.f) ? 0.f : pn - phiprev[n];
        }
        float *dst = out + (size_t)j * 3 * c3;
        dst[t] = v0;
        dst[c3 + t] = v1;
        dst[2 * c3 + t] = v2;
    }
}

}  // namespace

namespace ekl {

int warmstart_before_poisson(Ctx &c)
{
    WarmStart &ws = *(WarmStart *)c.net;
    const int N = (int)c.N;
    mean_k<<<1, 1024, 0, c.stream>>>(c.part_charge, c.charge_blocks, (double)c.n_fluid, ws.mean);
    const int bn = (N + 255) / 256;
    const int have = ws.have_prev;
    const int L = ws.level;
    // level 0: the inputs go straight to the network; level > 0: unscaled
    // into the lattice buffers, then restricted (and scaled) per cube
    float *x0 = L ? ws.dbf : ws.W.x, *x1 = L ? ws.phf : ws.W.x + N;
    const float sdb = L ? 1.f : ws.s_db, sph = L ? 1.f : ws.s_phi;
    if (c.prec == EKL_F64)
        ws_inputs<double, double><<<bn, 256, 0, c.stream>>>(N, c.mask, (const double *)c.rho, ws.mean, c.c4,
                                                           (const double *)c.phi, ws.bprev, have, sdb, sph, x0, x1,
                                                           ws.bcur, ws.collect ? ws.phiprev : nullptr);
    else
        ws_inputs<float, long long><<<bn, 256, 0, c.stream>>>(N, c.mask, (const float *)c.rho, ws.mean, c.c4,
                                                             (const long long *)c.phi, ws.bprev, have, sdb, sph, x0,
                                                             x1, ws.bcur, ws.collect ? ws.phiprev : nullptr);
    c.launches += 2;
    if (L) {
        ws_restrict<<<(ws.W.g.N + 255) / 256, 256, 0, c.stream>>>(ws.fine, ws.W.g, L, c.mask, ws.dbf, ws.phf,
                                                                  ws.s_db, ws.s_phi, ws.W.x);
        c.launches++;
    }
    if (ws.enabled && have) {
        net_forward(ws.W, NetInput{ws.W.x, nullptr}, 1, c.stream);
        if (L) {
            if (c.prec == EKL_F64)
                ws_apply_coarse<double><<<bn, 256, 0, c.stream>>>(ws.fine, ws.W.g, L, c.mask, ws.W.y, ws.s_out,
                                                                  (double *)c.phi);
            else
                ws_apply_coarse<long long><<<bn, 256, 0, c.stream>>>(ws.fine, ws.W.g, L, c.mask, ws.W.y, ws.s_out,
                                                                     (long long *)c.phi);
        } else {
            if (c.prec == EKL_F64) ws_apply<double><<<bn, 256, 0, c.stream>>>(N, c.mask, ws.W.y, ws.s_out, (double *)c.phi);
            else ws_apply<long long><<<bn, 256, 0, c.stream>>>(N, c.mask, ws.W.y, ws.s_out, (long long *)c.phi);
        }
        c.launches += 5;
    }
    std::swap(ws.bprev, ws.bcur);
    ws.have_prev = 1;
    return cudaGetLastError() == cudaSuccess ? EKL_OK : EKL_ERR_CUDA;
}

int warmstart_after_poisson(Ctx &c)
{
    WarmStart &ws = *(WarmStart *)c.net;
    if (ws.collect && ws.level && ws.used < ws.cap) {
        // one sample per step: the whole coarse grid (inputs as fed, target)
        const size_t NL = (size_t)ws.W.g.N;
        float *dst = ws.crops + (size_t)ws.used * 3 * NL;
        cudaMemcpyAsync(dst, ws.W.x, 2 * NL * 4, cudaMemcpyDeviceToDevice, c.stream);
        if (c.prec == EKL_F64)
            ws_coarse_target<double><<<(ws.W.g.N + 255) / 256, 256, 0, c.stream>>>(
                ws.fine, ws.W.g, ws.level, c.mask, (const double *)c.phi, ws.phiprev, dst + 2 * NL);
        else
            ws_coarse_target<long long><<<(ws.W.g.N + 255) / 256, 256, 0, c.stream>>>(
                ws.fine, ws.W.g, ws.level, c.mask, (const long long *)c.phi, ws.phiprev, dst + 2 * NL);
        c.launches++;
        ws.used++;
        return cudaGetLastError() == cudaSuccess ? EKL_OK : EKL_ERR_CUDA;
    }
    if (!ws.collect || ws.level || c.nb == 0 || ws.used + ws.ncrops > ws.cap) return EKL_OK;
    const size_t c3 = (size_t)ws.crop * ws.crop * ws.crop;
    float *dst = ws.crops + (size_t)ws.used * 3 * c3;
    if (c.prec == EKL_F64)
        ws_crops<double><<<ws.ncrops, 256, 0, c.stream>>>(ws.W.g, ws.W.x, ws.phiprev, (const double *)c.phi,
                                                         (const double *)c.R, c.nb, ws.crop, ws.ncrops, c.step,
                                                         ws.seed, dst);
    else
        ws_crops<long long><<<ws.ncrops, 256, 0, c.stream>>>(ws.W.g, ws.W.x, ws.phiprev, (const long long *)c.phi,
                                                            (const double *)c.R, c.nb, ws.crop, ws.ncrops, c.step,
                                                            ws.seed, dst);
    c.launches++;
    ws.used += ws.ncrops;
    return cudaGetLastError() == cudaSuccess ? EKL_OK : EKL_ERR_CUDA;
}

void warmstart_free(Ctx &c)
{
    if (!c.net) return;
    WarmStart *ws = (WarmStart *)c.net;
    work_free(ws->W);
    cudaFree(ws->bprev);
    cudaFree(ws->bcur);
    cudaFree(ws->phiprev);
    cudaFree(ws->dbf);
    cudaFree(ws->phf);
    cudaFree(ws->mean);
    cudaFree(ws->crops);
    delete ws;
    c.net = nullptr;
}

// the warm start's state on the network level `level` (recreated when the
// level changes; the parameters are installed afterwards)
static int warmstart_ensure(Ctx &c, int level = -1)
{
    if (c.net && (level < 0 || ((WarmStart *)c.net)->level == level)) return EKL_OK;
    if (c.net) warmstart_free(c);
    if (level < 0) level = 0;
    WarmStart *ws = new (std::nothrow) WarmStart();
    if (!ws) return EKL_ERR_ALLOC;
    const int32_t dims[3] = {c.nx, c.ny, c.nz};
    ws->fine = make_grid(dims, c.per);
    ws->level = level;
    const int32_t cdims[3] = {c.nx >> level, c.ny >> level, c.nz >> level};
    ws->W.g = make_grid(cdims, c.per);
    const int N = (int)c.N;
    int rc = work_alloc(ws->W, NET_EVAL, 1, true);
    cudaError_t e = rc == EKL_OK ? cudaSuccess : cudaErrorMemoryAllocation;
    if (e == cudaSuccess) e = cudaMalloc(&ws->bprev, (size_t)N * 4);
    if (e == cudaSuccess) e = cudaMalloc(&ws->bcur, (size_t)N * 4);
    if (e == cudaSuccess) e = cudaMalloc(&ws->phiprev, (size_t)N * 4);
    if (e == cudaSuccess && level) e = cudaMalloc(&ws->dbf, (size_t)N * 4);
    if (e == cudaSuccess && level) e = cudaMalloc(&ws->phf, (size_t)N * 4);
    if (e == cudaSuccess) e = cudaMalloc(&ws->mean, sizeof(double));
    c.net = ws;
    if (e != cudaSuccess) {
        warmstart_free(c);
        return EKL_ERR_ALLOC;
    }
    return EKL_OK;
}

}  // namespace ekl

// EKL_ERR_TIMEOUT when a tensor-core block gave up waiting for its MMAs
// (the flag is cleared on reading)
static int tc_check()
{
    int st = 0;
    if (cudaMemcpyFromSymbol(&st, tc_status, sizeof(int)) != cudaSuccess) return EKL_ERR_CUDA;
    if (!st) return EKL_OK;
    const int zero = 0;
    cudaMemcpyToSymbol(tc_status, &zero, sizeof(int));
    return EKL_ERR_TIMEOUT;
}

extern "C" {

int ekl_net_tensor_path(int32_t path)
{
    const int prev = g_tensor_path;
    if (path == 0 || path == 1) g_tensor_path = path;
    return prev;
}

int ekl_net_eval(const int32_t dims[3], const int32_t periodic[3], const float *x, const float *w, float *y)
{
    if (!dims || !x || !w || !y || !grid_ok(dims)) return EKL_ERR_ARG;
    NetWork W;
    W.g = make_grid(dims, periodic);
    int rc = work_alloc(W, NET_EVAL, 1, true);
    if (rc != EKL_OK) return rc;
    cudaError_t e = cudaMemcpy(W.x, x, 2 * (size_t)W.g.N * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(W.w, w, NPARAM * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        net_prepare(W, 0);
        net_forward(W, NetInput{W.x, nullptr}, 1, 0);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpy(y, W.y, (size_t)W.g.N * 4, cudaMemcpyDeviceToHost);
    }
    work_free(W);
    if (e == cudaSuccess) return tc_check();
    return cuda_err(e);
}

static long long mask_count(const uint8_t *mask, int N)
{
    long long cnt = N;
    if (mask) {
        cnt = 0;
        for (int i = 0; i < N; i++) cnt += mask[i] ? 1 : 0;
    }
    return cnt;
}

int ekl_net_loss_grad(const int32_t dims[3], const int32_t periodic[3], const float *x, const float *target,
                      const uint8_t *mask, const float *w, double *loss, float *grad)
{
    if (!dims || !x || !target || !w || !grad || !grid_ok(dims)) return EKL_ERR_ARG;
    NetWork W;
    W.g = make_grid(dims, periodic);
    const int N = W.g.N;
    char *extra = nullptr;
    const size_t tb = ((size_t)N * 4 + 255) & ~(size_t)255;
    const size_t more = tb + 256 + (mask ? (size_t)N : 0);
    int rc = work_alloc(W, NET_TRAIN, 1, true, more, &extra);
    if (rc != EKL_OK) rc = work_alloc(W, NET_TRAIN_TIGHT, 1, true, more, &extra);
    if (rc != EKL_OK) return rc;
    float *dt = (float *)extra;
    double *dloss = (double *)(extra + tb);
    uint8_t *dm = mask ? (uint8_t *)(extra + tb + 256) : nullptr;
    const long long cnt = mask_count(mask, N);
    const float inv_cnt = 1.f / (float)(cnt > 0 ? cnt : 1);
    cudaError_t e = wgrad_opt_in();
    if (e == cudaSuccess) e = cudaMemcpy(W.x, x, 2 * (size_t)N * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(W.w, w, NPARAM * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dt, target, (size_t)N * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && mask) e = cudaMemcpy(dm, mask, N, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        const NetInput in{W.x, nullptr};
        net_prepare(W, 0);
        net_forward(W, in, 1, 0);
        net_backward(W, in, 1, dt, dm, inv_cnt, false, (double)inv_cnt, dloss, 0);
        e = cudaGetLastError();
        if (e == cudaSuccess && loss) e = cudaMemcpy(loss, dloss, sizeof(double), cudaMemcpyDeviceToHost);
        if (e == cudaSuccess) e = cudaMemcpy(grad, W.grad, NPARAM * 4, cudaMemcpyDeviceToHost);
    }
    work_free(W);
    if (e == cudaSuccess) return tc_check();
    return cuda_err(e);
}

// Device memory for the buffers of one training pass.  The samples of a batch go
// through the network together as long as their buffers stay under it (168 bytes
// a node, and 61 KB of weight-gradient partials per sample and 512 nodes of it), else
// in several passes whose gradients add up.  Where the device has less to give,
// passes of half as many samples are tried, and at last one sample with the
// partials of one layer at a time.
static constexpr uint64_t NET_PASS_BYTES = 4ull << 30;
// sample numbers and losses that are on the device at a time
static constexpr int NET_DRAWS = 4096, NET_LOSSES = 512;

static int train_grid(int32_t nsamples, const int32_t dims[3], const int32_t periodic[3], const float *x,
                      const float *target, const uint8_t *mask, float *w, int32_t iters, int32_t batch, float lr,
                      uint64_t seed, float *loss_out, uint64_t pass_bytes)
{
    if (nsamples < 1 || !dims || !x || !target || !w || iters < 0 || batch < 1 || !grid_ok(dims)) return EKL_ERR_ARG;
    NetWork W;
    W.g = make_grid(dims, periodic);
    const int N = W.g.N;
    const size_t one = work_layout(W, NET_TRAIN, 1, false, nullptr);
    const size_t next = work_layout(W, NET_TRAIN, 2, false, nullptr) - one;  // bytes of one more sample
    const uint64_t fit = std::min<uint64_t>(pass_bytes / next, (1u << 30) / (unsigned)N);
    int group = (int)std::max<uint64_t>(1, std::min<uint64_t>(fit, (uint64_t)batch));
    NetUse use = pass_bytes ? NET_TRAIN : NET_TRAIN_TIGHT;
    const int64_t total = (int64_t)iters * batch;
    float *dx, *dt, *m1, *m2;
    uint8_t *dm = nullptr;
    int *dsmp, draws;
    double *dloss;
    for (;;) {
        draws = (int)std::max<int64_t>(group, std::min<int64_t>(total, NET_DRAWS));
        char *base = nullptr;
        size_t off = 0;
        auto carve = [&](auto *&p, size_t bytes) {
            p = (std::remove_reference_t<decltype(p)>)(base ? base + off : nullptr);
            off += (bytes + 255) & ~(size_t)255;
        };
        auto layout = [&] {
            off = 0;
            carve(dx, (size_t)nsamples * 2 * N * 4);
            carve(dt, (size_t)nsamples * N * 4);
            carve(m1, NPARAM * 4);
            carve(m2, NPARAM * 4);
            carve(dsmp, (size_t)draws * sizeof(int));
            carve(dloss, NET_LOSSES * sizeof(double));
            if (mask) carve(dm, (size_t)N);
        };
        layout();
        const int rc = work_alloc(W, use, group, false, off, &base);
        if (rc == EKL_OK) {
            layout();
            break;
        }
        if (group > 1) group = (group + 1) / 2;
        else if (use == NET_TRAIN) use = NET_TRAIN_TIGHT;
        else return rc;
    }
    std::unique_ptr<int[]> smp(new (std::nothrow) int[draws]);
    if (!smp) {
        work_free(W);
        return EKL_ERR_ALLOC;
    }
    const long long cnt = mask_count(mask, N);
    // seeded sample order (splitmix64), drawn and uploaded `draws` at a time
    uint64_t st = seed;
    auto next_draw = [&]() {
        st += 0x9E3779B97F4A7C15ull;
        uint64_t z = st;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        return z ^ (z >> 31);
    };
    int64_t drawn = 0;
    int at = 0, have = 0;  // the next sample's place and the number uploaded
    auto refill = [&] {    // (the copy follows the passes that read the last ones)
        std::copy(smp.get() + at, smp.get() + have, smp.get());
        have -= at;
        at = 0;
        for (; have < draws && drawn < total; have++, drawn++) smp[have] = (int)(next_draw() % (uint64_t)nsamples);
        return cudaMemcpy(dsmp, smp.get(), (size_t)have * sizeof(int), cudaMemcpyHostToDevice);
    };
    cudaError_t e = wgrad_opt_in();
    if (e == cudaSuccess) e = cudaMemcpy(dx, x, (size_t)nsamples * 2 * N * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dt, target, (size_t)nsamples * N * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && mask) e = cudaMemcpy(dm, mask, N, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(W.w, w, NPARAM * 4, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(m1, 0, NPARAM * 4);
    if (e == cudaSuccess) e = cudaMemset(m2, 0, NPARAM * 4);
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float inv_cnt = 1.f / (float)(cnt * batch);
    double losses[NET_LOSSES];
    for (int it = 0; it < iters && e == cudaSuccess; it++) {
        net_prepare(W, 0);
        for (int64_t k = 0; k < batch; k += group) {
            const int ns = (int)std::min<int64_t>(batch - k, group);
            if (have - at < ns) e = refill();
            if (e != cudaSuccess) break;
            const NetInput in{dx, dsmp + at};
            net_forward(W, in, ns, 0);
            net_backward(W, in, ns, dt, dm, inv_cnt, k > 0, (double)inv_cnt, dloss + it % NET_LOSSES, 0);
            at += ns;
        }
        const float c1 = 1.f - powf(b1, (float)(it + 1)), c2 = 1.f - powf(b2, (float)(it + 1));
        adam_k<<<(NPARAM + 255) / 256, 256>>>(NPARAM, W.w, W.grad, m1, m2, lr, b1, b2, eps, c1, c2);
        if (e == cudaSuccess) e = cudaGetLastError();
        const int filled = it % NET_LOSSES + 1;
        if (e == cudaSuccess && loss_out && (filled == NET_LOSSES || it + 1 == iters)) {
            e = cudaMemcpy(losses, dloss, (size_t)filled * sizeof(double), cudaMemcpyDeviceToHost);
            for (int k = 0; k < filled; k++) loss_out[it + 1 - filled + k] = (float)losses[k];
        }
    }
    if (e == cudaSuccess) e = cudaMemcpy(w, W.w, NPARAM * 4, cudaMemcpyDeviceToHost);
    work_free(W);
    if (e == cudaSuccess) return tc_check();
    return cuda_err(e);
}

int ekl_net_train_grid(int32_t nsamples, const int32_t dims[3], const int32_t periodic[3], const float *x,
                       const float *target, const uint8_t *mask, float *w, int32_t iters, int32_t batch, float lr,
                       uint64_t seed, float *loss_out)
{
    return train_grid(nsamples, dims, periodic, x, target, mask, w, iters, batch, lr, seed, loss_out, NET_PASS_BYTES);
}

// ekl_net_train_grid in passes of at most pass_bytes (at least one sample; 0: one
// sample and the partials of one layer at a time): the splits that a large batch or
// a nearly full device leads to, for the tests; not part of the interface
int ekl_net_train_in_passes(int32_t nsamples, const int32_t dims[3], const int32_t periodic[3], const float *x,
                            const float *target, const uint8_t *mask, float *w, int32_t iters, int32_t batch,
                            float lr, uint64_t seed, float *loss_out, uint64_t pass_bytes)
{
    return train_grid(nsamples, dims, periodic, x, target, mask, w, iters, batch, lr, seed, loss_out, pass_bytes);
}

int ekl_net_train(int32_t nsamples, const int32_t dims[3], const float *x, const float *target,
                  const uint8_t *mask, float *w, int32_t iters, int32_t batch, float lr, uint64_t seed,
                  float *loss_out)
{
    const int32_t closed[3] = {0, 0, 0};
    return ekl_net_train_grid(nsamples, dims, closed, x, target, mask, w, iters, batch, lr, seed, loss_out);
}

}  // extern "C"

extern "C" {

int ekl_warmstart_level(ekl_handle *h, int32_t level)
{
    if (!h || level < 0 || level > 4) return EKL_ERR_ARG;
    ekl::DeviceScope dscope(h->c.device);
    if (!dscope.ok()) {
        ekl::set_last_error("the handle's device cannot be made current");
        return EKL_ERR_ARG;
    }
    ekl::Ctx &c = h->c;
    const int B = 1 << level;
    if (c.nx % B || c.ny % B || c.nz % B) {
        ekl::set_last_error("every extent must be a multiple of 2^level");
        return EKL_ERR_ARG;
    }
    return ekl::warmstart_ensure(c, level);
}

int ekl_set_warmstart(ekl_handle *h, const float *w, const float scales[3])
{
    if (!h) return EKL_ERR_ARG;
    ekl::DeviceScope dscope(h->c.device);
    if (!dscope.ok()) {
        ekl::set_last_error("the handle's device cannot be made current");
        return EKL_ERR_ARG;
    }
    ekl::Ctx &c = h->c;
    if (!w) {
        if (c.net) ((WarmStart *)c.net)->enabled = 0;
        return EKL_OK;
    }
    int rc = ekl::warmstart_ensure(c);
    if (rc != EKL_OK) return rc;
    WarmStart &ws = *(WarmStart *)c.net;
    // ordered on the handle's stream: earlier steps still read the old parameters
    if (cudaStreamSynchronize(c.stream) != cudaSuccess ||
        cudaMemcpy(ws.W.w, w, NPARAM * 4, cudaMemcpyHostToDevice) != cudaSuccess)
        return EKL_ERR_CUDA;
    net_prepare(ws.W, c.stream);
    if (cudaGetLastError() != cudaSuccess) return EKL_ERR_CUDA;
    if (scales) {
        ws.s_db = scales[0];
        ws.s_phi = scales[1];
        ws.s_out = scales[2];
    }
    ws.enabled = 1;
    return EKL_OK;
}

int ekl_warmstart_collect(ekl_handle *h, int32_t nsteps, int32_t crop, int32_t ncrops, uint64_t seed, float *out,
                          int64_t *n_out)
{
    if (!h || nsteps < 1 || ncrops < 1 || !out) return EKL_ERR_ARG;
    ekl::DeviceScope dscope(h->c.device);
    if (!dscope.ok()) {
        ekl::set_last_error("the handle's device cannot be made current");
        return EKL_ERR_ARG;
    }
    ekl::Ctx &c = h->c;
    int rc = ekl::warmstart_ensure(c);
    if (rc != EKL_OK) return rc;
    WarmStart &ws = *(WarmStart *)c.net;
    if (!ws.level && (c.nb == 0 || crop < 4)) return EKL_ERR_ARG;  // bead-centred crops
    const int en = ws.enabled;
    const float s0 = ws.s_db, s1 = ws.s_phi, s2 = ws.s_out;
    ws.enabled = 0;
    ws.s_db = ws.s_phi = ws.s_out = 1.f;
    ws.collect = 1;
    ws.crop = crop;
    ws.ncrops = ncrops;
    ws.seed = seed;
    // level > 0: one sample per step, the whole coarse grid
    ws.cap = ws.level ? (long long)nsteps : (long long)nsteps * ncrops;
    ws.used = 0;
    const size_t c3 = ws.level ? (size_t)ws.W.g.N : (size_t)crop * crop * crop;
    if (cudaMalloc(&ws.crops, (size_t)ws.cap * 3 * c3 * 4) != cudaSuccess) {
        ws.collect = 0;
        return EKL_ERR_ALLOC;
    }
    rc = ekl_step(h, nsteps);
    if (rc >= 0) {
        if (cudaMemcpy(out, ws.crops, (size_t)ws.used * 3 * c3 * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
            rc = EKL_ERR_CUDA;
        if (n_out) *n_out = ws.used;
    }
    cudaFree(ws.crops);
    ws.crops = nullptr;
    ws.collect = 0;
    ws.enabled = en;
    ws.s_db = s0;
    ws.s_phi = s1;
    ws.s_out = s2;
    return rc;
}

}  // extern "C"
