// Message layers of the learned surrogate on the fifth-generation tensor cores (sm_103a).
// Forward (k_msg_layer_tc):
//     Y[n][j] = tanh( sum_k Z[n][k] W[k][j] + b[j] ),  h_next[n][j] = h[n][j] + Y[n][j],  j < 64,
// where the CTA forms its rows of Z (bfloat16 values) from the hidden states while staging
// them, so Z never goes to memory; W is bfloat16 and the products accumulate in FP32 in
// tensor memory.
//
// A CTA of 256 threads takes tiles of 128 rows one after another. It stages a tile of Z in shared
// memory in blocks of 64 features with the 128-byte swizzle and, once, the whole W (as W^T, from a
// copy packed once per weight update by k_pack_wt) in the K-major layout without swizzle: core
// matrices of 8 rows x 8 bf16 (16 bytes per row, 128 bytes each), core matrices adjacent along K
// 128 bytes apart, along N K * 16 bytes apart. One thread issues K/16 MMAs of shape 128 x 64 x 16 into a 64-column
// TMEM accumulator and commits them to an mbarrier; after a bounded wait the warps read the
// accumulator back with tcgen05.ld and turn it through shared memory, so that bias, activation,
// residual and the stores run in the coalesced order of the gather.
//
// Backward (k_bwd_layer_tc): one kernel per layer forms dA, rebuilds Z, and multiplies both
// gradients from the same staged tiles.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sesw_device.cuh"
#include "sesw_internal.h"
#include "sesw_msg.cuh"

namespace sesw {

namespace {

constexpr int TC_M = kMsgTile;   // rows per tile: one MMA with M = 128
constexpr int TC_N = 64;         // output columns: the hidden width
constexpr int TC_THREADS = 256;  // eight warps: warp w reads TMEM lanes 32 (w % 4) .. + 31, columns 32 (w / 4) .. + 31

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor (tcgen05) of a K-major operand without swizzle: start
// address, leading byte offset (between core matrices adjacent along K), stride byte
// offset (along M or N), all in 16-byte units; bit 46 is the descriptor version.
__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// The same for a tile of 128-byte rows with the 128-byte swizzle (layout type 2 in bits 61-63): 64
// bfloat16 per row, 16-byte chunk j of row r at chunk j ^ (r & 7), 8 rows per 1024-byte group.
__device__ __forceinline__ uint64_t umma_desc_sw(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return umma_desc(addr, lbo, sbo) | ((uint64_t)2 << 61);
}

// Instruction descriptor of tcgen05.mma kind::f16: FP32 accumulator (bits 4-5 = 1),
// BF16 A and B (bits 7-9 and 10-12 = 1), both K-major, N / 8 at bit 17, M / 16 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// Read 16 FP32 columns of this warp's 32 TMEM lanes.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int t = 0; t < 16; t++) v[t] = __uint_as_float(r[t]);
}

// W (K x 64, row-major bf16) as the shared-memory image of W^T that k_msg_layer_tc copies:
// 16-byte chunk c = (jg * K/8 + kc) * 8 + jl holds W[8 kc .. 8 kc + 7][8 jg + jl].
__global__ void k_pack_wt(int K, const __nv_bfloat16 *__restrict__ W, uint4 *__restrict__ out)
{
    const int KC = K / 8;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < TC_N * KC; c += gridDim.x * blockDim.x) {
        const int jl = c & 7, kc = (c >> 3) % KC, jg = (c >> 3) / KC;
        const int j = jg * 8 + jl;
        unsigned short h[8];
#pragma unroll
        for (int t = 0; t < 8; t++) h[t] = __bfloat16_as_ushort(W[(size_t)(kc * 8 + t) * TC_N + j]);
        out[c] = make_uint4((uint32_t)h[0] | ((uint32_t)h[1] << 16), (uint32_t)h[2] | ((uint32_t)h[3] << 16),
                            (uint32_t)h[4] | ((uint32_t)h[5] << 16), (uint32_t)h[6] | ((uint32_t)h[7] << 16));
    }
}

__device__ __forceinline__ uint4 pack_bf16x8(const float *v)
{
    return make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]),
                      pack_bf16x2(v[6], v[7]));
}

// Eight floats of global memory in one 32-byte access (32-byte aligned): the gathers are bound by the
// L1 pipe, which takes a whole sector per thread in half the passes of two 16-byte accesses.
__device__ __forceinline__ void load8(const float *p, float *v)
{
    asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
}

__device__ __forceinline__ void store8(float *p, const float *v)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
}

// Eight floats of the turned tile (shared memory) for channel octet cg: the upper four octets take
// their halves in the other order, so that a quarter warp reads all 32 banks.
__device__ __forceinline__ void load8_turned(const float *p, int cg, float *v)
{
    const bool up = cg >= 4;
    const float4 x = reinterpret_cast<const float4 *>(p)[up ? 1 : 0], y = reinterpret_cast<const float4 *>(p)[up ? 0 : 1];
    const float4 a = up ? y : x, b = up ? x : y;
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16 &hi, __nv_bfloat16 &lo)
{
    hi = __float2bfloat16_rn(v);
    lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

__device__ __forceinline__ uint32_t bf16x2_bits(__nv_bfloat16 a, __nv_bfloat16 b)
{
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}

// Element incidences of a vertex-layer tile's rows held in shared memory (more go through
// global memory, in the same order).
constexpr int MSG_INC_CAP = 1536;

// The turned accumulator: 128 rows of 64 floats, 68 apart (rows 17 x 16 bytes apart keep both
// the row-wise stores and the octet-wise loads free of bank conflicts).
constexpr int TURN_LD = 68;
constexpr size_t TURN_BYTES = (size_t)TC_M * TURN_LD * 4;

__host__ __device__ constexpr size_t cmax(size_t a, size_t b) { return a > b ? a : b; }

// Graph data of a tile's rows: KIND 0 the three corners of 128 elements; KIND 1 the 129 CSR
// offsets of the rows and the incidences (element << 2 | corner) and element areas of up to
// MSG_INC_CAP incidences.
__host__ __device__ constexpr size_t graph_smem(int kind)
{
    return kind == 0 ? (size_t)TC_M * 12 : (size_t)(TC_M + 4) * 4 + (size_t)MSG_INC_CAP * 8;
}

// Shared memory of k_msg_layer_tc: the A tile (128 x K bf16; the turned accumulator takes its
// place), W^T (64 x K bf16), the graph data. Three CTAs fit an SM.
__host__ __device__ constexpr size_t msg_a_smem(int kind)
{
    return cmax((size_t)TC_M * (kind == 0 ? 3 * TC_N : 2 * TC_N) * 2, TURN_BYTES);
}
__host__ __device__ constexpr size_t msg_layer_smem(int kind)
{
    return msg_a_smem(kind) + (size_t)TC_N * (kind == 0 ? 3 * TC_N : 2 * TC_N) * 2 + graph_smem(kind);
}

// The graph arrays of a layer and where a tile's share of them sits in shared memory.
struct TileGraph {
    int *tri;                    // KIND 0: [3][128]
    int *off, *inc;              // KIND 1
    float *area;
    int qbase;
    bool inc_smem;
};

template <int KIND>
__device__ __forceinline__ TileGraph tile_graph_at(unsigned char *gdata)
{
    TileGraph g;
    g.tri = reinterpret_cast<int *>(gdata);
    g.off = reinterpret_cast<int *>(gdata);
    g.inc = g.off + TC_M + 4;
    g.area = reinterpret_cast<float *>(g.inc + MSG_INC_CAP);
    g.qbase = 0;
    g.inc_smem = false;
    return g;
}

// Load the graph data of rows n0 .. n0 + 127 (rows past N: element 0's corners; empty CSR
// rows) so that every gather has its address at hand. Ends with a block barrier.
template <int KIND>
__device__ __forceinline__ void load_tile_graph(const MsgLayerArgs &a, int n0, TileGraph &g)
{
    if constexpr (KIND == 0) {
        for (int r = threadIdx.x; r < TC_M; r += TC_THREADS) {
            const int4 v = n0 + r < a.N ? a.etri[n0 + r] : make_int4(0, 0, 0, 0);
            g.tri[r] = v.x;
            g.tri[TC_M + r] = v.y;
            g.tri[2 * TC_M + r] = v.z;
        }
    } else {
        for (int r = threadIdx.x; r <= TC_M; r += TC_THREADS) g.off[r] = a.voff[min(n0 + r, a.N)];
        __syncthreads();
        g.qbase = g.off[0];
        const int nq = g.off[TC_M] - g.qbase;
        g.inc_smem = nq <= MSG_INC_CAP;
        if (g.inc_smem) {
            for (int t = threadIdx.x; t < nq; t += TC_THREADS) {
                const int ek = a.vinc[g.qbase + t];
                g.inc[t] = ek;
                g.area[t] = a.earea[ek >> 2];
            }
        }
    }
    __syncthreads();
}

// Thread item u of a tile: row r and the 8 hidden channels 8 cg .. 8 cg + 7; eight consecutive
// threads cover one row, so that each global access of a quarter warp is 256 contiguous bytes
// (with eight rows per quarter, every lane's access was an L1 pass of its own: 88 % of the
// L1 pipe, 334 us for the 910k-row element layer).
constexpr int ITEMS = TC_M * (TC_N / 8) / TC_THREADS;
__device__ __forceinline__ int item_row(int u) { return ((int)threadIdx.x >> 3) + u * (TC_THREADS / 8); }
__device__ __forceinline__ int item_cg() { return (int)threadIdx.x & 7; }

// A staged tile of 128 rows: blocks of 64 features (128 rows x 128 bytes, swizzled), one after
// another. Where chunk cg (8 features) of row r of block k sits, in 16-byte units.
constexpr int TILE_BLOCK = TC_M * TC_N * 2;   // bytes
__device__ __forceinline__ int tile_chunk(int r, int cg, int k)
{
    return k * (TILE_BLOCK / 16) + r * 8 + (cg ^ (r & 7));
}

// Read the accumulator's columns [col, col + 64) into the turned tile: warp w reads lanes
// 32 (w % 4) .. + 31 and 32 columns. The caller synchronises the block before the tile is read.
__device__ __forceinline__ void turn_tile(uint32_t tmem_col, float *turn)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, quarter = warp & 3, half = warp >> 2;
    const uint32_t taddr = tmem_col + ((uint32_t)(quarter * 32) << 16);
    float *row = turn + (size_t)(quarter * 32 + lane) * TURN_LD;
#pragma unroll
    for (int q = 2 * half; q < 2 * half + 2; q++) {
        float v[16];
        tmem_ld16(taddr + q * 16, v);
#pragma unroll
        for (int t = 0; t < 16; t += 4)
            *reinterpret_cast<float4 *>(row + q * 16 + t) = make_float4(v[t], v[t + 1], v[t + 2], v[t + 3]);
    }
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, int accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Bounded wait on phase `parity` of an mbarrier; false when the budget ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long budget)
{
    const long long t0 = clock64();
    while (true) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (clock64() - t0 > budget) return false;
    }
}

// The wait for committed MMAs: a wait that gives up flags the timeout and waits one more budget,
// so that TMEM is not freed under MMAs still in flight.
__device__ __forceinline__ bool mma_wait(uint32_t bar, uint32_t parity, long long budget, unsigned *status)
{
    if (mbar_wait(bar, parity, budget)) return true;
    atomicOr(status, 2u);
    mbar_wait(bar, parity, budget);
    return false;
}

// One message layer of the surrogate's forward pass (KIND 0: element rows, K = 192; KIND 1:
// vertex rows, K = 128): the CTA forms 128 rows of Z from the hidden states while it
// stages them as the A tile, so Z never goes to memory, then Y = tanh(Z W + b) and
// h_next = h + Y. Bound by the gathers of the hidden states (1.5 KB of FP32 rows per element
// row, 2 KB per vertex row, most of it from L2): persistent CTAs load W once, the rows' own
// hidden states stay in registers for the residual, and results leave coalesced (before, each
// lane stored its own row: 32 partial lines per store). Level 8 (459k vertices, 910k triangles):
// element layer 462 -> 190 us, vertex layer 313 -> 133 us.
template <int KIND>
__global__ void __launch_bounds__(TC_THREADS, 3)
k_msg_layer_tc(const MsgLayerArgs a, const uint4 *__restrict__ Wp, const float *__restrict__ bias,
               unsigned *__restrict__ status, long long wait_cycles)
{
    constexpr int K = KIND == 0 ? 3 * TC_N : 2 * TC_N;
    constexpr int KC = K / 8;    // core matrices along K
    extern __shared__ __align__(1024) unsigned char smem[];
    uint4 *As = reinterpret_cast<uint4 *>(smem);                              // 128 x K bf16
    float *turn = reinterpret_cast<float *>(smem);                            // in its place after the MMAs
    uint4 *Bs = reinterpret_cast<uint4 *>(smem + msg_a_smem(KIND));           // 64 x K bf16 (W^T)
    TileGraph g = tile_graph_at<KIND>(smem + msg_a_smem(KIND) + (size_t)TC_N * K * 2);
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base;
    __shared__ int s_ok;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int N = a.N, ntile = (N + TC_M - 1) / TC_M;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(TC_N));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        asm volatile("tcgen05.fence::before_thread_sync;");
    }
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&mbar)), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_ok = 1;
    }
    // B tile: the packed image of W^T, copied as is
#pragma unroll 4
    for (int c = tid; c < TC_N * KC; c += TC_THREADS) Bs[c] = Wp[c];
    const int cg = item_cg(), c8 = cg * 8;
    uint32_t parity = 0;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x, parity ^= 1u) {
        const int n0 = tile * TC_M;
        load_tile_graph<KIND>(a, n0, g);
        float hs[ITEMS][8];
#pragma unroll
        for (int u = 0; u < ITEMS; u++) {
            const int r = item_row(u), n = n0 + r, nc = min(n, N - 1);
            float m0[8], m1[8];
            if (KIND == 0) {
                float h0[8], h1[8], h2[8];
                const float4 gr = a.egrad[nc];
                load8(a.hself + (size_t)nc * TC_N + c8, hs[u]);
                load8(a.hother + (size_t)g.tri[r] * TC_N + c8, h0);
                load8(a.hother + (size_t)g.tri[TC_M + r] * TC_N + c8, h1);
                load8(a.hother + (size_t)g.tri[2 * TC_M + r] * TC_N + c8, h2);
#pragma unroll
                for (int t = 0; t < 8; t++) {
                    const float2 m = msg_elem_grad(gr, h0[t], h1[t], h2[t], a.L);
                    m0[t] = m.x;
                    m1[t] = m.y;
                }
            } else {
                load8(a.hself + (size_t)nc * TC_N + c8, hs[u]);
                const int q0 = g.off[r], q1 = g.off[r + 1];
#pragma unroll
                for (int t = 0; t < 8; t++) m0[t] = 0.0f;
                // three incidences' rows in flight, summed in incidence order
                for (int q = q0; q < q1; q += 3) {
                    float h[3][8], ar[3];
#pragma unroll
                    for (int j = 0; j < 3; j++) {
                        const int qj = min(q + j, q1 - 1);
                        const int e = (g.inc_smem ? g.inc[qj - g.qbase] : a.vinc[qj]) >> 2;
                        ar[j] = g.inc_smem ? g.area[qj - g.qbase] : a.earea[e];
                        load8(a.hother + (size_t)e * TC_N + c8, h[j]);
                    }
#pragma unroll
                    for (int j = 0; j < 3; j++)
                        if (q + j < q1)
#pragma unroll
                            for (int t = 0; t < 8; t++) m0[t] = msg_vert_acc(m0[t], ar[j], h[j][t]);
                }
                const float inv = a.vinvA[nc];
#pragma unroll
                for (int t = 0; t < 8; t++) m0[t] = msg_vert_mean(m0[t], inv);
            }
            if (n >= N) {
#pragma unroll
                for (int t = 0; t < 8; t++) hs[u][t] = m0[t] = m1[t] = 0.0f;
            }
            As[tile_chunk(r, cg, 0)] = pack_bf16x8(hs[u]);
            As[tile_chunk(r, cg, 1)] = pack_bf16x8(m0);
            if (KIND == 0) As[tile_chunk(r, cg, 2)] = pack_bf16x8(m1);
        }
        // make the generic-proxy writes of the tiles visible to the tensor core (async proxy)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        const uint32_t tmem = tmem_base;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t a0 = smem_u32(As), b0 = smem_u32(Bs);
            constexpr uint32_t idesc = idesc_bf16_f32(TC_M, TC_N);
#pragma unroll
            for (int ks = 0; ks < K / 16; ks++)
                mma_bf16(tmem, umma_desc_sw(a0 + (ks >> 2) * TILE_BLOCK + (ks & 3) * 32, 16, 1024),
                         umma_desc(b0 + ks * 256, 128, KC * 128), idesc, ks);
            mma_commit(smem_u32(&mbar));
            if (!mma_wait(smem_u32(&mbar), parity, wait_cycles, status)) s_ok = 0;
        }
        __syncthreads();
        if (!s_ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        turn_tile(tmem, turn);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < ITEMS; u++) {
            const int r = item_row(u), n = n0 + r;
            float acc[8];
            load8_turned(turn + (size_t)r * TURN_LD + c8, cg, acc);
            if (n < N) {
                float y[8];
#pragma unroll
                for (int t = 0; t < 8; t++) {
                    y[t] = tanhf(__fadd_rn(acc[t], bias[c8 + t]));
                    hs[u][t] = __fadd_rn(hs[u][t], y[t]);
                }
                if (a.Y) store8(a.Y + (size_t)n * TC_N + c8, y);
                store8(a.hnext + (size_t)n * TC_N + c8, hs[u]);
            }
        }
        __syncthreads();     // the next tile overwrites the turned one
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TC_N));
    }
}

// ---------------------------------------------------------------------------------
// Backward of a message layer (inputs Z [N][K] holding bfloat16 values, K = 128 or 192; weights
// W [K][64]; incoming gradient dh [N][64] of h_next), one kernel:
//   dh    = dh_in + the gradient that the layers behind sent through their messages (gathered
//           here from g0, g1, where they are per row of the other kind)
//   dA    = dh (1 - Y^2)                                         (FP32)
//   G     = Z^T dA, column sums of dA: weight and bias gradient  (partial sums, see bwd_layer_part)
//   dZ    = dA W^T; dh_out = dh + dZ[:, 0:64]; m0, m1 = the other 64-wide blocks of dZ, the
//           gradients of the layer's messages
// dA is not a bfloat16 value, so each of its elements is split into two bfloat16 parts,
// hi = bf16(dA) and lo = bf16(dA - hi), which carry 16 significant bits, and both parts
// are multiplied: the products accumulate in FP32 in tensor memory.
//
// One staged tile serves both products: for dA W^T the rows are the M (K-major A operand), for
// Z^T dA they are the reduction, which reads the same tile as MN-major operands. Before, Z, dA and dZ
// went through memory in six kernels per layer: 7.1 GB per layer at level 8 (459k vertices, 910k
// triangles), 2.2 ms; here 2.9 GB, 0.79 ms. Bound by the latency of the gathers.
// TMEM: columns 0..127 dZ (the third block of a K = 192 layer takes columns 0..63 once they are
// read), 128..191 G of features 0..127, 192..255 G of features 64..191 (its upper half is kept).
template <int KIND, int INIT>
__global__ void __launch_bounds__(TC_THREADS, 2)
k_bwd_layer_tc(const BwdLayerArgs b, unsigned *__restrict__ status, long long wait_cycles)
{
    constexpr int K = KIND == 0 ? 3 * TC_N : 2 * TC_N;
    constexpr int DC = TC_N / 8;                   // core matrices along the channels of W
    constexpr int P = KIND == 0 ? 4 : 1;           // INIT: outputs behind the last layer
    const MsgLayerArgs &a = b.m;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint4 *Zs = reinterpret_cast<uint4 *>(smem);                              // 128 x K bf16
    float *turn = reinterpret_cast<float *>(smem);                            // over Zs (and Ah) after the MMAs
    uint4 *Ah = reinterpret_cast<uint4 *>(smem + (size_t)TC_M * K * 2);       // 128 x 64 bf16
    uint4 *Al = Ah + TC_M * DC;
    uint4 *Ws = Al + TC_M * DC;                                               // K x 64 bf16
    TileGraph g = tile_graph_at<KIND>(reinterpret_cast<unsigned char *>(Ws + K * DC));
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ uint32_t tmem_base;
    __shared__ int s_ok;
    __shared__ float s_w[P][TC_N];
    float *s_bias = turn;                                                     // [32][64], after the last tile
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = a.N, ntile = (N + TC_M - 1) / TC_M;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(256));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        asm volatile("tcgen05.fence::before_thread_sync;");
    }
    if (tid == 0) {
        for (int k = 0; k < 2; k++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&mbar[k])), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_ok = 1;
    }
    // W: chunk (row i = 8 ig + il, channels 8 kc .. + 7) is 16 contiguous bytes
    for (int c = tid; c < K * DC; c += TC_THREADS) {
        const int il = c & 7, kc = (c >> 3) % DC, ig = (c >> 3) / DC;
        Ws[c] = reinterpret_cast<const uint4 *>(b.W)[(size_t)(ig * 8 + il) * DC + kc];
    }
    if (INIT)
        for (int c = tid; c < P * TC_N; c += TC_THREADS)    // Wout is 64 x P
            s_w[c % P][c / P] = __bfloat162float(b.Wout[c]);
    const int cg = item_cg(), c8 = cg * 8;
    float bsum[8];
#pragma unroll
    for (int t = 0; t < 8; t++) bsum[t] = 0.0f;
    // The CTA's sums so far (G in tensor memory, bias in registers) to a partial sum; zeros after a wait that
    // gave up. The bias adds the 32 threads of a channel octet in a fixed order.
    auto flush = [&](int part) {
        {
            const int t0 = tid >> 3;
#pragma unroll
            for (int t = 0; t < 8; t++) {
                s_bias[t0 * TC_N + c8 + t] = bsum[t];
                bsum[t] = 0.0f;
            }
        }
        __syncthreads();
        float *out = b.partial + (size_t)part * ((size_t)K * TC_N + TC_N);
        if (tid < TC_N) {
            float x = 0.0f;
            for (int k = 0; k < 32; k++) x += s_bias[k * TC_N + tid];
            out[(size_t)K * TC_N + tid] = x;
        }
        // G rows i: features 0..127 from the first accumulator, 128..191 from the second's lanes 64..127
        asm volatile("tcgen05.fence::after_thread_sync;");
        const int quarter = warp & 3, half = warp >> 2;
#pragma unroll
        for (int mt = 0; mt < (KIND == 0 ? 2 : 1); mt++) {
            const int i = mt * 64 + quarter * 32 + lane;
#pragma unroll
            for (int q = 2 * half; q < 2 * half + 2; q++) {
                float v[16];
                if (s_ok) {
                    tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + 128 + 64 * mt + q * 16, v);
                } else {
#pragma unroll
                    for (int t = 0; t < 16; t++) v[t] = 0.0f;
                }
                if (mt == 0 || quarter >= 2) {
                    float4 *dst = reinterpret_cast<float4 *>(out + (size_t)i * TC_N + q * 16);
#pragma unroll
                    for (int t = 0; t < 16; t += 4) dst[t / 4] = make_float4(v[t], v[t + 1], v[t + 2], v[t + 3]);
                }
            }
        }
    };
    uint32_t parity = 0;
    int done = 0;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x, parity ^= 1u, done++) {
        const int n0 = tile * TC_M;
        load_tile_graph<KIND>(a, n0, g);
        float dh[ITEMS][8];
#pragma unroll
        for (int u = 0; u < ITEMS; u++) {
            const int r = item_row(u), n = n0 + r, nc = min(n, N - 1);
            float hs[8], m0[8], m1[8], y[8];
            load8(a.hself + (size_t)nc * TC_N + c8, hs);
            load8(b.Y + (size_t)nc * TC_N + c8, y);
            if (INIT) {
#pragma unroll
                for (int t = 0; t < 8; t++) {
                    float s = 0.0f;
#pragma unroll
                    for (int j = 0; j < P; j++) s = fmaf(b.dout[(size_t)nc * P + j], s_w[j][c8 + t], s);
                    dh[u][t] = s;
                }
            } else {
                load8(b.dh_in + (size_t)nc * TC_N + c8, dh[u]);
            }
            if (KIND == 0) {
                float h[3][8], d[3][8], w[3];
                const float4 gr = a.egrad[nc];
                const float ar = a.earea[nc];
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const int v = g.tri[k * TC_M + r];
                    load8(a.hother + (size_t)v * TC_N + c8, h[k]);
                    load8(b.g0 + (size_t)v * TC_N + c8, d[k]);
                    w[k] = a.vinvA[v];
                }
#pragma unroll
                for (int t = 0; t < 8; t++) {
                    const float2 m = msg_elem_grad(gr, h[0][t], h[1][t], h[2][t], a.L);
                    m0[t] = m.x;
                    m1[t] = m.y;
                    dh[u][t] += ar * (w[0] * d[0][t] + w[1] * d[1][t] + w[2] * d[2][t]);
                }
            } else {
                float ds[8];
#pragma unroll
                for (int t = 0; t < 8; t++) m0[t] = ds[t] = 0.0f;
                const int q1 = g.off[r + 1];
                for (int q = g.off[r]; q < q1; q++) {
                    const int ek = g.inc_smem ? g.inc[q - g.qbase] : a.vinc[q], e = ek >> 2, k = ek & 3;
                    const float ar = g.inc_smem ? g.area[q - g.qbase] : a.earea[e];
                    float h[8];
                    load8(a.hother + (size_t)e * TC_N + c8, h);
                    if (!INIT) {
                        float d0[8], d1[8];
                        load8(b.g0 + (size_t)e * TC_N + c8, d0);
                        load8(b.g1 + (size_t)e * TC_N + c8, d1);
                        const float4 gr = a.egrad[e];
                        const float gx = k == 0 ? gr.x : (k == 1 ? gr.z : -(gr.x + gr.z));
                        const float gy = k == 0 ? gr.y : (k == 1 ? gr.w : -(gr.y + gr.w));
#pragma unroll
                        for (int t = 0; t < 8; t++) ds[t] += gx * d0[t] + gy * d1[t];
                    }
#pragma unroll
                    for (int t = 0; t < 8; t++) m0[t] = msg_vert_acc(m0[t], ar, h[t]);
                }
                const float inv = a.vinvA[nc];
#pragma unroll
                for (int t = 0; t < 8; t++) {
                    m0[t] = msg_vert_mean(m0[t], inv);
                    if (!INIT) dh[u][t] += a.L * ds[t];
                }
            }
            float dA[8];
#pragma unroll
            for (int t = 0; t < 8; t++) dA[t] = dh[u][t] * (1.0f - y[t] * y[t]);
            if (n >= N) {
#pragma unroll
                for (int t = 0; t < 8; t++) hs[t] = m0[t] = m1[t] = dA[t] = 0.0f;
            }
            uint32_t wh[4], wl[4];
#pragma unroll
            for (int t = 0; t < 8; t += 2) {
                __nv_bfloat16 x0, x1, l0, l1;
                split_bf16(dA[t], x0, l0);
                split_bf16(dA[t + 1], x1, l1);
                wh[t / 2] = bf16x2_bits(x0, x1);
                wl[t / 2] = bf16x2_bits(l0, l1);
                bsum[t] += dA[t];
                bsum[t + 1] += dA[t + 1];
            }
            Zs[tile_chunk(r, cg, 0)] = pack_bf16x8(hs);
            Zs[tile_chunk(r, cg, 1)] = pack_bf16x8(m0);
            if (KIND == 0) Zs[tile_chunk(r, cg, 2)] = pack_bf16x8(m1);
            Ah[tile_chunk(r, cg, 0)] = make_uint4(wh[0], wh[1], wh[2], wh[3]);
            Al[tile_chunk(r, cg, 0)] = make_uint4(wl[0], wl[1], wl[2], wl[3]);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        const uint32_t tmem = tmem_base;
        const uint32_t z0 = smem_u32(Zs), ah = smem_u32(Ah), al = smem_u32(Al), w0 = smem_u32(Ws);
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;");
            // dZ[:, 0:128] = dA W[0:128]^T
            constexpr uint32_t id1 = idesc_bf16_f32(TC_M, 128);
#pragma unroll
            for (int ks = 0; ks < DC / 2; ks++) {
                const uint64_t bd = umma_desc(w0 + ks * 256, 128, DC * 128);
                mma_bf16(tmem, umma_desc_sw(ah + ks * 32, 16, 1024), bd, id1, ks > 0);
                mma_bf16(tmem, umma_desc_sw(al + ks * 32, 16, 1024), bd, id1, 1);
            }
            // G += Z^T dA: both operands MN-major (bits 15 and 16), 16 rows per step: the next 8 rows are
            // the next 1024-byte group, the next 64 features the next block of the tile
            constexpr uint32_t id2 = idesc_bf16_f32(TC_M, TC_N) | (1u << 15) | (1u << 16);
#pragma unroll
            for (int ks = 0; ks < TC_M / 16; ks++) {
                const uint64_t bh = umma_desc_sw(ah + ks * 2048, TILE_BLOCK, 1024);
                const uint64_t bl = umma_desc_sw(al + ks * 2048, TILE_BLOCK, 1024);
#pragma unroll
                for (int mt = 0; mt < (KIND == 0 ? 2 : 1); mt++) {
                    const uint64_t ad = umma_desc_sw(z0 + mt * TILE_BLOCK + ks * 2048, TILE_BLOCK, 1024);
                    mma_bf16(tmem + 128 + 64 * mt, ad, bh, id2, done % kGradTiles > 0 || ks > 0);
                    mma_bf16(tmem + 128 + 64 * mt, ad, bl, id2, 1);
                }
            }
            mma_commit(smem_u32(&mbar[0]));
            if (!mma_wait(smem_u32(&mbar[0]), parity, wait_cycles, status)) s_ok = 0;
        }
        __syncthreads();
        if (!s_ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        turn_tile(tmem, turn);
        asm volatile("tcgen05.fence::before_thread_sync;");
        __syncthreads();
        if (KIND == 0 && tid == 0) {
            // dZ[:, 128:192] into the columns that were just read (Zs and the turned tile are not touched)
            asm volatile("tcgen05.fence::after_thread_sync;");
            constexpr uint32_t id3 = idesc_bf16_f32(TC_M, TC_N);
#pragma unroll
            for (int ks = 0; ks < DC / 2; ks++) {
                const uint64_t bd = umma_desc(w0 + 16 * DC * 128 + ks * 256, 128, DC * 128);
                mma_bf16(tmem, umma_desc_sw(ah + ks * 32, 16, 1024), bd, id3, ks > 0);
                mma_bf16(tmem, umma_desc_sw(al + ks * 32, 16, 1024), bd, id3, 1);
            }
            mma_commit(smem_u32(&mbar[1]));
        }
        auto put = [&](float *out, bool add) {
#pragma unroll
            for (int u = 0; u < ITEMS; u++) {
                const int r = item_row(u), n = n0 + r;
                float v[8];
                load8_turned(turn + (size_t)r * TURN_LD + c8, cg, v);
                if (add)
#pragma unroll
                    for (int t = 0; t < 8; t++) v[t] += dh[u][t];
                if (n < N) store8(out + (size_t)n * TC_N + c8, v);
            }
            __syncthreads();
        };
        put(b.dh_out, true);
        turn_tile(tmem + 64, turn);
        __syncthreads();
        put(b.m0, false);
        if (KIND == 0) {
            if (tid == 0 && !mma_wait(smem_u32(&mbar[1]), parity, wait_cycles, status)) s_ok = 0;
            __syncthreads();
            if (!s_ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            turn_tile(tmem, turn);
            __syncthreads();
            put(b.m1, false);
        }
        if ((done + 1) % kGradTiles == 0 || tile + (int)gridDim.x >= ntile)
            flush(bwd_layer_part(gridDim.x, blockIdx.x, done));
        asm volatile("tcgen05.fence::before_thread_sync;");
    }
    if (!s_ok) {
        // a wait gave up: the rest of the CTA's partial sums are zeros
        for (; blockIdx.x + done * gridDim.x < ntile; done += kGradTiles - done % kGradTiles) {
            __syncthreads();
            flush(bwd_layer_part(gridDim.x, blockIdx.x, done));
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(256));
    }
}

__host__ __device__ constexpr size_t bwd_layer_smem(int kind)
{
    const size_t K = kind == 0 ? 3 * TC_N : 2 * TC_N;
    return (size_t)TC_M * K * 2 + 2 * (size_t)TC_M * TC_N * 2 + K * TC_N * 2 + graph_smem(kind);
}

}  // namespace

bool linear_tc_supported(int K, int P) { return P == TC_N && (K == 128 || K == 192); }

cudaError_t launch_bwd_layer_tc(const BwdLayerArgs &b, unsigned *status, cudaStream_t st)
{
    const int grid = bwd_layer_ctas(b.m.N);
    const size_t smem = bwd_layer_smem(b.m.kind);
    const bool init = b.dout != nullptr;
    const void *fn = b.m.kind == 0 ? (init ? (const void *)k_bwd_layer_tc<0, 1> : (const void *)k_bwd_layer_tc<0, 0>)
                                   : (init ? (const void *)k_bwd_layer_tc<1, 1> : (const void *)k_bwd_layer_tc<1, 0>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    long long cycles = 2000000000ll;   // about one second
    void *args[] = {const_cast<BwdLayerArgs *>(&b), &status, &cycles};
    return cudaLaunchKernel(fn, dim3(grid), dim3(TC_THREADS), args, smem, st);
}

size_t linear_tc_packed_elems(int K) { return (size_t)TC_N * K; }

cudaError_t pack_linear_tc(int K, const __nv_bfloat16 *W, __nv_bfloat16 *packed, cudaStream_t st)
{
    const int n = TC_N * K / 8;
    k_pack_wt<<<(n + 255) / 256, 256, 0, st>>>(K, W, reinterpret_cast<uint4 *>(packed));
    return cudaGetLastError();
}

cudaError_t launch_msg_layer_tc(const MsgLayerArgs &a, const __nv_bfloat16 *packed, const float *bias,
                                unsigned *status, cudaStream_t st)
{
    const uint4 *Wp = reinterpret_cast<const uint4 *>(packed);
    if (a.kind != 0 && a.kind != 1) return cudaErrorInvalidValue;
    const int grid = std::min((a.N + TC_M - 1) / TC_M, 3 * 152);   // three CTAs per SM
    if (grid == 0) return cudaSuccess;
    const size_t smem = msg_layer_smem(a.kind);
    const void *fn = a.kind == 0 ? (const void *)k_msg_layer_tc<0> : (const void *)k_msg_layer_tc<1>;
    // a per-kernel, per-device attribute: set on every launch (cheap) so that any device works
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // about one second of SM clock for the MMA completion wait
    if (a.kind == 0)
        k_msg_layer_tc<0><<<grid, TC_THREADS, smem, st>>>(a, Wp, bias, status, 2000000000ll);
    else
        k_msg_layer_tc<1><<<grid, TC_THREADS, smem, st>>>(a, Wp, bias, status, 2000000000ll);
    return cudaGetLastError();
}

}  // namespace sesw
