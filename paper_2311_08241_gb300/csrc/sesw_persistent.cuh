// Shared parts of the persistent step kernels of libsesw (sm_103a): kernel arguments,
// the tagged exchange of halo values through L2 and the shared-memory layout of a patch.
// Included by sesw_persistent.cu (the SE substep of Eq. 4.10), sesw_persistent_stream.cu
// (the same for patches whose state is streamed from L2) and sesw_persistent_sesm.cu (the
// SESM substep of Eqs. 4.7-4.8).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "sesw_device.cuh"
#include "sesw_internal.h"

namespace sesw {

namespace {

// A launch of the persistent kernels is cooperative, with every patch of a pack resident: one
// block per patch (k_persistent_sesm and the streaming kernels) or one team of warps of a
// block (k_persistent, k_persistent_sesm_teams). It takes n baroclinic steps of M substeps, its
// substeps counted on from step to step (the streaming kernels: n = 1).
//
// Exchange protocol. Every exchanged value (the elevation, or for SESM its AM4
// combination) is one 64-bit word holding a tag (high
// half) and its value (low half), written and read as a single relaxed access at GPU
// scope. The tag of substep m is base + m, where base is this launch's tag base. A
// reader uses a word only when its tag is the one it needs, re-reading it (bounded)
// otherwise, so it can never take a stale or a torn value, and no flag, fence or
// block-wide barrier is needed for the exchange. Within a launch, a block overwrites a
// parity buffer (tag m with m + 2) only after its substep m + 1, which needed every
// neighbour's tag-(m + 1) values; a neighbour writes those only after its own substep
// m, in which it read the tag-m values (the neighbour relation is symmetric: each patch
// reads halo values from every patch that reads from it). Between launches, the last
// patch of a pack to leave advances its base by n M + 1 (one word per pack in the flag buffer), so
// every word left by an earlier launch carries a tag that this launch never waits for
// and the buffers need no clearing. Tags wrap modulo 2^32; a wrapped tag could only
// match a word that no launch has rewritten since, and every launch rewrites every word
// that is read.
// Incidences of a vertex in the padded form (PArgs::inc8): at most this many per vertex.
constexpr int kIncWidth = 8;

struct PArgs {
    const int *patch_slot, *patch_own, *patch_int, *patch_v, *patch_halo, *halo_v;
    const int *vcsr_off;
    const uint32_t *vcsr;
    const int4 *sv;
    const ushort4 *sl;
    const uint2 *sf;           // where each corner's flux goes (DevMesh::slot_f)
    const uint32_t *vover;     // each vertex's overflow quads (DevMesh::v_over)
    const float4 *sg, *sc;
    const float4 *sk;          // step coefficients of each slot (DevMesh::slot_k)
    const float2 *R;
    float2 *U, *Umean;
    const float *inv_av;
    const float *patch_dt;
    const float *eta_in;
    float *eta_out;
    float *eta_sum;         // null, or sum over the substeps of eta^0 .. eta^{M-1} (own vertices)
    const float *W;         // null, or the freshwater flux of each vertex (Eq. 4.5)
    unsigned long long *xb[2];  // tagged elevation words (tag << 32 | float bits), per substep parity
    unsigned *flags;        // line 0: abort word; line 1 + 2k: tag base of pack k; line 2 + 2k: its exit count
    unsigned *status;
    const int *pack_patch;  // patch of each block: pack_patch[pack_base + blockIdx.x]
    int pack_base, pack_index;   // launches of one pack (the SESM kernels)
    const int *pack_off;         // [npack + 1] ranges of pack_patch
    int pack_first, pack_last;   // launches of a group of packs (the SE kernels)
    StepArgs a;
    int M, npatch;
    int nsteps;                  // baroclinic steps of this launch (k_persistent)
    int npb;                     // patches of the pack (launches of one pack)
    unsigned tmem_cols;          // tensor-memory columns of a block (k_persistent, a power of two)
    int row_quads, row_vertices; // 16-byte quads of a vertex's row of fluxes; vertices per quad array
    int over;                    // overflow quads (0: the rows hold every vertex's fluxes)
    int off_dummy, off_f01, off_f2, off_slo, off_hist, off_over, off_omask;   // k_persistent: see SeLayout
    int team_threads, team_smem; // threads and shared-memory bytes of each patch of a block (k_persistent)
    // shared-memory carve-up (CACHED), in bytes from the dynamic shared base
    int off_flux, off_g, off_c, off_r, off_l, off_off, off_csr, off_inv, off_halo;
    // inc8: the cached incidences are one row of 8 16-bit byte offsets per own vertex (into the
    // dynamic shared memory: the corner fluxes, padded with a zero word) at off_off, in place of
    // the CSR (offsets at off_off, entries at off_csr); zero_off: the zero word's byte offset
    int inc8, zero_off;
};

__device__ __forceinline__ unsigned long long ld_relaxed_gpu_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}

__device__ __forceinline__ void st_relaxed_gpu_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned ld_relaxed_gpu(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The flag buffer holds 2 npatch + 1 lines of 128 bytes (at most one pack per patch).
constexpr int kFlagStride = 32;

// The halo elevation of vertex v with tag `tag`, given the exchange word `w` already
// read from xs[v]: re-read until the word carries that tag. A wait that exceeds the
// budget (or finds the abort word set to this launch's `abort_val`) gives up: it sets
// the timeout bit and the abort word, which makes every other wait of the launch give
// up too, and clears `ok`; the value returned then is meaningless. (The first reads of
// a slot's corners are issued together by the caller, so that their latencies overlap.)
// The word is re-read at once, without a pause, and the abort word and the clock are looked at
// only every 64th time: a pause of 20 ns and an abort read in every turn made each turn two
// L2 round trips and cost the level-8 sphere 7 % of its step (1450 -> 1357 us per 4 steps from the
// pause alone).
__device__ __forceinline__ float halo_eta(const PArgs &P, const unsigned long long *xs, int v,
                                          unsigned long long w, unsigned tag, unsigned abort_val, bool &ok)
{
    if ((unsigned)(w >> 32) == tag) return __uint_as_float((unsigned)w);
    const unsigned *abort_word = P.flags;
    const long long t0 = clock64();
    for (unsigned turn = 1; ok; turn++) {
        w = ld_relaxed_gpu_u64(xs + v);
        if ((unsigned)(w >> 32) == tag) return __uint_as_float((unsigned)w);
        if ((turn & 63u) == 0 && (ld_relaxed_gpu(abort_word) == abort_val || clock64() - t0 > P.a.wait_cycles)) {
            ok = false;
            atomicOr(P.status, 2u);
            atomicExch(const_cast<unsigned *>(abort_word), abort_val);
        }
    }
    return 0.0f;
}

// ---------------------------------------------------------------------------------
// Tensor memory as the store of the slots' static data. An SM has 256 KB of it beside the
// 256 KB of registers and 228 KB of shared memory: 64 words for each of 1024 threads. A warp
// reads and writes only its own 32 lanes (32 (w % 4) .. + 31), which suits data that
// belongs to one thread: word k of a thread is its lane of column base + k. A tcgen05.ld of
// 8 words costs the shared-memory pipe nothing, where the same words from shared memory take
// 8 of its cycles per warp (the element pass and the vertex pass keep that pipe busy with
// the gathers of the elevation and the fluxes).
__device__ __forceinline__ void tmem_alloc(uint32_t *smem_slot, unsigned cols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(smem_slot)),
                 "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t base, unsigned cols)
{
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols));
}

__device__ __forceinline__ void tmem_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared memory by 32-bit address (so that no access goes through a generic one); ordered
// among themselves and by the teams' barriers.
__device__ __forceinline__ float lds(uint32_t a)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ float2 lds2(uint32_t a)
{
    float2 v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ float4 lds4(uint32_t a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a)
{
    unsigned short v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v)); }
__device__ __forceinline__ void sts2(uint32_t a, float2 v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y));
}

__device__ __forceinline__ void tmem_st2(uint32_t t, uint32_t a, uint32_t b)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(t), "r"(a), "r"(b) : "memory");
}

__device__ __forceinline__ void tmem_st4(uint32_t t, float a, float b, float c, float d)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(t), "f"(a), "f"(b), "f"(c),
                 "f"(d)
                 : "memory");
}

constexpr int kMaxTeams = 4;


// Barrier `bar` (1 ..) of a team of T threads (whole warps); barrier 0 is the block's.
__device__ __forceinline__ void team_sync(int bar, int T)
{
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(T) : "memory");
}

// Shared-memory address of a corner's flux: place e (21 bits of HostMesh::slot_f) of the patch's vertex l
// (v0: its first); corners that are not own vertices write to the lane's dummy word.
__device__ __forceinline__ uint32_t flux_place(const PArgs &P, uint32_t team, uint32_t dummy, uint32_t e, int v0,
                                               uint32_t l)
{
    if (e == 0x1fffffu) return dummy;
    if (e < 4u * (uint32_t)P.row_quads)
        return team + (uint32_t)P.off_flux + 16u * ((e >> 2) * (uint32_t)P.row_vertices + l) + 4u * (e & 3u);
    return team + (uint32_t)P.off_over + 16u * (P.vover[v0 + (int)l] & 0xffffu) + 4u * (e - (uint32_t)kRowFluxes);
}

// Clear the flux rows and overflow quads, and mark the own vertices that have any: one bit per vertex, so
// that a vertex pass looks at a vertex's overflow only where there is some. By the T threads of a team, which the
// caller synchronises afterwards.
__device__ __forceinline__ void clear_rows(const PArgs &P, unsigned char *smem_raw, int v0, int nown, int tid, int T)
{
    const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float4 *rows = reinterpret_cast<float4 *>(smem_raw + P.off_flux);
    for (int i = tid; i < P.row_quads * P.row_vertices; i += T) rows[i] = z;
    if (P.over == 0) return;
    float4 *over = reinterpret_cast<float4 *>(smem_raw + P.off_over);
    unsigned *mask = reinterpret_cast<unsigned *>(smem_raw + P.off_omask);
    for (int i = tid; i < P.over; i += T) over[i] = z;
    const unsigned in_row = (unsigned)(P.row_quads - kRowFluxes / 4);      // of the quads that v_over counts
    for (int i = tid; i < ((nown + 31) & ~31); i += T) {
        const unsigned m = __ballot_sync(0xffffffffu, i < nown && P.vover[v0 + min(i, nown - 1)] >> 16 > in_row);
        if ((i & 31) == 0) mask[i >> 5] = m;
    }
}

__device__ __forceinline__ float add4(float sum, const float4 c)
{
    return __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(sum, c.x), c.y), c.z), c.w);
}

// The sum of own vertex i's fluxes in incidence order (zeros behind the last). The first eight have both loads
// in flight before the sums (four steps of the 200k-vertex channel: 401 us in the loop, 380 us), but not in kernels
// without registers to spare (TIGHT: 7 slots per thread, sphere 1375 us in the loop, 1402 us).
template <bool TIGHT>
__device__ __forceinline__ float row_flux_sum(const PArgs &P, uint32_t team, int v0, int i)
{
    uint32_t row = team + (uint32_t)P.off_flux + 16u * (uint32_t)i;
    const uint32_t step = 16u * (uint32_t)P.row_vertices;
    float sum = 0.0f;
    if (TIGHT) {
        for (int k = 0; k < P.row_quads; k++, row += step) sum = add4(sum, lds4(row));
    } else {
        const float4 a = lds4(row), b = lds4(row + step);
        sum = add4(add4(sum, a), b);
        if (P.row_quads > 2) {
            sum = add4(sum, lds4(row + 2u * step));
            if (P.row_quads > 3) sum = add4(sum, lds4(row + 3u * step));
        }
    }
    if (P.over && (lds_u32(team + (uint32_t)P.off_omask + 4u * (uint32_t)(i >> 5)) >> (i & 31)) & 1u) {
        const uint32_t o = __ldg(P.vover + v0 + i);
        for (uint32_t k = (uint32_t)P.row_quads - kRowFluxes / 4; k < o >> 16; k++)
            sum = add4(sum, lds4(team + (uint32_t)P.off_over + 16u * ((o & 0xffffu) + k)));
    }
    return sum;
}

// A slot's static data: gradients, step coefficients (DevMesh::slot_k), forcing, and the
// shared-memory addresses of its corners' elevations and of the places of its three fluxes.
struct SlotData {
    float4 g, c;
    float2 r;
    uint32_t a0, a1, a2, f0, f1, f2;
};

// The data of one slot as a thread's words hold it, waited for. No memory clobber: what a launch
// stores in tensor memory is stored before its first barrier and never changes.
__device__ __forceinline__ void tmem_ld16(uint32_t t, SlotData &q)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15}, [%16];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=f"(q.g.x), "=f"(q.g.y), "=f"(q.g.z), "=f"(q.g.w), "=f"(q.c.x), "=f"(q.c.y), "=f"(q.c.z),
                   "=f"(q.c.w), "=f"(q.r.x), "=f"(q.r.y), "=r"(q.a0), "=r"(q.a1), "=r"(q.a2), "=r"(q.f0), "=r"(q.f1),
                   "=r"(q.f2)
                 : "r"(t));
}

__device__ __forceinline__ void tmem_ld12(uint32_t t8, uint32_t t4, SlotData &q, uint32_t &l01, uint32_t &l2)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%12];\n"
                 "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8, %9, %10, %11}, [%13];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=f"(q.g.x), "=f"(q.g.y), "=f"(q.g.z), "=f"(q.g.w), "=f"(q.c.x), "=f"(q.c.y), "=f"(q.c.z),
                   "=f"(q.c.w), "=f"(q.r.x), "=f"(q.r.y), "=r"(l01), "=r"(l2)
                 : "r"(t8), "r"(t4));
}

__device__ __forceinline__ void tmem_ld10(uint32_t t8, uint32_t t2, SlotData &q, uint32_t &l01, uint32_t &l2)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%10];\n"
                 "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%8, %9}, [%11];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=f"(q.g.x), "=f"(q.g.y), "=f"(q.g.z), "=f"(q.g.w), "=f"(q.c.x), "=f"(q.c.y), "=f"(q.c.z),
                   "=f"(q.c.w), "=r"(l01), "=r"(l2)
                 : "r"(t8), "r"(t2));
}

// Words 4, 2, 2 and 1 of a thread at four places, waited for (a streamed SESM slot's state).
__device__ __forceinline__ void tmem_ld9(uint32_t t4, uint32_t t2, uint32_t p2, uint32_t p1, float *f6, uint32_t &a,
                                         uint32_t &b, uint32_t &c)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%9];\n"
                 "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%4, %5}, [%10];\n"
                 "tcgen05.ld.sync.aligned.32x32b.x2.b32 {%6, %7}, [%11];\n"
                 "tcgen05.ld.sync.aligned.32x32b.x1.b32 {%8}, [%12];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=f"(f6[0]), "=f"(f6[1]), "=f"(f6[2]), "=f"(f6[3]), "=f"(f6[4]), "=f"(f6[5]), "=r"(a), "=r"(b),
                   "=r"(c)
                 : "r"(t4), "r"(t2), "r"(p2), "r"(p1));
}

__device__ __forceinline__ void tmem_ld8(uint32_t t8, SlotData &q)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=f"(q.g.x), "=f"(q.g.y), "=f"(q.g.z), "=f"(q.g.w), "=f"(q.c.x), "=f"(q.c.y), "=f"(q.c.z),
                   "=f"(q.c.w)
                 : "r"(t8));
}

// Where the data of a thread's SPT slots live. Up to 4 slots per thread each slot has 16 words
// of tensor memory: everything, with the shared-memory offsets ready to use, so that a slot's
// update spends no instruction on addresses. With 5, 12 words (offsets of the corners packed as
// 16-bit word indices); with 6, 10 words (without the forcing); with 7 and 8, 8 words and the
// corners of the first four slots of 7. From 5 slots per thread the places of the fluxes are
// 16-bit word indices in shared memory; the forcing and corners left over come from L2
// (coalesced, their addresses known ahead). load is called by whole warps; s is the slot's
// index in the mesh, i in the patch, team the address of the team's shared memory.
template <int SPT>
struct TmemSlots {
    static constexpr int kWords = SPT <= 4 ? 16 * SPT : (SPT <= 6 ? 60 : 64);
    static constexpr bool kTmem = true;
    static constexpr bool kFluxShared = SPT >= 5;
    __device__ static __forceinline__ void store(uint32_t tm, int j, const SlotData &q)
    {
        auto f = [](uint32_t x) { return __uint_as_float(x); };
        const int b = (SPT <= 4 ? 16 : 8) * j;
        tmem_st4(tm + b, q.g.x, q.g.y, q.g.z, q.g.w);
        tmem_st4(tm + b + 4, q.c.x, q.c.y, q.c.z, q.c.w);
        const uint32_t l01 = (q.a0 >> 2) | (q.a1 << 14), l2 = q.a2;
        if (SPT <= 4) {
            tmem_st4(tm + b + 8, q.r.x, q.r.y, f(q.a0), f(q.a1));
            tmem_st4(tm + b + 12, f(q.a2), f(q.f0), f(q.f1), f(q.f2));
        } else if (SPT == 5) {
            tmem_st4(tm + 8 * SPT + 4 * j, q.r.x, q.r.y, f(l01), f(l2));
        } else if (SPT == 6 || (SPT == 7 && j < 4)) {
            tmem_st2(tm + 8 * SPT + 2 * j, l01, l2);
        }
    }
    __device__ static __forceinline__ SlotData load(uint32_t tm, int j, const PArgs &P, int s, int i, uint32_t team)
    {
        SlotData q;
        if (SPT <= 4) {
            tmem_ld16(tm + 16 * j, q);
            return q;
        }
        uint32_t l01, l2;
        if (SPT >= 6) q.r = __ldg(P.R + s);
        if (SPT == 5) {
            tmem_ld12(tm + 8 * j, tm + 8 * SPT + 4 * j, q, l01, l2);
        } else if (SPT == 6 || (SPT == 7 && j < 4)) {
            tmem_ld10(tm + 8 * j, tm + 8 * SPT + 2 * j, q, l01, l2);
        }
        if (SPT <= 6 || (SPT == 7 && j < 4)) {
            q.a0 = (l01 & 0xffffu) * 4u;
            q.a1 = (l01 >> 16) * 4u;
            q.a2 = l2;
        } else {
            const uint2 l = __ldg(reinterpret_cast<const uint2 *>(P.sl + s));
            tmem_ld8(tm + 8 * j, q);
            q.a0 = team + (l.x & 0xffffu) * 4u;
            q.a1 = team + (l.x >> 16) * 4u;
            q.a2 = team + (l.y & 0xffffu) * 4u;
        }
        const uint32_t f01 = lds_u32(team + P.off_f01 + 4 * i);
        q.f0 = (f01 & 0xffffu) * 4u;
        q.f1 = (f01 >> 16) * 4u;
        q.f2 = lds_u16(team + P.off_f2 + 2 * i) * 4u;
        return q;
    }
};

// The same interface with everything read from L2 and the fluxes slot by slot (three words each)
// at P.off_flux.
template <int SPT>
struct GlobalSlots {
    static constexpr bool kTmem = false;
    static constexpr bool kFluxShared = false;
    __device__ static __forceinline__ void store(uint32_t, int, const SlotData &) {}
    __device__ static __forceinline__ SlotData load(uint32_t, int, const PArgs &P, int s, int i, uint32_t team)
    {
        SlotData q;
        const ushort4 l = P.sl[s];
        q.g = P.sg[s];
        q.c = P.sk[s];
        q.r = P.R[s];
        q.a0 = team + 4u * l.x;
        q.a1 = team + 4u * l.y;
        q.a2 = team + 4u * l.z;
        q.f0 = team + (uint32_t)P.off_flux + 12u * (uint32_t)i;
        q.f1 = q.f0 + 4u;
        q.f2 = q.f0 + 8u;
        return q;
    }
};

// Tensor-memory columns of a block of `threads` threads with `words` words each: ceil(warps / 4)
// column groups, rounded up to the allocation unit (a power of two of at least 32).
inline unsigned tmem_columns(int threads, int words)
{
    const int need = ((threads / 32 + 3) / 4) * words;
    unsigned c = 32;
    while ((int)c < need) c *= 2;
    return c;
}

// Shared memory a block must take so that its share of the SM's shared memory is its share of
// the SM's 512 tensor-memory columns, less the 1 KB that the system reserves per block and at
// most 1/32 (and 1 KB) of rounding. Blocks of different launches (other contexts, other streams)
// may share an SM; columns come in units of 32 = 1/16 of the SM, so blocks of the persistent kernels that
// fit its shared memory together always find their columns free, and none of them can wait for columns
// that another persistent launch holds. The surrogate's kernels take columns without this floor (two vertex
// blocks of the backward pass hold all 512 with 190 KB of shared memory), but their blocks wait for no
// other block and give their columns back at their end, so a wait for those ends too.
inline size_t tmem_smem_floor(unsigned cols, size_t smem_per_sm)
{
    const size_t share = smem_per_sm / 512 * cols;
    return share - 1024 - std::min<size_t>(1024, share / 32);
}

// Copy the incidences of a patch's own vertices into shared memory (cached layouts): with
// P.inc8, one row of kIncWidth 16-bit byte offsets (inc8 = 1) or word indices (inc8 = 2) per
// vertex, pointing at its corner fluxes in incidence order and padded with the zero word; else
// the CSR with flux indices 3 * slot + corner. Also clears the zero word. Run by T threads (tid
// 0 .. T - 1) on the shared memory of one patch; the caller synchronises them afterwards.
__device__ __forceinline__ void cache_incidences(const PArgs &P, unsigned char *smem_raw, int v0, int nown, int tid,
                                                 int T)
{
    const int c0 = P.vcsr_off[v0], ncsr = P.vcsr_off[v0 + nown] - c0;
    if (P.inc8) {
        uint4 *rows = reinterpret_cast<uint4 *>(smem_raw + P.off_off);
        for (int i = tid; i < nown; i += T) {
            const int k0 = P.vcsr_off[v0 + i], deg = P.vcsr_off[v0 + i + 1] - k0;
            unsigned h[kIncWidth];
#pragma unroll
            for (int k = 0; k < kIncWidth; k++) {
                unsigned off = (unsigned)P.zero_off;
                if (k < deg) {
                    const uint32_t q = P.vcsr[k0 + k];
                    off = (unsigned)P.off_flux + 4u * (3u * (q >> 2) + (q & 3u));
                }
                h[k] = P.inc8 == 2 ? off >> 2 : off;
            }
            rows[i] = make_uint4(h[0] | (h[1] << 16), h[2] | (h[3] << 16), h[4] | (h[5] << 16), h[6] | (h[7] << 16));
        }
        if (tid == 0) *reinterpret_cast<float *>(smem_raw + P.zero_off) = 0.0f;
    } else {
        unsigned short *s_off = reinterpret_cast<unsigned short *>(smem_raw + P.off_off);
        unsigned short *s_csr = reinterpret_cast<unsigned short *>(smem_raw + P.off_csr);
        for (int i = tid; i <= nown; i += T) s_off[i] = (unsigned short)(P.vcsr_off[v0 + i] - c0);
        for (int k = tid; k < ncsr; k += T) {
            const uint32_t q = P.vcsr[c0 + k];
            s_csr[k] = (unsigned short)(3u * (q >> 2) + (q & 3u));
        }
    }
}

// Sum of the corner fluxes of own vertex i in its incidence order (cached layouts; see
// cache_incidences). The padded form adds zeros after the last incidence, which leaves the
// sum unchanged.
__device__ __forceinline__ float cached_flux_sum(const PArgs &P, const unsigned char *smem_raw, int i)
{
    float sum = 0.0f;
    if (P.inc8 == 1) {
        const uint4 q = reinterpret_cast<const uint4 *>(smem_raw + P.off_off)[i];
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            sum = __fadd_rn(sum, *reinterpret_cast<const float *>(smem_raw + (w[k] & 0xffffu)));
            sum = __fadd_rn(sum, *reinterpret_cast<const float *>(smem_raw + (w[k] >> 16)));
        }
    } else if (P.inc8 == 2) {
        const uint4 q = reinterpret_cast<const uint4 *>(smem_raw + P.off_off)[i];
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
        const float *words = reinterpret_cast<const float *>(smem_raw);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            sum = __fadd_rn(sum, words[w[k] & 0xffffu]);
            sum = __fadd_rn(sum, words[w[k] >> 16]);
        }
    } else {
        const unsigned short *s_off = reinterpret_cast<const unsigned short *>(smem_raw + P.off_off);
        const unsigned short *s_csr = reinterpret_cast<const unsigned short *>(smem_raw + P.off_csr);
        const float *sflux = reinterpret_cast<const float *>(smem_raw + P.off_flux);
        const int k1 = s_off[i + 1];
        for (int k = s_off[i]; k < k1; k++) sum = __fadd_rn(sum, sflux[s_csr[k]]);
    }
    return sum;
}

inline size_t flag_bytes(int npatch) { return sizeof(unsigned) * (2 * (size_t)npatch + 1) * kFlagStride; }


struct SmemLayout {
    int off_flux, off_g, off_c, off_r, off_l, off_off, off_csr, off_inv, off_halo;
    int inc8, zero_off;
    size_t total_plain;     // elevation, corner fluxes and the zero word
    size_t total_cached;    // ... the vertices' data (1/A_v, halo ids, incidences) and the slots' static data
};

inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// Shared-memory layout of a patch: [elevation of own and halo vertices | corner fluxes, zero
// word | 1/A_v, halo ids, incidences | per slot: gradients, coefficients, forcing, corners].
// The SESM kernel that keeps everything on chip uses the whole layout, the streaming kernels only
// the first part (the kernels with tensor memory have their own, se_layout and sesm_layout).
inline SmemLayout smem_layout(const PatchMax &m)
{
    SmemLayout L;
    size_t o = align16(sizeof(float) * (size_t)m.local);
    L.off_flux = (int)o;
    // the corner fluxes, then one zero word (the padding target of the padded incidence rows)
    L.zero_off = (int)(o + sizeof(float) * 3 * (size_t)m.slots);
    o = align16(o + sizeof(float) * (3 * (size_t)m.slots + 1));
    L.total_plain = o;
    L.off_inv = (int)o;
    o = align16(o + sizeof(float) * (size_t)m.vertices);
    L.off_halo = (int)o;
    o = align16(o + sizeof(int) * (size_t)m.halo);
    L.off_off = (int)o;
    const size_t csr_end = align16(align16(o + sizeof(unsigned short) * ((size_t)m.vertices + 1)) +
                                   sizeof(unsigned short) * (size_t)m.csr);
    L.off_csr = (int)align16(o + sizeof(unsigned short) * ((size_t)m.vertices + 1));
    // padded rows when every vertex has at most kIncWidth incidences: 16-bit byte offsets of the
    // corner fluxes when they fit 16 bits (inc8 = 1), else 16-bit word indices (inc8 = 2); they
    // take the place of the CSR
    L.inc8 = m.deg > kIncWidth ? 0 : (L.zero_off + 4 <= 65535 ? 1 : (L.zero_off / 4 + 1 <= 65535 ? 2 : 0));
    const size_t inc_end = o + sizeof(unsigned short) * kIncWidth * (size_t)m.vertices;
    o = L.inc8 ? align16(inc_end) : csr_end;
    L.off_g = (int)o;
    o += sizeof(float4) * (size_t)m.slots;
    L.off_c = (int)o;
    o += sizeof(float4) * (size_t)m.slots;
    L.off_r = (int)o;
    o = align16(o + sizeof(float2) * (size_t)m.slots);
    L.off_l = (int)o;
    o = align16(o + sizeof(ushort4) * (size_t)m.slots);
    L.total_cached = o;
    return L;
}


inline PArgs make_pargs(const DevMesh &m, const DevState &s, const StepArgs &a, int M, int parity, const PatchMax &mx)
{
    PArgs P;
    P.patch_slot = m.patch_slot;
    P.patch_own = m.patch_own;
    P.patch_int = m.patch_int;
    P.patch_v = m.patch_v;
    P.patch_halo = m.patch_halo;
    P.halo_v = m.halo_v;
    P.vcsr_off = m.vcsr_off;
    P.vcsr = m.vcsr;
    P.sv = m.slot_v;
    P.sl = m.slot_l;
    P.sf = m.slot_f;
    P.vover = m.v_over;
    P.over = 0;
    P.sg = m.slot_g;
    P.sc = m.slot_c;
    P.sk = m.slot_k;
    P.R = s.R;
    P.U = s.U;
    P.Umean = s.Umean;
    P.inv_av = m.inv_av;
    P.patch_dt = m.patch_dt;
    P.eta_in = s.eta[parity];
    P.eta_out = s.eta[parity ^ 1];
    P.eta_sum = s.eta_sum;
    P.W = s.W;
    P.xb[0] = reinterpret_cast<unsigned long long *>(s.xbuf[0]);
    P.xb[1] = reinterpret_cast<unsigned long long *>(s.xbuf[1]);
    P.flags = s.flags;
    P.status = s.status;
    P.a = a;
    P.M = M;
    P.nsteps = 1;
    P.npb = 0;
    P.tmem_cols = 0;
    P.team_threads = P.team_smem = 0;
    P.npatch = m.npatch;
    const SmemLayout L = smem_layout(mx);
    P.off_flux = L.off_flux;
    P.off_g = L.off_g;
    P.off_c = L.off_c;
    P.off_r = L.off_r;
    P.off_l = L.off_l;
    P.off_off = L.off_off;
    P.off_csr = L.off_csr;
    P.off_inv = L.off_inv;
    P.off_halo = L.off_halo;
    P.inc8 = L.inc8;
    P.zero_off = L.zero_off;
    P.pack_patch = m.pack_patch;
    P.pack_base = 0;
    P.pack_index = 0;
    P.pack_off = m.pack_off_d;
    P.pack_first = 0;
    P.pack_last = 0;
    return P;
}

// Shared memory of one team, from its largest patch: elevation of own and halo vertices; the
// fluxes, then 32 dummy words; 1/A_v and halo ids; from 5 slots per thread the flux places, from
// 6 the low parts of the compensated sums; where a vertex has more than kRowFluxes triangles, the
// overflow quads and the vertices' marks. Vertex-major fluxes (cached): each own vertex has a row
// of 8 to 16 words (quad k of all vertices in array k), which the
// element pass fills and the vertex pass reads 16 bytes at a time, in the place of an
// index row and eight dependent 4-byte reads (the reads' bank conflicts kept the
// shared-memory pipe busy longer than the element pass). Rows as wide as the largest degree gave
// every vertex that width: a level-8 sphere with a vertex of nine triangles took 264 KB and left the chip
// (four steps of a 468k-vertex basin, every 144th vertex of nine triangles: 1715 us streamed, 1200 us here).
// Not cached: three words per slot.
struct SeLayout {
    size_t flux, dummy, inv, halo, f01, f2, slo, hist, over, omask, total;
    int quads, nover;            // width of the rows; overflow quads beside them
};

// wide: rows for the largest degree up to 16, with overflow quads only beyond that; else rows of
// kRowFluxes.
inline SeLayout se_layout(const PatchMax &m, int spt, int cached, int wide)
{
    SeLayout L{};
    const size_t slots = ((size_t)m.slots + 31) & ~(size_t)31;   // whole warps
    size_t o = align16(sizeof(float) * (size_t)m.local);
    L.flux = o;
    if (!cached) {
        L.total = align16(o + 12 * slots);
        return L;
    }
    L.quads = wide ? std::min(4, std::max(kRowFluxes / 4, (m.deg + 3) / 4)) : kRowFluxes / 4;
    L.nover = m.deg > 4 * L.quads ? m.over : 0;
    o += 16 * (size_t)L.quads * (size_t)m.vertices;
    L.over = o;
    o += 16 * (size_t)L.nover;
    L.dummy = o;
    o += 128;
    L.inv = o;
    o = align16(o + sizeof(float) * (size_t)m.vertices);
    L.halo = o;
    o = align16(o + sizeof(int) * (size_t)m.halo);
    L.f01 = o;
    if (spt >= 5) o += 4 * slots;
    L.f2 = o;
    if (spt >= 5) o = align16(o + 2 * slots);
    L.slo = o;
    if (spt >= 6) o += sizeof(float2) * slots;
    L.omask = o;
    if (L.nover > 0) o += 4 * (((size_t)m.vertices + 31) / 32);
    L.total = align16(o);
    return L;
}

// The SESM teams: elevation (eta_AM) of own and halo vertices, fluxes, vertices' data as above, the
// three levels of elevation that each own vertex keeps, and U_AB of the slots.
inline SeLayout sesm_layout(const PatchMax &m, int wide)
{
    SeLayout L = se_layout(m, 1, 1, wide);
    L.hist = L.total;
    L.slo = align16(L.hist + 3 * sizeof(float) * (size_t)m.vertices);
    L.total = L.slo + sizeof(float2) * (((size_t)m.slots + 31) & ~(size_t)31);
    return L;
}

inline void set_layout(PArgs &P, const SeLayout &L, const PatchMax &m)
{
    P.off_flux = (int)L.flux;
    P.off_dummy = (int)L.dummy;
    P.off_inv = (int)L.inv;
    P.off_halo = (int)L.halo;
    P.off_f01 = (int)L.f01;
    P.off_f2 = (int)L.f2;
    P.off_slo = (int)L.slo;
    P.off_hist = (int)L.hist;
    P.off_over = (int)L.over;
    P.off_omask = (int)L.omask;
    P.over = L.nover;
    P.row_quads = L.quads;
    P.row_vertices = m.vertices;
}

}  // namespace

}  // namespace sesw
