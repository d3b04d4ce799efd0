// The persistent step kernel of libsesw (sm_103a): one cooperative launch runs all M
// substeps of Eq. (4.10) of one or several baroclinic steps, with the time-mean transport of
// Eq. (4.12) and the freshwater flux of Eq. (4.5).
#include <type_traits>

#include "sesw_persistent.cuh"

namespace sesw {

namespace {

// ---------------------------------------------------------------------------------
// Persistent kernel: one launch runs P.nsteps baroclinic steps (M substeps each) with one block
// per SM, all blocks resident (cooperative launch). A block holds one to four teams of warps
// (blocks_per_sm in the interface), each of which runs a patch of its own: own barriers, own
// share of the block's shared and tensor memory, nothing exchanged with the other teams but
// through the exchange buffers, so that one team's barriers and halo waits are filled by
// the others. (Teams and not blocks, because a kernel that uses tensor memory gets one block
// per SM from a cooperative launch.) A team keeps the elevation of its own
// and halo vertices, the per-corner fluxes, and its vertices' data (incidences, 1/A_v, halo
// ids) in shared memory, the transport and the compensated flux sum of its slots in registers,
// and the slots' static data (gradients, step coefficients, and as far as it reaches the
// corner indices and the forcing) in tensor memory, for all substeps.
//
// Substep m: update the interior slots (corners all own vertices); update the other
// slots, whose halo elevation comes from the exchange buffer of parity m; vertex pass;
// write the own vertices' new elevation to the exchange buffer of parity m+1 (the
// exchange protocol is described in sesw_persistent.cuh). One thread per halo vertex requests
// its tagged word before the interior rounds and stores its value to shared memory after them.
//
// Vertex order. Mesh preparation puts the vertices that other patches read first in
// each patch, so the vertex pass publishes them in its first round.
//
// Steps. The last substep of a step is followed at once by the first of the next: its
// elevation is exchanged like any other, and only the sums restart. A launch of n steps loads
// the patch once instead of n times.

__device__ __forceinline__ float4 slot_coef(const float4 c, float g, float dt)
{
    const float aa = __fmul_rn(c.z, __fmul_rn(0.5f, dt));
    return make_float4(__fmul_rn(dt, c.x), __fmul_rn(g, c.y), aa, __frcp_rn(__fmaf_rn(aa, aa, 1.0f)));
}

// The step coefficients of every slot, once per parameter change: the persistent kernels
// read them instead of forming them each substep (or in each launch's prologue).
__global__ void k_slot_coef(int npatch, const int *__restrict__ patch_slot, const float *__restrict__ patch_dt,
                            const float4 *__restrict__ sc, float g, float4 *__restrict__ sk)
{
    for (int p = blockIdx.x; p < npatch; p += gridDim.x) {
        const float dt = patch_dt[p];
        for (int s = patch_slot[p] + threadIdx.x; s < patch_slot[p + 1]; s += blockDim.x) sk[s] = slot_coef(sc[s], g, dt);
    }
}

// The P.nsteps baroclinic steps of patch p, this team's patch in pack `pack` (of npb patches).
// tm: this warp's tensor-memory words (see TmemSlots); smem_raw: the team's shared memory;
// tid, T: the thread in the team and the team's size; bar: the team's barrier.
// EXTRA: the optional per-vertex terms (freshwater flux, step-mean elevation) may be set;
// the instantiation without them carries neither load nor branch.
template <int SPT, int NONLIN, int CACHED, int EXTRA>
__device__ __forceinline__ void persistent_patch(const PArgs &P, const int p, const int pack, const int npb,
                                                 const uint32_t tm, unsigned char *smem_raw, int &s_abort,
                                                 const int tid, const int T, const int bar)
{
    using TS = std::conditional_t<CACHED != 0, TmemSlots<SPT>, GlobalSlots<SPT>>;
    // the low parts of the compensated sums live in shared memory where registers run short
    constexpr bool kSloShared = CACHED != 0 && SPT >= 6;
    const uint32_t team = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const int wbase = __shfl_sync(0xffffffffu, tid & ~31, 0);   // the warp's first thread
    const int s0 = P.patch_slot[p], ns = P.patch_slot[p + 1] - s0;
    const int nsp = (ns + 31) & ~31;    // slots of whole warps
    const int nown_s = P.patch_own[p], nint = P.patch_int[p];
    const int v0 = P.patch_v[p], nown = P.patch_v[p + 1] - v0;
    const int hb = P.patch_halo[p], nhalo = P.patch_halo[p + 1] - hb;
    const StepArgs a = P.a;
    const float dt = P.patch_dt[p];
    unsigned *base_word = P.flags + (size_t)(1 + 2 * pack) * kFlagStride;
    unsigned *exit_count = base_word + kFlagStride;
    const unsigned base = ld_relaxed_gpu(base_word);
    const unsigned abort_val = base + 1u == 0u ? 1u : base + 1u;   // never 0, unique per launch

    float *seta = reinterpret_cast<float *>(smem_raw);
    float *s_inv = reinterpret_cast<float *>(smem_raw + P.off_inv);
    int *s_halo = reinterpret_cast<int *>(smem_raw + P.off_halo);
    const uint32_t slo_at = team + (uint32_t)P.off_slo;

    for (int i = tid; i < nown; i += T) seta[i] = P.eta_in[v0 + i];
    for (int i = tid; i < nhalo; i += T) seta[nown + i] = P.eta_in[P.halo_v[hb + i]];
    if (CACHED) {
        clear_rows(P, smem_raw, v0, nown, tid, T);
        for (int i = tid; i < nown; i += T) s_inv[i] = P.inv_av[v0 + i];
        for (int i = tid; i < nhalo; i += T) s_halo[i] = P.halo_v[hb + i];
    }
    const int *hid = CACHED ? s_halo : P.halo_v + hb;
    if (tid == 0) s_abort = 0;
    // Threads without a slot in their last round hold an all-zero one, so that the update needs
    // no per-thread condition. The fluxes of corners that are not own vertices, and of such empty
    // slots, go to one of 32 dummy words (one per lane).
    const uint32_t dummy = team + (uint32_t)P.off_dummy + 4u * (tid & 31);
    float2 u[SPT], shi[SPT], slo[kSloShared ? 1 : SPT];
#pragma unroll
    for (int j = 0; j < SPT; j++) {
        const int i = tid + j * T;
        const bool in = i < ns;
        const int s = s0 + (in ? i : 0);
        if (TS::kTmem) {
            const ushort4 l = P.sl[s];
            SlotData q;
            q.g = in ? P.sg[s] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            q.c = in ? P.sk[s] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            q.r = in ? P.R[s] : make_float2(0.0f, 0.0f);
            q.a0 = team + 4u * l.x;
            q.a1 = team + 4u * l.y;
            q.a2 = team + 4u * l.z;
            const uint2 f = in ? P.sf[s] : make_uint2(0xffffffffu, 0x7fffffffu);
            q.f0 = flux_place(P, team, dummy, f.x & 0x1fffffu, v0, l.x);
            q.f1 = flux_place(P, team, dummy, (f.x >> 21) | ((f.y & 0x3ffu) << 11), v0, l.y);
            q.f2 = flux_place(P, team, dummy, (f.y >> 10) & 0x1fffffu, v0, l.z);
            TS::store(tm, j, q);
            if (TS::kFluxShared && i < nsp) {
                *reinterpret_cast<uint32_t *>(smem_raw + P.off_f01 + 4 * i) = (q.f0 >> 2) | (q.f1 << 14);
                *reinterpret_cast<unsigned short *>(smem_raw + P.off_f2 + 2 * i) = (unsigned short)(q.f2 >> 2);
            }
        }
        u[j] = in ? P.U[s] : make_float2(0.0f, 0.0f);
        shi[j] = make_float2(0.0f, 0.0f);
        if (!kSloShared) slo[j] = make_float2(0.0f, 0.0f);
        if (kSloShared && i < nsp) sts2(slo_at + 8 * i, make_float2(0.0f, 0.0f));
    }
    if (TS::kTmem) tmem_wait_st();
    team_sync(bar, T);

    const float one_p_theta = __fadd_rn(1.0f, a.theta);
    bool ok = true;
    // Update the slots [lo, hi) (multiples of 32, whole warps): transport (Eq. 4.10, first row),
    // theta-weighted flux into the corners' cells, compensated sum. Guest copies sum as well
    // (their sums are not used): a branch around it would cost the owned ones more.
    auto elements = [&](int lo, int hi) {
#pragma unroll
        for (int j = 0; j < SPT; j++) {
            const int w = wbase + j * T;
            if (w >= lo && w < hi) {
                const int i = tid + j * T;
                const SlotData q = TS::load(tm, j, P, s0 + min(i, ns - 1), i, team);
                const float e0 = lds(q.a0), e1 = lds(q.a1), e2 = lds(q.a2);
                const float2 F = se_transport<NONLIN, 1>(e0, e1, e2, q.g, q.c.y, a.g, q.c.z, q.c.w, dt, q.r, one_p_theta,
                                                         a.theta, u[j]);
                float2 low = kSloShared ? lds2(slo_at + 8 * i) : slo[kSloShared ? 0 : j];
                two_sum_acc2<0>(shi[j], low, F);
                if (kSloShared) sts2(slo_at + 8 * i, low); else slo[kSloShared ? 0 : j] = low;
                float f3[3];
                corner_fluxes<0>(F, q.g, q.c.x, f3);
                sts(q.f0, f3[0]);
                sts(q.f1, f3[1]);
                sts(q.f2, f3[2]);
            }
        }
    };

    // Slots updated first: whole rounds of interior slots (one per thread each), so that
    // no thread does more rounds in total than ceil(ns / T); the interior slots left over
    // go with the boundary slots, whose halo reads may have to wait for a neighbour. (Fewer than
    // one round of interior slots: whole warps of them.)
    const int npre = nint >= T ? (nint / T) * T : nint & ~31;
    const int total = P.M * P.nsteps;
    // substeps below it publish: all but the last, for the failure test's patch none of the last step
    const int publish_end = p == a.silent_patch ? total - P.M : total - 1;
    for (int m = 0, ms = 0; m < total; m++) {
        if (m == 0) {
            elements(0, nsp);    // every halo elevation is in shared memory
        } else {
            // this thread's halo word is requested before the interior rounds and stored to
            // shared memory after them; the other slots follow a barrier
            const unsigned long long *xs = P.xb[m & 1];
            const int hv = tid < nhalo ? hid[tid] : -1;
            const unsigned long long hw = hv >= 0 ? ld_relaxed_gpu_u64(xs + hv) : 0ull;
            elements(0, npre);
            if (hv >= 0) seta[nown + tid] = halo_eta(P, xs, hv, hw, base + (unsigned)m, abort_val, ok);
            for (int k = tid + T; k < nhalo; k += T) {
                const int v = hid[k];
                seta[nown + k] = halo_eta(P, xs, v, ld_relaxed_gpu_u64(xs + v), base + (unsigned)m, abort_val, ok);
            }
            team_sync(bar, T);
            elements(npre, nsp);
            if (!ok) s_abort = 1;
        }
        team_sync(bar, T);
        if (s_abort) break;

        // vertex pass; the new elevation of own vertices also goes to the exchange buffer
        const bool more = m + 1 < total;
        unsigned long long *xout = P.xb[(m + 1) & 1];
        const unsigned long long tag_out = (unsigned long long)(base + (unsigned)(m + 1)) << 32;
        const bool publish = m < publish_end;
        bool bad = false;
        for (int i = tid; i < nown; i += T) {
            float sum = 0.0f, inv;
            if (CACHED) {
                sum = row_flux_sum<(SPT >= 7)>(P, team, v0, i);
                inv = s_inv[i];
            } else {
                const int k1 = P.vcsr_off[v0 + i + 1];
                for (int k = P.vcsr_off[v0 + i]; k < k1; k++) {
                    const uint32_t q = P.vcsr[k];
                    sum = __fadd_rn(sum, reinterpret_cast<const float *>(smem_raw + P.off_flux)[3u * (q >> 2) + (q & 3u)]);
                }
                inv = P.inv_av[v0 + i];
            }
            const float e0 = seta[i];
            float e = vertex_eta(e0, sum, inv);
            if (EXTRA) {
                if (P.W) e = __fmaf_rn(-dt, __ldg(P.W + v0 + i), e);
                if (P.eta_sum) P.eta_sum[v0 + i] = (ms == 0 ? 0.0f : P.eta_sum[v0 + i]) + e0;
            }
            seta[i] = e;
            if (publish) st_relaxed_gpu_u64(xout + v0 + i, tag_out | __float_as_uint(e));
            bad |= !(fabsf(e) <= a.eta_bound);
        }
        if (bad) atomicOr(P.status, 1u);
        team_sync(bar, T);
        if (!more) break;
        if (++ms == P.M) {
            // a step ends: the sums of the next one start from zero (the low parts in shared memory by
            // sts2, which keeps its order to the lds2 of the next substep: no barrier lies between)
            ms = 0;
#pragma unroll
            for (int j = 0; j < SPT; j++) {
                const int i = tid + j * T;
                shi[j] = make_float2(0.0f, 0.0f);
                if (!kSloShared) slo[j] = make_float2(0.0f, 0.0f);
                if (kSloShared && i < nsp) sts2(slo_at + 8 * i, make_float2(0.0f, 0.0f));
            }
        }
    }
    team_sync(bar, T);

    for (int i = tid; i < nown; i += T) P.eta_out[v0 + i] = seta[i];
#pragma unroll
    for (int j = 0; j < SPT; j++) {
        const int i = tid + j * T;
        if (i < ns) {
            P.U[s0 + i] = u[j];
            if (i < nown_s) {
                const int w = P.sv[s0 + i].w;
                const float2 lo = kSloShared ? lds2(slo_at + 8 * i) : slo[kSloShared ? 0 : j];
                P.Umean[w] = make_float2((shi[j].x + lo.x) * a.inv_M, (shi[j].y + lo.y) * a.inv_M);
            }
        }
    }
    // the last block of the pack to leave (every block of the pack has read the base by
    // then) sets the base of the pack's next launch
    if (tid == 0 && atomicAdd(exit_count, 1u) == (unsigned)npb - 1u) {
        *exit_count = 0u;
        *base_word = base + (unsigned)total + 1u;
    }
}

// A launch runs packs [P.pack_first, P.pack_last) one after another: team t of block b takes
// patch b + t gridDim of each pack that has it. Packs exchange nothing with each other (a pack
// holds whole basins), so a team goes on to its next pack as soon as it is done with the last
// one, while others still finish theirs; every team of a pack is resident, so the waits of a
// pack always end.
// CACHED: the vertices' data in shared memory and the slots' in tensor memory; 0 reads both from L2.
template <int SPT, int NONLIN, int CACHED, int EXTRA>
__global__ void __launch_bounds__(1024, 1) k_persistent(PArgs P)
{
    extern __shared__ __align__(16) unsigned char smem_all[];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort[kMaxTeams];
    const int warp = threadIdx.x >> 5;
    uint32_t base = 0, tm = 0;
    if (CACHED) {
        if (warp == 0) tmem_alloc(&s_tmem, P.tmem_cols);
        __syncthreads();
        tmem_fence_after_sync();
        base = s_tmem;
        // warp w holds lanes 32 (w % 4) .. + 31 and its own columns
        tm = base + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * TmemSlots<SPT>::kWords;
    }
    const int T = P.team_threads, team = (int)threadIdx.x / T, tid = (int)threadIdx.x - team * T;
    for (int k = P.pack_first; k < P.pack_last; k++) {
        const int b0 = P.pack_off[k], npb = P.pack_off[k + 1] - b0, q = (int)blockIdx.x + team * (int)gridDim.x;
        if (q < npb) {
            persistent_patch<SPT, NONLIN, CACHED, EXTRA>(P, P.pack_patch[b0 + q], k, npb, tm,
                                                         smem_all + (size_t)team * P.team_smem, s_abort[team], tid, T,
                                                         team + 1);
            team_sync(team + 1, T);   // the next pack reuses the shared memory
        }
    }
    if (CACHED) {
        tmem_fence_before_sync();
        __syncthreads();
        if (warp == 0) tmem_dealloc(base, P.tmem_cols);
    }
}

// extra: the freshwater flux or the step-mean elevation is set
template <int SPT, int CACHED>
void *persistent_fn(int nonlin, int extra)
{
    if (extra) return nonlin ? (void *)k_persistent<SPT, 1, CACHED, 1> : (void *)k_persistent<SPT, 0, CACHED, 1>;
    return nonlin ? (void *)k_persistent<SPT, 1, CACHED, 0> : (void *)k_persistent<SPT, 0, CACHED, 0>;
}

void *persistent_kernel(int spt, int nonlin, int cached, int extra)
{
    if (cached) {
        switch (spt) {
        case 1: return persistent_fn<1, 1>(nonlin, extra);
        case 2: return persistent_fn<2, 1>(nonlin, extra);
        case 3: return persistent_fn<3, 1>(nonlin, extra);
        case 4: return persistent_fn<4, 1>(nonlin, extra);
        case 5: return persistent_fn<5, 1>(nonlin, extra);
        case 6: return persistent_fn<6, 1>(nonlin, extra);
        case 7: return persistent_fn<7, 1>(nonlin, extra);
        case 8: return persistent_fn<8, 1>(nonlin, extra);
        default: return nullptr;
        }
    }
    switch (spt) {
    case 1: return persistent_fn<1, 0>(nonlin, extra);
    case 2: return persistent_fn<2, 0>(nonlin, extra);
    case 3: return persistent_fn<3, 0>(nonlin, extra);
    case 4: return persistent_fn<4, 0>(nonlin, extra);
    case 6: return persistent_fn<6, 0>(nonlin, extra);
    case 8: return persistent_fn<8, 0>(nonlin, extra);
    default: return nullptr;
    }
}

int tmem_words(int spt) { return spt <= 4 ? 16 * spt : (spt <= 6 ? 60 : 64); }

}  // namespace

size_t persistent_flag_bytes(int npatch) { return flag_bytes(npatch); }

PersistentPlan persistent_plan(const PatchMax &m, int blocks_per_sm)
{
    PersistentPlan plan;
    int dev = 0, smem_optin = 0, smem_sm = 0, nsm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) {
        cudaGetLastError();
        return plan;
    }
    const int teams = std::min(std::max(blocks_per_sm, 1), kMaxTeams), max_threads = 1024 / teams;
    // per team: its part of the block's share of the SM's capacity (1 KB is reserved by the
    // system, plus the kernel's static shared)
    if (smem_optin < 2048 || smem_sm < 4096) return plan;
    const size_t budget = std::min((size_t)smem_optin - 1024, (size_t)smem_sm - 2048);
    // Fewest slots per thread such that one team of at most max_threads covers the largest
    // patch, first with the patch's static data on chip (vertices' data in shared memory, slots'
    // in tensor memory; from 6 slots per thread also the low parts of the sums in shared
    // memory), else with all of it read from L2 (5 and 7 slots per thread exist only on chip).
    // The team is sized to the largest patch (a multiple of 32).
    for (int cached = 1; cached >= 0; cached--)
        for (int spt = 1; spt <= 8; spt++) {
            const int t = std::max(32, ((m.slots + spt - 1) / spt + 31) / 32 * 32);
            if (t > max_threads || !persistent_kernel(spt, 0, cached, 0)) continue;
            const unsigned cols = cached ? tmem_columns(teams * t, tmem_words(spt)) : 0u;
            // rows of the largest degree where they fit, else rows of kRowFluxes and overflow quads
            int wide = 1;
            size_t team_smem = 0, smem = 0;
            for (; wide >= 0; wide--) {
                team_smem = se_layout(m, spt, cached, wide).total;
                smem = teams * team_smem;
                if (cached) smem = std::max(smem, tmem_smem_floor(cols, (size_t)smem_sm));
                if (smem <= budget) break;
            }
            if (wide < 0 || cols > 512u) break;
            // every variant the plan may launch must be able to run
            bool fits = true;
            for (int nonlin = 0; nonlin < 2 && fits; nonlin++)
                for (int extra = 0; extra < 2 && fits; extra++) {
                    void *fn = persistent_kernel(spt, nonlin, cached, extra);
                    int occ = 0;
                    if (!fn || raise_smem_limit(fn) < (int)smem ||
                        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, teams * t, smem) != cudaSuccess ||
                        occ < 1) {
                        cudaGetLastError();
                        fits = false;
                    }
                }
            if (!fits) break;
            plan.slots_per_thread = spt;
            plan.threads = t;
            plan.cached = cached ? (spt <= 5 ? 1 : 2) : 0;
            plan.wide_rows = wide;
            plan.over16 = cached && m.deg > 16;
            plan.teams = teams;
            plan.team_smem = (int)team_smem;
            plan.tmem_cols = (int)cols;
            plan.grid = nsm;
            plan.smem = smem;
            return plan;
        }
    return plan;
}

cudaError_t persistent_prepare(const PersistentPlan &plan)
{
    for (int nonlin = 0; nonlin < 2; nonlin++)
        for (int extra = 0; extra < 2; extra++) {
            void *fn = persistent_kernel(plan.slots_per_thread, nonlin, plan.cached, extra);
            if (!fn || raise_smem_limit(fn) < (int)plan.smem) return cudaErrorInvalidValue;
        }
    return cudaSuccess;
}

cudaError_t launch_persistent(const DevMesh &m, const DevState &s, const StepArgs &a, int M, int parity,
                              int nsteps, const std::vector<PackGroup> &groups,
                              cudaStream_t stream)
{
    const int extra = s.W != nullptr || s.eta_sum != nullptr;
    if (m.cluster.blocks > 0) return launch_cluster(m, s, a, M, parity, nsteps, stream);   // a small mesh
    for (const PackGroup &g : groups) {
        cudaError_t e;
        if (g.plan.stream) {
            if (nsteps != 1) return cudaErrorInvalidValue;   // one step per launch
            e = launch_persistent_stream_group(m, s, a, M, parity, g, stream);
        } else {
            void *fn = persistent_kernel(g.plan.slots_per_thread, a.nonlinear_h, g.plan.cached, extra);
            if (!fn) return cudaErrorInvalidValue;
            PArgs P = make_pargs(m, s, a, M, parity, g.mx);
            set_layout(P, se_layout(g.mx, g.plan.slots_per_thread, g.plan.cached, g.plan.wide_rows), g.mx);
            P.pack_first = g.first;
            P.pack_last = g.last;
            P.nsteps = nsteps;
            P.tmem_cols = (unsigned)g.plan.tmem_cols;
            P.team_threads = g.plan.threads;
            P.team_smem = g.plan.team_smem;
            void *args[] = {&P};
            e = cudaLaunchCooperativeKernel(fn, dim3(std::min(g.plan.grid, g.nblocks)),
                                            dim3(g.plan.teams * g.plan.threads), args, g.plan.smem, stream);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_slot_coef(const DevMesh &m, float g, cudaStream_t stream)
{
    if (m.npatch <= 0) return cudaSuccess;
    k_slot_coef<<<std::min(m.npatch, 152 * 16), 256, 0, stream>>>(m.npatch, m.patch_slot, m.patch_dt, m.slot_c, g,
                                                                 m.slot_k);
    return cudaGetLastError();
}

}  // namespace sesw
