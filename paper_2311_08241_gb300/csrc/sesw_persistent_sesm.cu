// The SESM step kernels of libsesw (sm_103a): one cooperative launch runs one or several baroclinic
// steps of the AB3-AM4 substep of Eqs. (4.7)-(4.8), with the time-mean transport of Eq.
// (4.12) and the freshwater flux of Eq. (4.5).
#include "sesw_persistent.cuh"

namespace sesw {

namespace {

// ---------------------------------------------------------------------------------
// The SESM substep (AB3-AM4, Eqs. 4.7-4.8) in the persistent form: one launch runs the
// M + 1 element passes and M vertex passes of a baroclinic step. Substep m (m >= 1)
// completes the momentum update
//     U^m = U^{m-1} + dt ( -f e_z x U_AB^{m-1} - g H_AM grad(eta_AM^m) + R ),
//     eta_AM^m = am0 eta^m + am1 eta^{m-1} + am2 eta^{m-2} + am3 eta^{m-3},
// then (m < M) forms U_AB^m = ab0 U^m + ab1 U^{m-1} + ab2 U^{m-2}, adds it to the
// compensated sum and updates eta^{m+1} = eta^m - dt (div(U_AB^m) + W). Levels before the
// start of the subcycle are level 0. A slot keeps U^{m-1}, U^{m-2}, U_AB^{m-1} and its sum
// in registers; a vertex keeps eta^m, eta^{m-1}, eta^{m-2} in the registers of the thread
// that updates it. The element pass needs only eta_AM at the corners, so the owner of a
// vertex forms eta_AM^{m+1} right after eta^{m+1} and exchanges that one value, with the
// same tagged words as the SE kernel (tag base + x for substep x = 1 .. n M of a launch of n
// steps; a launch loads the patch once for all of them).
constexpr int kSesmThreads = 384;         // two blocks per SM; registers: 65536 / (2 x 384) = 85 per thread
constexpr int kSesmVpt = 2;         // own vertices per thread at most

template <int SPT, int NONLIN>
__global__ void __launch_bounds__(kSesmThreads, 2) k_persistent_sesm(PArgs P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_abort;
    const int p = P.pack_patch[P.pack_base + blockIdx.x];
    const int T = blockDim.x;
    const int s0 = P.patch_slot[p], ns = P.patch_slot[p + 1] - s0;
    const int nown_s = P.patch_own[p], nint = P.patch_int[p];
    const int v0 = P.patch_v[p], nown = P.patch_v[p + 1] - v0;
    const int hb = P.patch_halo[p], nhalo = P.patch_halo[p + 1] - hb;
    const StepArgs a = P.a;
    const float dt = P.patch_dt[p];
    unsigned *base_word = P.flags + (size_t)(1 + 2 * P.pack_index) * kFlagStride;
    unsigned *exit_count = base_word + kFlagStride;
    const unsigned base = ld_relaxed_gpu(base_word);
    const unsigned abort_val = base + 1u == 0u ? 1u : base + 1u;   // never 0, unique per launch

    float *sem = reinterpret_cast<float *>(smem_raw);   // eta_AM of the own vertices, then of the halo
    float *sflux = reinterpret_cast<float *>(smem_raw + P.off_flux);
    float4 *s_g = reinterpret_cast<float4 *>(smem_raw + P.off_g);
    float4 *s_c = reinterpret_cast<float4 *>(smem_raw + P.off_c);
    float2 *s_r = reinterpret_cast<float2 *>(smem_raw + P.off_r);
    ushort4 *s_l = reinterpret_cast<ushort4 *>(smem_raw + P.off_l);
    float *s_inv = reinterpret_cast<float *>(smem_raw + P.off_inv);
    int *s_halo = reinterpret_cast<int *>(smem_raw + P.off_halo);

    for (int i = threadIdx.x; i < ns; i += T) {
        s_g[i] = P.sg[s0 + i];
        s_c[i] = P.sc[s0 + i];
        s_r[i] = P.R[s0 + i];
        s_l[i] = P.sl[s0 + i];
    }
    cache_incidences(P, smem_raw, v0, nown, threadIdx.x, T);
    for (int i = threadIdx.x; i < nown; i += T) s_inv[i] = P.inv_av[v0 + i];
    for (int i = threadIdx.x; i < nhalo; i += T) s_halo[i] = P.halo_v[hb + i];
    if (threadIdx.x == 0) s_abort = 0;
    // slot state: U^{m-1}, U^{m-2}, U_AB^{m-1}, compensated sum; vertex state: eta^m,
    // eta^{m-1}, eta^{m-2}
    float2 u1[SPT], u2[SPT], uab[SPT], shi[SPT], slo[SPT];
#pragma unroll
    for (int j = 0; j < SPT; j++) {
        const int i = threadIdx.x + j * T;
        u1[j] = i < ns ? P.U[s0 + i] : make_float2(0.0f, 0.0f);
        u2[j] = u1[j];
        uab[j] = make_float2(0.0f, 0.0f);
        shi[j] = make_float2(0.0f, 0.0f);
        slo[j] = make_float2(0.0f, 0.0f);
    }
    float eh0[kSesmVpt], eh1[kSesmVpt], eh2[kSesmVpt];
#pragma unroll
    for (int k = 0; k < kSesmVpt; k++) {
        const int i = threadIdx.x + k * T;
        eh0[k] = i < nown ? P.eta_in[v0 + i] : 0.0f;
        eh1[k] = eh0[k];
        eh2[k] = eh0[k];
    }
    __syncthreads();

    // U_AB of a slot, its flux contributions and (owned slots) the compensated sum
    auto transport = [&](int j, int i, float2 u0, float2 ua, float2 ub, float4 g, float area) {
        const float2 F = sesm_ab3(u0, ua, ub, a.ab0, a.ab1, a.ab2);
        if (i < nown_s) {
            two_sum_acc2(shi[j], slo[j], F);
        }
        corner_fluxes(F, g, __fmul_rn(dt, area), sflux + 3 * i);
        uab[j] = F;
    };
    bool ok = true;
    // momentum update of slot i (round j) from its corner eta_AM
    auto slot = [&](int j, int i, float e0, float e1, float e2, bool vertex) {
        const float4 g = s_g[i], c = s_c[i];
        const float2 r = s_r[i];
        const float2 u0 = sesm_momentum<NONLIN>(e0, e1, e2, g, c.y, a.g, c.z, dt, r, u1[j], uab[j]);
        if (vertex) transport(j, i, u0, u1[j], u2[j], g, c.x);
        u2[j] = u1[j];
        u1[j] = u0;
    };
    const int npre = nint >= T ? (nint / T) * T : nint;
    // One thread per halo vertex requests its tagged word before the interior rounds and stores
    // the value after them; the other slots follow a barrier. x counts the substeps of the launch
    // (the exchange's tags), m those of the running step, whose closing pass (m = M) is the momentum
    // update of its last substep.
    const int total = P.M * P.nsteps;
    const int last_publish = p == a.silent_patch ? total - P.M : total;   // failure test: none in the last step
    for (int x = 0, m = 0; x <= total; m++) {
        const bool vertex = m < P.M;
        if (m == 0) {
            // no momentum update: U_AB^0 from level 0 and its aliases; the sums start
#pragma unroll
            for (int j = 0; j < SPT; j++) {
                const int i = threadIdx.x + j * T;
                shi[j] = make_float2(0.0f, 0.0f);
                slo[j] = make_float2(0.0f, 0.0f);
                u2[j] = u1[j];
                if (i < ns) transport(j, i, u1[j], u1[j], u1[j], s_g[i], s_c[i].x);
            }
#pragma unroll
            for (int k = 0; k < kSesmVpt; k++) eh1[k] = eh2[k] = eh0[k];
        } else {
            const unsigned long long *xs = P.xb[x & 1];
            const unsigned tag = base + (unsigned)x;
            const int hv = (int)threadIdx.x < nhalo ? s_halo[threadIdx.x] : -1;
            const unsigned long long hw = hv >= 0 ? ld_relaxed_gpu_u64(xs + hv) : 0ull;
#pragma unroll
            for (int j = 0; j < SPT; j++) {
                const int i = threadIdx.x + j * T;
                if (i < npre) {
                    const ushort4 l = s_l[i];
                    slot(j, i, sem[l.x], sem[l.y], sem[l.z], vertex);
                }
            }
            if (hv >= 0) sem[nown + threadIdx.x] = halo_eta(P, xs, hv, hw, tag, abort_val, ok);
            for (int k = threadIdx.x + T; k < nhalo; k += T) {
                const int v = s_halo[k];
                sem[nown + k] = halo_eta(P, xs, v, ld_relaxed_gpu_u64(xs + v), tag, abort_val, ok);
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < SPT; j++) {
                const int i = threadIdx.x + j * T;
                if (i >= npre && i < ns) {
                    const ushort4 l = s_l[i];
                    slot(j, i, sem[l.x], sem[l.y], sem[l.z], vertex);
                }
            }
            if (!ok) s_abort = 1;
        }
        if (!vertex) {
            if (x == total) break;
            m = -1;               // the next step starts at the same x; its first pass reads no halo
            __syncthreads();
            if (s_abort) break;
            continue;
        }
        __syncthreads();
        if (s_abort) break;
        x++;

        // vertex pass: eta^{m+1}, then eta_AM^{m+1} for the own slots and the neighbours
        unsigned long long *xout = P.xb[x & 1];
        const unsigned long long tag_out = (unsigned long long)(base + (unsigned)x) << 32;
        const bool publish = x <= last_publish;
        bool bad = false;
#pragma unroll
        for (int k = 0; k < kSesmVpt; k++) {
            const int i = threadIdx.x + k * T;
            if (i < nown) {
                const float sum = cached_flux_sum(P, smem_raw, i);
                float e = vertex_eta(eh0[k], sum, s_inv[i]);
                if (P.W) e = __fmaf_rn(-dt, __ldg(P.W + v0 + i), e);
                const float em = sesm_am4(e, eh0[k], eh1[k], eh2[k], a.am0, a.am1, a.am2, a.am3);
                eh2[k] = eh1[k];
                eh1[k] = eh0[k];
                eh0[k] = e;
                sem[i] = em;
                if (publish) st_relaxed_gpu_u64(xout + v0 + i, tag_out | __float_as_uint(em));
                bad |= !(fabsf(e) <= a.eta_bound);
            }
        }
        if (bad) atomicOr(P.status, 1u);
        __syncthreads();
    }
    __syncthreads();

#pragma unroll
    for (int k = 0; k < kSesmVpt; k++) {
        const int i = threadIdx.x + k * T;
        if (i < nown) P.eta_out[v0 + i] = eh0[k];
    }
#pragma unroll
    for (int j = 0; j < SPT; j++) {
        const int i = threadIdx.x + j * T;
        if (i < ns) {
            P.U[s0 + i] = u1[j];
            if (i < nown_s) {
                const int w = P.sv[s0 + i].w;
                P.Umean[w] = make_float2((shi[j].x + slo[j].x) * a.inv_M, (shi[j].y + slo[j].y) * a.inv_M);
            }
        }
    }
    if (threadIdx.x == 0 && atomicAdd(exit_count, 1u) == gridDim.x - 1) {
        *exit_count = 0u;
        *base_word = base + (unsigned)total + 1u;
    }
}

// ---------------------------------------------------------------------------------
// The same for larger patches (up to 7 slots per thread): one block per SM holds one to four
// teams, each with its own patch, with the flux rows and tensor memory of the SE kernel
// (sesw_persistent.cu). U^{m-1} of a slot lives in registers, U_AB^{m-1} in shared memory, U^{m-2}, the
// sum and the packed addresses (9 words) in tensor memory; the static data (40 B per slot and
// substep) come from L2. Before, all state streamed from L2 as well (k_persistent_sesm_stream, now
// for patches beyond this): 408k vertices, two steps, 1003 -> 639 us.
// (On-chip patches stay with k_persistent_sesm: teams with their static data in tensor memory measured
// the same, 488 against 490 us for four steps of the 200k-vertex channel.)
constexpr int kSesmTeamThreads = 1024;   // 64 registers per thread

// A thread's words in tensor memory: the sums (4 per slot), then U^{m-2} (2), then the
// addresses of the three corners and three flux places as 16-bit word indices (2 and 1).
template <int SPT>
struct SesmState {
    __device__ static __forceinline__ void store(uint32_t tm, int j, float2 hi, float2 lo, float2 u)
    {
        tmem_st4(tm + 4 * j, hi.x, hi.y, lo.x, lo.y);
        tmem_st2(tm + 4 * SPT + 2 * j, __float_as_uint(u.x), __float_as_uint(u.y));
    }
    __device__ static __forceinline__ void store_places(uint32_t tm, int j, const SlotData &q)
    {
        tmem_st2(tm + 6 * SPT + 2 * j, (q.a0 >> 2) | (q.a1 << 14), (q.a2 >> 2) | (q.f0 << 14));
        asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(tm + 8 * SPT + j),
                     "r"((q.f1 >> 2) | (q.f2 << 14))
                     : "memory");
    }
    __device__ static __forceinline__ void load(uint32_t tm, int j, float2 &hi, float2 &lo, float2 &u, SlotData &q)
    {
        float st[6];
        uint32_t p0, p1, p2;
        tmem_ld9(tm + 4 * j, tm + 4 * SPT + 2 * j, tm + 6 * SPT + 2 * j, tm + 8 * SPT + j, st, p0, p1, p2);
        hi = make_float2(st[0], st[1]);
        lo = make_float2(st[2], st[3]);
        u = make_float2(st[4], st[5]);
        q.a0 = (p0 & 0xffffu) * 4u;
        q.a1 = (p0 >> 16) * 4u;
        q.a2 = (p1 & 0xffffu) * 4u;
        q.f0 = (p1 >> 16) * 4u;
        q.f1 = (p2 & 0xffffu) * 4u;
        q.f2 = (p2 >> 16) * 4u;
    }
};

// Tensor-memory words of a thread.
__host__ __device__ constexpr int sesm_words(int spt) { return (9 * spt + 3) & ~3; }

template <int SPT, int NONLIN>
__device__ __forceinline__ void sesm_patch(const PArgs &P, const int p, const int pack, const int npb,
                                           const uint32_t tm, unsigned char *smem_raw, int &s_abort, const int tid,
                                           const int T, const int bar)
{
    using SS = SesmState<SPT>;
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

    float *sem = reinterpret_cast<float *>(smem_raw);   // eta_AM of the own vertices, then of the halo
    float *s_inv = reinterpret_cast<float *>(smem_raw + P.off_inv);
    int *s_halo = reinterpret_cast<int *>(smem_raw + P.off_halo);
    float *hist = reinterpret_cast<float *>(smem_raw + P.off_hist);   // three levels of row_vertices each
    clear_rows(P, smem_raw, v0, nown, tid, T);
    for (int i = tid; i < nown; i += T) {
        s_inv[i] = P.inv_av[v0 + i];
        hist[i] = P.eta_in[v0 + i];
    }
    for (int i = tid; i < nhalo; i += T) s_halo[i] = P.halo_v[hb + i];
    if (tid == 0) s_abort = 0;
    // threads without a slot in their last round hold an all-zero one (see k_persistent)
    const uint32_t dummy = team + (uint32_t)P.off_dummy + 4u * (tid & 31);
    const uint32_t uab_at = team + (uint32_t)P.off_slo;      // U_AB^{m-1} of the slots
    float2 u1[SPT];
#pragma unroll
    for (int j = 0; j < SPT; j++) {
        const int i = tid + j * T;
        const bool in = i < ns;
        const int s = s0 + (in ? i : 0);
        const ushort4 l = P.sl[s];
        const uint2 f = in ? P.sf[s] : make_uint2(0xffffffffu, 0x7fffffffu);
        SlotData q;
        q.a0 = team + 4u * l.x;
        q.a1 = team + 4u * l.y;
        q.a2 = team + 4u * l.z;
        q.f0 = flux_place(P, team, dummy, f.x & 0x1fffffu, v0, l.x);
        q.f1 = flux_place(P, team, dummy, (f.x >> 21) | ((f.y & 0x3ffu) << 11), v0, l.y);
        q.f2 = flux_place(P, team, dummy, (f.y >> 10) & 0x1fffffu, v0, l.z);
        SS::store_places(tm, j, q);
        u1[j] = in ? P.U[s] : make_float2(0.0f, 0.0f);
    }
    tmem_wait_st();
    team_sync(bar, T);

    // Slots [lo, hi) (multiples of 32, whole warps) at substep ms of the step: the momentum update (ms > 0),
    // then (vertex) U_AB, its fluxes and the compensated sum. At ms = 0 every earlier level is level 0
    // and the sum starts.
    auto elements = [&](int lo, int hi, int ms, bool vertex) {
#pragma unroll
        for (int j = 0; j < SPT; j++) {
            const int w = wbase + j * T;
            if (w >= lo && w < hi) {
                const int i = tid + j * T;
                SlotData q;
                float2 v2, hi2, lo2;
                const int s = s0 + min(i, ns - 1);
                q.g = __ldg(P.sg + s);
                q.c = __ldg(P.sc + s);
                q.r = __ldg(P.R + s);
                SS::load(tm, j, hi2, lo2, v2, q);
                if (i >= ns) {
                    q.g = q.c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    q.r = make_float2(0.0f, 0.0f);
                }
                float2 u0 = u1[j], up = u1[j];
                if (ms > 0) {
                    const float e0 = lds(q.a0), e1 = lds(q.a1), e2 = lds(q.a2);
                    u0 = sesm_momentum<NONLIN>(e0, e1, e2, q.g, q.c.y, a.g, q.c.z, dt, q.r, up,
                                               lds2(uab_at + 8 * i));
                } else {
                    v2 = u0;
                    hi2 = lo2 = make_float2(0.0f, 0.0f);
                }
                u1[j] = u0;
                if (vertex) {
                    const float2 F = sesm_ab3(u0, up, v2, a.ab0, a.ab1, a.ab2);
                    two_sum_acc2<0>(hi2, lo2, F);
                    float f3[3];
                    corner_fluxes<0>(F, q.g, __fmul_rn(dt, q.c.x), f3);
                    sts(q.f0, f3[0]);
                    sts(q.f1, f3[1]);
                    sts(q.f2, f3[2]);
                    sts2(uab_at + 8 * i, F);
                    SS::store(tm, j, hi2, lo2, up);    // U^{m-1} of this substep is U^{m-2} of the next
                }
            }
        }
        tmem_wait_st();
    };

    bool ok = true;
    const int npre = nint >= T ? (nint / T) * T : nint & ~31;
    // x counts the substeps of the launch (the exchange's tags); ms those of the running step, whose
    // closing pass (ms = M) is the momentum update of its last substep
    const int total = P.M * P.nsteps;
    const int last_publish = p == a.silent_patch ? total - P.M : total;   // failure test: none in the last step
    int cur = 0;                      // level of hist with eta^m
    for (int x = 0, ms = 0; x <= total; ms++) {
        const bool vertex = ms < P.M;
        if (ms == 0) {
            elements(0, nsp, 0, true);
        } else {
            const unsigned long long *xs = P.xb[x & 1];
            const unsigned tag = base + (unsigned)x;
            const int hv = tid < nhalo ? s_halo[tid] : -1;
            const unsigned long long hw = hv >= 0 ? ld_relaxed_gpu_u64(xs + hv) : 0ull;
            elements(0, npre, ms, vertex);
            if (hv >= 0) sem[nown + tid] = halo_eta(P, xs, hv, hw, tag, abort_val, ok);
            for (int k = tid + T; k < nhalo; k += T) {
                const int v = s_halo[k];
                sem[nown + k] = halo_eta(P, xs, v, ld_relaxed_gpu_u64(xs + v), tag, abort_val, ok);
            }
            team_sync(bar, T);
            elements(npre, nsp, ms, vertex);
            if (!ok) s_abort = 1;
        }
        if (!vertex) {
            if (x == total) break;
            ms = -1;                  // the next step starts at the same x; its first pass reads no halo
            team_sync(bar, T);
            if (s_abort) break;
            continue;
        }
        team_sync(bar, T);
        if (s_abort) break;

        // vertex pass: eta^{m+1}, then eta_AM^{m+1} for the own slots and the neighbours
        x++;
        unsigned long long *xout = P.xb[x & 1];
        const unsigned long long tag_out = (unsigned long long)(base + (unsigned)x) << 32;
        const bool publish = x <= last_publish;
        const int nv = P.row_vertices, nxt = cur == 2 ? 0 : cur + 1, prv = cur == 0 ? 2 : cur - 1;
        bool bad = false;
        for (int i = tid; i < nown; i += T) {
            const float sum = row_flux_sum<false>(P, team, v0, i);
            const float h0 = hist[cur * nv + i];
            const float h1 = ms == 0 ? h0 : hist[prv * nv + i], h2 = ms == 0 ? h0 : hist[nxt * nv + i];
            float e = vertex_eta(h0, sum, s_inv[i]);
            if (P.W) e = __fmaf_rn(-dt, __ldg(P.W + v0 + i), e);
            const float em = sesm_am4(e, h0, h1, h2, a.am0, a.am1, a.am2, a.am3);
            hist[nxt * nv + i] = e;
            if (ms == 0) hist[prv * nv + i] = h0;
            sem[i] = em;
            if (publish) st_relaxed_gpu_u64(xout + v0 + i, tag_out | __float_as_uint(em));
            bad |= !(fabsf(e) <= a.eta_bound);
        }
        cur = nxt;
        if (bad) atomicOr(P.status, 1u);
        team_sync(bar, T);
    }
    team_sync(bar, T);

    for (int i = tid; i < nown; i += T) P.eta_out[v0 + i] = hist[cur * P.row_vertices + i];
#pragma unroll
    for (int j = 0; j < SPT; j++) {
        const int i = tid + j * T;
        SlotData q;
        float2 hi2, lo2, u;
        SS::load(tm, j, hi2, lo2, u, q);
        if (i < ns) {
            P.U[s0 + i] = u1[j];
            if (i < nown_s) {
                const int w = P.sv[s0 + i].w;
                P.Umean[w] = make_float2((hi2.x + lo2.x) * a.inv_M, (hi2.y + lo2.y) * a.inv_M);
            }
        }
        __syncwarp();
    }
    if (tid == 0 && atomicAdd(exit_count, 1u) == (unsigned)npb - 1u) {
        *exit_count = 0u;
        *base_word = base + (unsigned)total + 1u;
    }
}

template <int SPT, int NONLIN>
__global__ void __launch_bounds__(kSesmTeamThreads, 1) k_persistent_sesm_teams(PArgs P)
{
    extern __shared__ __align__(16) unsigned char smem_all[];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort[kMaxTeams];
    const int warp = threadIdx.x >> 5;
    if (warp == 0) tmem_alloc(&s_tmem, P.tmem_cols);
    __syncthreads();
    tmem_fence_after_sync();
    const uint32_t base = s_tmem;
    const uint32_t tm = base + ((uint32_t)(warp & 3) << 21) + (uint32_t)((warp >> 2) * sesm_words(SPT));
    const int T = P.team_threads, team = (int)threadIdx.x / T, tid = (int)threadIdx.x - team * T;
    const int npb = P.npb, q = (int)blockIdx.x + team * (int)gridDim.x;
    if (q < npb)
        sesm_patch<SPT, NONLIN>(P, P.pack_patch[P.pack_base + q], P.pack_index, npb, tm,
                                smem_all + (size_t)team * P.team_smem, s_abort[team], tid, T, team + 1);
    tmem_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(base, P.tmem_cols);
}

void *sesm_kernel(int spt, int nonlin)
{
    switch (spt) {
    case 1: return nonlin ? (void *)k_persistent_sesm<1, 1> : (void *)k_persistent_sesm<1, 0>;
    case 2: return nonlin ? (void *)k_persistent_sesm<2, 1> : (void *)k_persistent_sesm<2, 0>;
    case 3: return nonlin ? (void *)k_persistent_sesm<3, 1> : (void *)k_persistent_sesm<3, 0>;
    case 4: return nonlin ? (void *)k_persistent_sesm<4, 1> : (void *)k_persistent_sesm<4, 0>;
    default: return nullptr;
    }
}

void *sesm_teams_kernel(int spt, int nonlin)
{
    switch (spt) {
    case 4: return nonlin ? (void *)k_persistent_sesm_teams<4, 1> : (void *)k_persistent_sesm_teams<4, 0>;
    case 5: return nonlin ? (void *)k_persistent_sesm_teams<5, 1> : (void *)k_persistent_sesm_teams<5, 0>;
    case 6: return nonlin ? (void *)k_persistent_sesm_teams<6, 1> : (void *)k_persistent_sesm_teams<6, 0>;
    case 7: return nonlin ? (void *)k_persistent_sesm_teams<7, 1> : (void *)k_persistent_sesm_teams<7, 0>;
    default: return nullptr;
    }
}

}  // namespace

PersistentPlan persistent_plan_sesm(const PatchMax &m, int blocks_per_sm)
{
    PersistentPlan plan;
    int dev = 0, smem_optin = 0, smem_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) {
        cudaGetLastError();
        return plan;
    }
    if (blocks_per_sm < 1) blocks_per_sm = 1;
    // fewest slots per thread such that one block of at most kSesmThreads covers the
    // largest patch, whose own vertices must then fit kSesmVpt per thread
    int spt = 0, t = 0;
    for (int cand = 1; cand <= 4; cand++) {
        const int need = (m.slots + cand - 1) / cand;
        const int tt = std::max(32, ((need + 31) / 32) * 32);
        if (tt <= kSesmThreads) {
            spt = cand;
            t = tt;
            break;
        }
    }
    if (!spt || m.vertices > kSesmVpt * t) return plan;
    const SmemLayout L = smem_layout(m);
    size_t budget = (size_t)smem_optin - 1024;
    const size_t share = (size_t)smem_sm / (size_t)blocks_per_sm;
    if (share < 2048) return plan;
    budget = std::min(budget, share - 2048);
    if (L.total_cached > budget || m.csr >= 65536 || m.slots >= 16384) return plan;
    for (int nonlin = 0; nonlin < 2; nonlin++) {
        void *fn = sesm_kernel(spt, nonlin);
        int occ = 0;
        if (!fn || raise_smem_limit(fn) < (int)L.total_cached ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, t, L.total_cached) != cudaSuccess ||
            occ < blocks_per_sm) {
            cudaGetLastError();
            return plan;
        }
    }
    plan.slots_per_thread = spt;
    plan.threads = t;
    plan.cached = 1;
    plan.blocks_per_sm = blocks_per_sm;
    plan.smem = L.total_cached;
    return plan;
}

PersistentPlan persistent_plan_sesm_teams(const PatchMax &m, int blocks_per_sm)
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
    if (m.deg > 16) return plan;   // such meshes stream (k_persistent_sesm_stream)
    const int teams = std::min(std::max(blocks_per_sm, 1), kMaxTeams);
    const int max_threads = kSesmTeamThreads / teams / 32 * 32;
    if (smem_optin < 2048 || smem_sm < 4096) return plan;
    const size_t budget = std::min((size_t)smem_optin - 1024, (size_t)smem_sm - 2048);
    for (int spt = 4; spt <= 7; spt++) {
        const int t = std::max(32, ((m.slots + spt - 1) / spt + 31) / 32 * 32);
        if (t > max_threads) continue;
        const unsigned cols = tmem_columns(teams * t, sesm_words(spt));
        int wide = 1;
        size_t team_smem = 0, smem = 0;
        for (; wide >= 0; wide--) {
            team_smem = sesm_layout(m, wide).total;
            smem = std::max(teams * team_smem, tmem_smem_floor(cols, (size_t)smem_sm));
            if (smem <= budget) break;
        }
        if (wide < 0 || cols > 512u) return plan;
        for (int nonlin = 0; nonlin < 2; nonlin++) {
            void *fn = sesm_teams_kernel(spt, nonlin);
            int occ = 0;
            if (!fn || raise_smem_limit(fn) < (int)smem ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, teams * t, smem) != cudaSuccess || occ < 1) {
                cudaGetLastError();
                return plan;
            }
        }
        plan.slots_per_thread = spt;
        plan.threads = t;
        plan.cached = 1;
        plan.stream = 1;
        plan.wide_rows = wide;
        plan.blocks_per_sm = blocks_per_sm;
        plan.teams = teams;
        plan.team_smem = (int)team_smem;
        plan.tmem_cols = (int)cols;
        plan.grid = nsm;
        plan.smem = smem;
        return plan;
    }
    return plan;
}

cudaError_t persistent_prepare_sesm(const PersistentPlan &plan)
{
    for (int nonlin = 0; nonlin < 2; nonlin++) {
        void *fn = plan.teams ? sesm_teams_kernel(plan.slots_per_thread, nonlin)
                              : sesm_kernel(plan.slots_per_thread, nonlin);
        if (!fn || raise_smem_limit(fn) < (int)plan.smem) return cudaErrorInvalidValue;
    }
    return cudaSuccess;
}

cudaError_t launch_persistent_sesm(const DevMesh &m, const DevState &s, const StepArgs &a, int M, int parity, int nsteps,
                                   const std::vector<PackPlan> &packs, cudaStream_t stream)
{
    // one cooperative launch per pack, each with its own plan, layout and tag base
    for (size_t k = 0; k < packs.size(); k++) {
        const PackPlan &pk = packs[k];
        const PersistentPlan &pl = pk.plan_sesm;
        if (pl.stream && !pl.teams) {
            if (nsteps != 1) return cudaErrorInvalidValue;   // one step per launch
            const cudaError_t e = launch_persistent_sesm_stream_pack(m, s, a, M, parity, pk, (int)k, stream);
            if (e != cudaSuccess) return e;
            continue;
        }
        void *fn = pl.teams ? sesm_teams_kernel(pl.slots_per_thread, a.nonlinear_h)
                            : sesm_kernel(pl.slots_per_thread, a.nonlinear_h);
        if (!fn) return cudaErrorInvalidValue;
        PArgs P = make_pargs(m, s, a, M, parity, pk.mx);
        P.pack_base = pk.base;
        P.pack_index = (int)k;
        P.npb = pk.nblocks;
        P.nsteps = nsteps;
        int grid = pk.nblocks, threads = pl.threads;
        if (pl.teams) {
            set_layout(P, sesm_layout(pk.mx, pl.wide_rows), pk.mx);
            P.tmem_cols = (unsigned)pl.tmem_cols;
            P.team_threads = pl.threads;
            P.team_smem = pl.team_smem;
            grid = std::min(pl.grid, pk.nblocks);
            threads = pl.teams * pl.threads;
        }
        void *args[] = {&P};
        const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(grid), dim3(threads), args, pl.smem, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace sesw
