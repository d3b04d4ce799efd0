// The SE step kernel for small meshes (sm_103a): one thread-block cluster advances the whole mesh, all
// substeps of P.nsteps baroclinic steps in one launch, exchanging the elevation through the
// cluster's distributed shared memory.
//
// On a small mesh a substep of k_persistent is one chain of latencies: the new elevation goes to L2
// and comes back as a tagged word (about 0.7 us), between three block barriers and two short
// passes. Here every block of the cluster keeps the elevation of the whole mesh in shared memory
// (two levels); the owner of a vertex sends the new value into the blocks that read it, and each
// block waits until the values it reads have arrived (st.async counting bytes on an mbarrier: one
// way, where a cluster barrier after plain remote stores costs two round trips). Fewer SMs work
// (16 of 152), so this pays as long as the chain and not the work bounds the substep: one slot per
// thread, its static data and state in registers. us per 160 substeps with the state transfers,
// k_persistent and here: 720 vertices 183 and 125, 2000 196 and 136, 3905 192 and 154, 4800 185 and
// 171. With two slots per thread it was the slower one (8800 vertices: 189 and 217).
//
// Levels and barriers alternate with the substep. A block sends level m + 1 in its vertex pass m;
// it writes a reader's level again in pass m + 2, which follows its wait for the reader's values
// of pass m + 1, sent after the reader's last use of that level (who reads from a block is also
// read by it: a triangle across the border has a copy on both sides).
#include "sesw_persistent.cuh"

namespace sesw {

namespace {

struct CArgs {
    PArgs P;
    const int *grp;              // [cluster + 1] patch ranges of the blocks
    const unsigned *readers;     // per vertex: bit b set when block b, not the owner, reads it
    const int *halo;             // per block: vertices that it reads and does not own
    int nv;
    int off_eta, off_mask;       // shared memory: two levels of elevation, interleaved; readers of the own vertices
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// All earlier stores of the cluster's threads, remote ones too, are visible after the barrier.
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Send v to the shared-memory address of block `rank` that `local` is here, counting 4 bytes on that
// block's mbarrier.
__device__ __forceinline__ void send(uint32_t local, uint32_t bar, uint32_t rank, float v)
{
    uint32_t ra, rb;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(bar), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(ra),
                 "r"(__float_as_uint(v)), "r"(rb)
                 : "memory");
}

// Bounded wait for phase `parity` of an mbarrier of this block; false when the budget ran out.
__device__ __forceinline__ bool wait_phase(uint32_t bar, uint32_t parity, long long budget)
{
    const long long t0 = clock64();
    while (true) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
        if (clock64() - t0 > budget) return false;
    }
}

template <int NONLIN, int EXTRA>
__global__ void __launch_bounds__(1024, 1) k_cluster(const CArgs A)
{
    const PArgs &P = A.P;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_stop;
    __shared__ __align__(8) uint64_t s_bar[2];
    const int tid = threadIdx.x, T = blockDim.x;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(s_bar);
    if (tid == 0) {
        s_stop = 0;
        for (int k = 0; k < 2; k++)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar + 8u * k), "r"(1));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const uint32_t rank = cluster_rank();
    const unsigned halo_bytes = 4u * (unsigned)A.halo[rank];
    const int p0 = A.grp[rank], p1 = A.grp[rank + 1];
    const int s0 = P.patch_slot[p0], ns = P.patch_slot[p1] - s0;
    const int v0 = P.patch_v[p0], nown = P.patch_v[p1] - v0;
    const StepArgs a = P.a;
    const float dt = P.patch_dt[p0];             // one mesh, one substep length
    const bool silent = a.silent_patch >= p0 && a.silent_patch < p1;   // failure test: sends nothing in the last step
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(smem);
    const uint32_t eta = base + (uint32_t)A.off_eta, rows = base + (uint32_t)P.off_flux;
    const uint32_t dummy = base + (uint32_t)P.off_dummy + 4u * (tid & 31);
    float *s_inv = reinterpret_cast<float *>(smem + P.off_inv);
    unsigned *s_mask = reinterpret_cast<unsigned *>(smem + A.off_mask);

    for (int v = tid; v < A.nv; v += T) sts(eta + 8u * (uint32_t)v, P.eta_in[v]);
    for (int i = tid; i < P.row_quads * P.row_vertices; i += T)
        reinterpret_cast<float4 *>(smem + P.off_flux)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int i = tid; i < nown; i += T) {
        s_inv[i] = P.inv_av[v0 + i];
        s_mask[i] = silent && P.nsteps == 1 ? 0u : A.readers[v0 + i];
    }
    // threads without a slot hold an all-zero one (see k_persistent)
    SlotData q;
    float2 u, shi = make_float2(0.0f, 0.0f), slo = shi;
    {
        const bool in = tid < ns;
        const int s = s0 + (in ? tid : 0);
        const int4 v = P.sv[s];
        const uint2 f = in ? P.sf[s] : make_uint2(0xffffffffu, 0x7fffffffu);
        // the flux of a corner that its slot's patch owns: its place in the vertex's row (at most 16)
        auto place = [&](uint32_t e, int vc) {
            return e == 0x1fffffu
                       ? dummy
                       : rows + 16u * ((e >> 2) * (uint32_t)P.row_vertices + (uint32_t)(vc - v0)) + 4u * (e & 3u);
        };
        q.g = in ? P.sg[s] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        q.c = in ? P.sk[s] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        q.r = in ? P.R[s] : make_float2(0.0f, 0.0f);
        q.a0 = eta + 8u * (uint32_t)v.x;
        q.a1 = eta + 8u * (uint32_t)v.y;
        q.a2 = eta + 8u * (uint32_t)v.z;
        q.f0 = place(f.x & 0x1fffffu, v.x);
        q.f1 = place((f.x >> 21) | ((f.y & 0x3ffu) << 11), v.y);
        q.f2 = place((f.y >> 10) & 0x1fffffu, v.z);
        u = in ? P.U[s] : make_float2(0.0f, 0.0f);
    }
    cluster_sync();       // every block's elevation and barriers are in place before anything is sent

    const float one_p_theta = __fadd_rn(1.0f, a.theta);
    const int total = P.M * P.nsteps;
    // one substep from level L of the elevation (byte offset) to the other
    auto substep = [&](const int m, const int ms, const uint32_t L) {
        {
            const float e0 = lds(q.a0 + L), e1 = lds(q.a1 + L), e2 = lds(q.a2 + L);
            const float2 F = se_transport<NONLIN, 1>(e0, e1, e2, q.g, q.c.y, a.g, q.c.z, q.c.w, dt, q.r, one_p_theta,
                                                     a.theta, u);
            two_sum_acc2<0>(shi, slo, F);
            float f3[3];
            corner_fluxes<0>(F, q.g, q.c.x, f3);
            sts(q.f0, f3[0]);
            sts(q.f1, f3[1]);
            sts(q.f2, f3[2]);
        }
        __syncthreads();
        const bool more = m + 1 < total;
        const uint32_t mbar = bar + 8u * (uint32_t)(m & 1);
        if (more && tid == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(halo_bytes) : "memory");
        bool bad = false;
        for (int i = tid; i < nown; i += T) {
            float sum = 0.0f;
            uint32_t row = rows + 16u * (uint32_t)i;
            for (int k = 0; k < P.row_quads; k++, row += 16u * (uint32_t)P.row_vertices) {
                const float4 c = lds4(row);
                sum = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(sum, c.x), c.y), c.z), c.w);
            }
            const uint32_t at = eta + 8u * (uint32_t)(v0 + i);
            const float e0 = lds(at + L);
            float e = vertex_eta(e0, sum, s_inv[i]);
            if (EXTRA) {
                if (P.W) e = __fmaf_rn(-dt, __ldg(P.W + v0 + i), e);
                if (P.eta_sum) P.eta_sum[v0 + i] = (ms == 0 ? 0.0f : P.eta_sum[v0 + i]) + e0;
            }
            sts(at + (L ^ 4u), e);
            if (more)
                for (unsigned r = s_mask[i]; r; r &= r - 1) send(at + (L ^ 4u), mbar, (uint32_t)__ffs((int)r) - 1u, e);
            bad |= !(fabsf(e) <= a.eta_bound);
        }
        if (bad) atomicOr(P.status, 1u);
        if (more && !wait_phase(mbar, (uint32_t)(m >> 1) & 1u, a.wait_cycles)) {
            // gives up: flags the timeout, and gives the values in flight one more budget to land
            atomicOr(P.status, 2u);
            wait_phase(mbar, (uint32_t)(m >> 1) & 1u, a.wait_cycles);
            s_stop = 1;
        }
        __syncthreads();
    };
    for (int m = 0, ms = 0; m < total; m++) {
        if (m & 1) substep(m, ms, 4u); else substep(m, ms, 0u);
        if (s_stop) break;
        if (++ms == P.M && m + 1 < total) {
            // a step ends: the sums of the next one start from zero
            ms = 0;
            shi = slo = make_float2(0.0f, 0.0f);
            if (silent && m + 1 + P.M == total)
                for (int i = tid; i < nown; i += T) s_mask[i] = 0u;
        }
    }
    const uint32_t last = eta + ((total & 1) ? 4u : 0u);
    for (int i = tid; i < nown; i += T) P.eta_out[v0 + i] = lds(last + 8u * (uint32_t)(v0 + i));
    if (tid < ns) {
        P.U[s0 + tid] = u;
        const int w = P.sv[s0 + tid].w;
        if (w >= 0) P.Umean[w] = make_float2((shi.x + slo.x) * a.inv_M, (shi.y + slo.y) * a.inv_M);
    }
    cluster_sync();       // no block leaves while another may still send to it
}

void *cluster_kernel(int nonlin, int extra)
{
    if (extra) return nonlin ? (void *)k_cluster<1, 1> : (void *)k_cluster<0, 1>;
    return nonlin ? (void *)k_cluster<1, 0> : (void *)k_cluster<0, 0>;
}

// Shared memory of a block: the flux rows and dummy words of its vertices, 1/A_v, readers, and two
// levels of the whole mesh's elevation.
struct ClusterLayout {
    size_t dummy, inv, mask, eta, total;
    int quads;
};

ClusterLayout cluster_layout(int nv, int own, int deg)
{
    ClusterLayout L;
    L.quads = std::max(2, (deg + 3) / 4);
    L.dummy = 16 * (size_t)L.quads * (size_t)own;
    L.inv = L.dummy + 128;
    L.mask = L.inv + align16(4 * (size_t)own);
    L.eta = L.mask + align16(4 * (size_t)own);
    L.total = L.eta + align16(8 * (size_t)nv);
    return L;
}

cudaLaunchConfig_t cluster_config(const ClusterPlan &pl, cudaStream_t stream, cudaLaunchAttribute *attr)
{
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)pl.blocks;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)pl.blocks);
    cfg.blockDim = dim3((unsigned)pl.threads);
    cfg.dynamicSmemBytes = pl.smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

}  // namespace

ClusterPlan cluster_plan(const HostMesh &hm, int deg, std::vector<int> &grp, std::vector<unsigned> &readers,
                         std::vector<int> &halo)
{
    ClusterPlan pl;
    int dev = 0, smem_optin = 0, smem_sm = 0;
    if (hm.nbasin != 1 || deg > 16 || hm.nslot > 16 * 1024 || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess) {
        cudaGetLastError();
        return pl;
    }
    for (int blocks : {16, 8}) {
        if (hm.npatch < blocks) continue;
        // consecutive patches, as many slots per block as possible alike
        grp.assign(1, 0);
        int slots = 0, own = 0;
        for (int b = 1; b <= blocks; b++) {
            const long long want = (long long)hm.nslot * b / blocks;
            int p = grp.back() + 1;
            while (p < hm.npatch - (blocks - b) && hm.patch_slot[p] < want) p++;
            if (b == blocks) p = hm.npatch;
            slots = std::max(slots, hm.patch_slot[p] - hm.patch_slot[grp.back()]);
            own = std::max(own, hm.patch_v[p] - hm.patch_v[grp.back()]);
            grp.push_back(p);
        }
        if (slots > 1024) continue;            // one slot per thread
        pl.threads = std::max(32, (slots + 31) / 32 * 32);
        pl.own = own;
        pl.deg = deg;
        pl.smem = cluster_layout(hm.nv, own, deg).total;
        bool fits = pl.smem <= std::min((size_t)smem_optin - 1024, (size_t)smem_sm - 2048);
        pl.blocks = blocks;
        for (int nonlin = 0; nonlin < 2 && fits; nonlin++)
            for (int extra = 0; extra < 2 && fits; extra++) {
                void *fn = cluster_kernel(nonlin, extra);
                cudaLaunchAttribute attr;
                const cudaLaunchConfig_t cfg = cluster_config(pl, nullptr, &attr);
                int nc = 0;
                fits = fn && raise_smem_limit(fn) >= (int)pl.smem &&
                       cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                       cudaOccupancyMaxActiveClusters(&nc, fn, &cfg) == cudaSuccess && nc >= 1;
            }
        if (!fits) {
            cudaGetLastError();
            pl = ClusterPlan();
            continue;
        }
        // the blocks that read a vertex without owning it
        readers.assign(hm.nv, 0u);
        for (int b = 0; b < blocks; b++)
            for (int s = hm.patch_slot[grp[b]]; s < hm.patch_slot[grp[b + 1]]; s++) {
                const int4 c = hm.slot_v[s];
                for (int v : {c.x, c.y, c.z})
                    if (v < hm.patch_v[grp[b]] || v >= hm.patch_v[grp[b + 1]]) readers[v] |= 1u << b;
            }
        halo.assign(blocks, 0);
        for (unsigned r : readers)
            for (int b = 0; b < blocks; b++) halo[b] += (int)(r >> b & 1u);
        return pl;
    }
    return ClusterPlan();
}

cudaError_t launch_cluster(const DevMesh &m, const DevState &s, const StepArgs &a, int M, int parity, int nsteps,
                           cudaStream_t stream)
{
    const ClusterPlan &pl = m.cluster;
    void *fn = cluster_kernel(a.nonlinear_h, s.W != nullptr || s.eta_sum != nullptr);
    if (!fn) return cudaErrorInvalidValue;
    PatchMax mx;
    CArgs A;
    A.P = make_pargs(m, s, a, M, parity, mx);
    const ClusterLayout L = cluster_layout(m.nv, pl.own, pl.deg);
    A.P.off_flux = 0;
    A.P.off_dummy = (int)L.dummy;
    A.P.off_inv = (int)L.inv;
    A.P.row_quads = L.quads;
    A.P.row_vertices = pl.own;
    A.P.nsteps = nsteps;
    A.grp = m.cluster_grp;
    A.readers = m.cluster_readers;
    A.halo = m.cluster_halo;
    A.nv = m.nv;
    A.off_mask = (int)L.mask;
    A.off_eta = (int)L.eta;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(pl, stream, &attr);
    void *args[] = {&A};
    return cudaLaunchKernelExC(&cfg, fn, args);
}

}  // namespace sesw
