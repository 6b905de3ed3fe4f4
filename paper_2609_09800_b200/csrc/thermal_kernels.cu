// Kernels of hbf_thermal_step: power map -> explicit Euler substeps of the RC network (Eq. 1) ->
// hotspots and the four-state throttle controller.
//
// The field is kept as the rise above ambient, theta, in float32 with a float32 compensation term per
// cell (Kahan summation of the substep increments): plain float32 accumulation drifts by several mK over
// 10^4..10^5 substeps and stalls once an increment drops under half an ulp of the state.
#include <algorithm>
#include <mutex>
#include <vector>

#include <cooperative_groups.h>

#include "device_utils.cuh"

namespace cg = cooperative_groups;

namespace hbf {

// Power of each region over the window: sum of its dies' energy / dt (pJ/ns = mW), idle and external
// power; then spread evenly over the region's cells.  One thread per region walks that region's dies in
// a fixed order, so the sum is reproducible.  The window's energy is consumed.
__global__ void k_power_map(ThermalDev t, int64_t *pending, int64_t dt_ns, int has_ext) {
    const int tid = threadIdx.x;
    for (uint32_t g = tid; g < t.n_regions; g += blockDim.x) {
        double p = 0.0;
        for (int32_t k = t.region_die_ptr[g]; k < t.region_die_ptr[g + 1]; ++k)
            p += ((double)pending[t.region_die_list[k]] * 1e-12) / ((double)dt_ns * 1e-9);
        p += (double)t.region_idle_w[g];
        if (has_ext) p += (double)t.ext_power[g];
        t.region_power[g] = p;
    }
    __syncthreads();
    const uint32_t nc = t.H * t.W;
    for (uint32_t i = tid; i < nc; i += blockDim.x) {
        const int32_t g = t.cell_region[i];
        t.P[i] = g >= 0 ? (float)(t.region_power[g] * (double)t.region_inv_cells[g]) : 0.0f;
    }
    for (uint32_t d = tid; d < t.n_dies; d += blockDim.x) pending[d] = 0;
}

// One explicit Euler substep, every cell from the previous substep's field (Jacobi).
__global__ void __launch_bounds__(256)
k_euler_substep(ThermalDev t, const float *__restrict__ th_in, float *__restrict__ th_out, float dt_sub) {
    const uint32_t x = blockIdx.x * 32 + (threadIdx.x & 31), y = blockIdx.y * 8 + (threadIdx.x >> 5);
    if (x >= t.W || y >= t.H) return;
    const uint32_t W = t.W, H = t.H, i = y * W + x;
    const float Ti = th_in[i];
    float flow = 0.0f;
    if (x + 1 < W) flow += t.Gx[i] * (Ti - th_in[i + 1]);
    if (x > 0)     flow += t.Gx[i - 1] * (Ti - th_in[i - 1]);
    if (y + 1 < H) flow += t.Gy[i] * (Ti - th_in[i + W]);
    if (y > 0)     flow += t.Gy[i - W] * (Ti - th_in[i - W]);
    const float inc = dt_sub / t.C[i] * (t.P[i] - flow - t.Gs[i] * Ti);
    const float yv = inc - t.comp[i];
    const float tn = Ti + yv;
    t.comp[i] = (tn - Ti) - yv;
    th_out[i] = tn;
}

__device__ __forceinline__ long long quantise_mk(float t_c) { return (long long)floor((double)t_c * 1000.0 + 0.5); }

__device__ __forceinline__ int next_mode(const ThermalDev &t, int mode, long long mk) {
    if (mode == HBF_MODE_SHUTDOWN || mk >= t.shut_mk) return HBF_MODE_SHUTDOWN;
    if (mode == HBF_MODE_NORMAL) return mk >= t.stt_mk ? HBF_MODE_SEVERE : mk >= t.ltt_mk ? HBF_MODE_LIGHT : HBF_MODE_NORMAL;
    if (mode == HBF_MODE_LIGHT) return mk >= t.stt_mk ? HBF_MODE_SEVERE : mk <= t.rtt_mk ? HBF_MODE_NORMAL : HBF_MODE_LIGHT;
    return mk <= t.rtt_mk ? HBF_MODE_NORMAL : mk <= t.ltt_mk ? HBF_MODE_LIGHT : HBF_MODE_SEVERE;
}

// Hottest cell per medium, the controller's transition on the HBF hotspot (quantised to integer mK),
// and the published mode / service fraction for the next batch.
__global__ void __launch_bounds__(1024)
k_controller(ThermalDev t, const float *__restrict__ th, DevState *state, float *temps_out) {
    __shared__ float s_hot[3][32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float hot[3] = {-INFINITY, -INFINITY, -INFINITY};
    const uint32_t nc = t.H * t.W;
    for (uint32_t i = tid; i < nc; i += blockDim.x) {
        const float T = t.ambient_c + th[i];
        if (temps_out) temps_out[i] = T;
        const int32_t g = t.cell_region[i];
        if (g < 0) continue;
        const int32_t k = t.region_kind[g];
        const int slot = k == HBF_KIND_HBF ? 0 : k == HBF_KIND_HBM ? 1 : k == HBF_KIND_GPU ? 2 : -1;
        if (slot == 0) hot[0] = fmaxf(hot[0], T); else if (slot == 1) hot[1] = fmaxf(hot[1], T); else if (slot == 2) hot[2] = fmaxf(hot[2], T);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o > 0; o >>= 1) hot[k] = fmaxf(hot[k], __shfl_xor_sync(0xffffffffu, hot[k], o));
        if (lane == 0) s_hot[k][warp] = hot[k];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            float v = lane < (int)(blockDim.x >> 5) ? s_hot[k][lane] : -INFINITY;
            for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
            hot[k] = v == -INFINITY ? t.ambient_c : v;
        }
        if (lane == 0) {
            t.hot[0] = hot[0]; t.hot[1] = hot[1]; t.hot[2] = hot[2];
            const int mode = next_mode(t, state->mode, quantise_mk(hot[0]));
            state->mode = mode;
            if (mode == HBF_MODE_NORMAL) state->q_ppm = 1000000;
            else if (mode == HBF_MODE_LIGHT) state->q_ppm = t.q_light_ppm;
        }
    }
}

static cudaError_t launch_thermal_generic(const ThermalDev &t, DevState *state, int64_t *pending, int64_t dt_ns, int has_ext,
                                          float *d_temps_out, int *cur, cudaStream_t st) {
    k_power_map<<<1, 1024, 0, st>>>(t, pending, dt_ns, has_ext);
    const float dt_sub = (float)((double)dt_ns * 1e-9 / (double)t.n_sub);
    dim3 grid((t.W + 31) / 32, (t.H + 7) / 8);
    int c = *cur;
    for (uint32_t k = 0; k < t.n_sub; ++k) {
        k_euler_substep<<<grid, 256, 0, st>>>(t, t.theta[c], t.theta[c ^ 1], dt_sub);
        c ^= 1;
    }
    *cur = c;
    g_kernel_launches += 2ull + t.n_sub;
    k_controller<<<1, 1024, 0, st>>>(t, t.theta[c], state, d_temps_out);
    return cudaGetLastError();
}


// ======================================================================================================
// The whole step in one launch, for grids that fit the shared memory of one thread-block cluster: the blocks each keep a
// band of rows of the field (both Jacobi buffers, with one halo row above and below) in shared memory and every cell's
// constants, power and compensation term in registers.  After each substep a block sends its first and last row into its
// neighbours' halo rows (st.async, counted in bytes by a barrier in the neighbour's shared memory): a block waits for its two
// neighbours only, not for the whole cluster.  A neighbour cannot run ahead into a buffer that is still read: it needs this
// block's rows of a substep before it starts the next.  The arithmetic of a cell is the same, in the same order, as in
// k_euler_substep (a missing neighbour has conductance 0, which adds nothing); the power map is formed by every block for its
// own cells and the hotspots are reduced through block 0.
// 16,384 cells are far too few to fill the device: a step lasts as long as its chain of substeps (read the neighbours, twelve
// dependent operations, send, wait).  With CPT cells per thread known at compile time, no tests and no division in the
// substep, and waits for neighbours only: see launch_thermal_step for what it measured.
// ======================================================================================================
constexpr int kThClusterBlocks = 16;                       // blocks of the cluster when the device takes that many (not a portable size), else 8
constexpr int kThClusterPortable = 8;
constexpr int kThThreads = 512;
constexpr int kThCellsPerThread = 8;
constexpr int kThMaxRegions = 1024;
constexpr uint32_t kThTermDies = 1024;                     // dies whose power terms are formed a thread each
constexpr uint32_t kThWaitPolls = 1u << 22;

__device__ __forceinline__ uint32_t th_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t th_remote(uint32_t addr, uint32_t rank) {
    uint32_t r; asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank)); return r;
}
__device__ __forceinline__ void th_send(uint32_t addr, float v, uint32_t bar) {
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.u32 [%0], %1, [%2];" ::"r"(addr), "r"(__float_as_uint(v)), "r"(bar) : "memory");
}
__device__ __forceinline__ bool th_poll(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0u;
}

template <int CPT>
__global__ void __launch_bounds__(kThThreads, 1)
k_thermal_cluster(const __grid_constant__ ThermalDev t, float *theta, DevState *state, int64_t *pending, unsigned long long *bin_row, int64_t dt_ns,
                  int has_ext, float dt_sub, float *temps_out) {
    extern __shared__ __align__(16) unsigned char th_smem_buf[];
    __shared__ double s_region_power[kThMaxRegions];
    __shared__ double s_term[kThTermDies];
    __shared__ float s_hot[kThClusterBlocks][3];
    __shared__ float s_part[3][kThThreads / 32];
    __shared__ __align__(8) uint64_t s_bar[2];
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), n_blocks = cluster.num_blocks();      // (the cluster's size is chosen at launch)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t H = t.H, W = t.W;
    const uint32_t rows = (H + n_blocks - 1) / n_blocks;
    const uint32_t y0 = min(H, rank * rows), y1 = min(H, y0 + rows);
    const uint32_t band_cells = (y1 - y0) * W;
    const uint32_t pitch = (rows + 2) * W;                    // one buffer: halo row, band, halo row
    float *buf0 = reinterpret_cast<float *>(th_smem_buf);
    const bool has_up = rank > 0u && y1 > y0, has_down = y1 < H && y1 > y0;
    if (tid < 2) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(th_smem(&s_bar[tid])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // what no kernel changes: this thread's cells' constants
    float kC[CPT], gE[CPT], gW_[CPT], gS[CPT], gN[CPT], gs[CPT], P[CPT], cmp[CPT];
    uint32_t off[CPT], up[CPT], down[CPT];                    // place in a buffer; the same cell in the neighbours' halo rows (0: not a boundary row)
    int32_t region[CPT];
    bool live[CPT];
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        const uint32_t li = (uint32_t)c * kThThreads + tid;   // cell of the band, row-major
        live[c] = li < band_cells;
        off[c] = W; up[c] = down[c] = 0u; region[c] = -1;
        kC[c] = gE[c] = gW_[c] = gS[c] = gN[c] = gs[c] = P[c] = cmp[c] = 0.0f;
        if (live[c]) {
            const uint32_t r = li / W, x = li - r * W, y = y0 + r;
            const uint64_t i = (uint64_t)y * W + x;
            off[c] = (r + 1) * W + x;
            kC[c] = dt_sub / t.C[i];
            if (x + 1 < W) gE[c] = t.Gx[i];
            if (x > 0) gW_[c] = t.Gx[i - 1];
            if (y + 1 < H) gS[c] = t.Gy[i];
            if (y > 0) gN[c] = t.Gy[i - W];
            gs[c] = t.Gs[i];
            region[c] = t.cell_region[i];
            const uint32_t b0 = th_smem(buf0);
            if (r == 0u && has_up) up[c] = th_remote(b0 + ((rows + 1) * W + x) * 4u, rank - 1u);              // (a block above another is full: its lower halo row sits behind `rows` rows)
            if (r + 1u == y1 - y0 && has_down) down[c] = th_remote(b0 + x * 4u, rank + 1u);
        }
    }
    const uint32_t bar0 = th_smem(&s_bar[0]);
    const uint32_t up_bar = has_up ? th_remote(bar0, rank - 1u) : 0u, down_bar = has_down ? th_remote(bar0, rank + 1u) : 0u;
    const uint32_t expect = ((has_up ? 1u : 0u) + (has_down ? 1u : 0u)) * W * 4u;
    pdl_wait();                                               // from here on: what the kernels before left
    pdl_trigger();
    // field: own rows and the neighbours' boundary rows, from global memory (the second buffer's rows outside the grid stay 0)
    for (uint32_t i = tid; i < pitch; i += kThThreads) {
        const uint32_t r = i / W, x = i - r * W;
        const int64_t y = (int64_t)y0 + r - 1;
        buf0[i] = (r < y1 - y0 + 2 && y >= 0 && y < (int64_t)H) ? theta[(uint64_t)y * W + x] : 0.0f;
        buf0[pitch + i] = 0.0f;
    }
#pragma unroll
    for (int c = 0; c < CPT; ++c) if (live[c]) cmp[c] = t.comp[(uint64_t)y0 * W + (uint32_t)c * kThThreads + tid];
    // power of every region over the window (every block forms the same values, summed in the order of the region's dies), then
    // of this block's cells.  The ledger's bin, when there is one, is taken with the pending totals.
    auto term = [&](uint32_t d) {
        const int64_t e = pending[d] + (bin_row ? (int64_t)bin_row[d] : 0);
        return ((double)e * 1e-12) / ((double)dt_ns * 1e-9);
    };
    const bool by_die = t.n_dies <= kThTermDies;
    if (by_die) {
        for (uint32_t d = tid; d < t.n_dies; d += kThThreads) s_term[d] = term(d);
        __syncthreads();
    }
    for (uint32_t g = tid; g < t.n_regions; g += kThThreads) {
        double p = 0.0;
        const int32_t k0 = t.region_die_ptr[g], k1 = t.region_die_ptr[g + 1];
        for (int32_t k = k0; k < k1; k += 8) {
            uint32_t d[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) d[j] = k + j < k1 ? (uint32_t)t.region_die_list[k + j] : 0u;
#pragma unroll
            for (int j = 0; j < 8; ++j) if (k + j < k1) p += by_die ? s_term[d[j]] : term(d[j]);
        }
        p += (double)t.region_idle_w[g];
        if (has_ext) p += (double)t.ext_power[g];
        s_region_power[g] = p;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < CPT; ++c) if (region[c] >= 0) P[c] = (float)(s_region_power[region[c]] * (double)t.region_inv_cells[region[c]]);
    cluster.sync();                                           // every block's buffers and barriers stand, and every block has read the energies
    if (rank == 0)
        for (uint32_t d = tid; d < t.n_dies; d += kThThreads) { pending[d] = 0; if (bin_row) bin_row[d] = 0ull; }

    bool lost = false;
    for (uint32_t k = 0; k < t.n_sub; ++k) {
        const uint32_t ob = (k + 1u) & 1u;                    // the buffer written
        const float *in = buf0 + (k & 1u) * pitch;
        float *out = buf0 + ob * pitch;
        const bool more = k + 1u < t.n_sub;
        if (more && expect && tid == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar0 + ob * 8u), "r"(expect) : "memory");
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
            if (live[c]) {
                const uint32_t o = off[c];
                const float Ti = in[o];
                float flow = 0.0f;
                flow += gE[c] * (Ti - in[o + 1]);
                flow += gW_[c] * (Ti - in[o - 1]);
                flow += gS[c] * (Ti - in[o + W]);
                flow += gN[c] * (Ti - in[o - W]);
                const float inc = kC[c] * (P[c] - flow - gs[c] * Ti);
                const float yv = inc - cmp[c];
                const float tn = Ti + yv;
                cmp[c] = (tn - Ti) - yv;
                out[o] = tn;
                if (more) {
                    if (up[c]) th_send(up[c] + ob * pitch * 4u, tn, up_bar + ob * 8u);
                    if (down[c]) th_send(down[c] + ob * pitch * 4u, tn, down_bar + ob * 8u);
                }
            }
        }
        if (more && expect && !lost) {
            uint32_t polls = 0;
            while (!th_poll(bar0 + ob * 8u, (k >> 1) & 1u)) if (++polls > kThWaitPolls) { lost = true; break; }
        }
        __syncthreads();
    }
    if (lost) state->poisoned = 1;                            // a neighbour's rows never came: the context is given up
    // results: field and compensation back to global memory, hotspots to block 0
    const float *in = buf0 + (t.n_sub & 1u) * pitch;
    float hot[3] = {-INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        if (live[c]) {
            const uint64_t i = (uint64_t)y0 * W + (uint32_t)c * kThThreads + tid;
            const float th = in[off[c]];
            theta[i] = th; t.comp[i] = cmp[c];
            const float T = t.ambient_c + th;
            if (temps_out) temps_out[i] = T;
            if (region[c] >= 0) {
                const int32_t kind = t.region_kind[region[c]];
                if (kind == HBF_KIND_HBF) hot[0] = fmaxf(hot[0], T); else if (kind == HBF_KIND_HBM) hot[1] = fmaxf(hot[1], T);
                else if (kind == HBF_KIND_GPU) hot[2] = fmaxf(hot[2], T);
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        for (int o = 16; o > 0; o >>= 1) hot[k] = fmaxf(hot[k], __shfl_xor_sync(0xffffffffu, hot[k], o));
        if (lane == 0) s_part[k][warp] = hot[k];
    }
    __syncthreads();
    if (tid < 3) {
        float v = -INFINITY;
        for (int w = 0; w < kThThreads / 32; ++w) v = fmaxf(v, s_part[tid][w]);
        float *dst = cluster.map_shared_rank(&s_hot[0][0], 0);
        dst[rank * 3 + tid] = v;
    }
    cluster.sync();
    if (rank == 0 && tid == 0) {
        float h[3];
        for (int k = 0; k < 3; ++k) {
            float v = -INFINITY;
            for (uint32_t b = 0; b < n_blocks; ++b) v = fmaxf(v, s_hot[b][k]);
            h[k] = v == -INFINITY ? t.ambient_c : v;
            t.hot[k] = h[k];
        }
        const int mode = next_mode(t, state->mode, quantise_mk(h[0]));
        state->mode = mode;
        if (mode == HBF_MODE_NORMAL) state->q_ppm = 1000000;
        else if (mode == HBF_MODE_LIGHT) state->q_ppm = t.q_light_ppm;
    }
}

using ThermalKernel = void (*)(const ThermalDev, float *, DevState *, int64_t *, unsigned long long *, int64_t, int, float, float *);
// the kernel whose threads hold just as many cells as the grid needs on a cluster of n_blocks
static ThermalKernel thermal_cluster_kernel(const ThermalDev &t, int n_blocks) {
    const uint64_t cells = (uint64_t)((t.H + n_blocks - 1) / n_blocks) * t.W;
    return cells <= 1u * kThThreads ? k_thermal_cluster<1> : cells <= 2u * kThThreads ? k_thermal_cluster<2> : cells <= 4u * kThThreads ? k_thermal_cluster<4>
                                                                                                               : k_thermal_cluster<kThCellsPerThread>;
}

static bool thermal_cluster_fits(const ThermalDev &t, int n_blocks, size_t *smem_bytes) {
    const uint32_t rows = (t.H + n_blocks - 1) / n_blocks;
    const size_t smem = (size_t)2 * (rows + 2) * t.W * sizeof(float);
    *smem_bytes = smem;
    return (size_t)rows * t.W <= (size_t)kThThreads * kThCellsPerThread && smem <= 200u * 1024u && t.n_regions <= (uint32_t)kThMaxRegions;
}

// How many blocks the cluster of the one-launch step gets on the current device: 16 where the device can place such a
// cluster (a size beyond the portable 8 has to be allowed per kernel), else 8; 0 when the grid does not fit either.  Asked
// once per (device, shared-memory size) and remembered.
static int thermal_cluster_blocks(const ThermalDev &t, size_t *smem_bytes) {
    struct Entry { int device; size_t smem16; const void *fn; int blocks; };
    static std::mutex mu;
    static std::vector<Entry> known;
    size_t smem16 = 0, smem8 = 0;
    const bool fits16 = thermal_cluster_fits(t, kThClusterBlocks, &smem16), fits8 = thermal_cluster_fits(t, kThClusterPortable, &smem8);
    if (!fits8 && !fits16) return 0;
    int blocks = fits8 ? kThClusterPortable : 0;
    if (fits16) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return blocks;
        std::lock_guard<std::mutex> lock(mu);
        bool found = false;
        for (const Entry &e : known) if (e.device == dev && e.smem16 == smem16 && e.fn == (const void *)thermal_cluster_kernel(t, kThClusterBlocks)) { if (e.blocks) blocks = e.blocks; found = true; break; }
        if (!found) {
            int got = 0;
            const void *fn = (const void *)thermal_cluster_kernel(t, kThClusterBlocks);
            if (ensure_dyn_smem(fn, smem16) == cudaSuccess && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
                cudaLaunchConfig_t cfg = {};
                cfg.gridDim = dim3(kThClusterBlocks); cfg.blockDim = dim3(kThThreads); cfg.dynamicSmemBytes = smem16;
                cudaLaunchAttribute at[1];
                at[0].id = cudaLaunchAttributeClusterDimension; at[0].val.clusterDim.x = kThClusterBlocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
                cfg.attrs = at; cfg.numAttrs = 1;
                int n = 0;
                if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) == cudaSuccess && n >= 1) got = kThClusterBlocks;
            }
            (void)cudaGetLastError();                          // a refusal here only means the portable size is used
            known.push_back(Entry{dev, smem16, fn, got});
            if (got) blocks = got;
        }
    }
    *smem_bytes = blocks == kThClusterBlocks ? smem16 : smem8;
    return blocks;
}

// (1 ms step of the 128 x 128 package, 16 substeps, one after the other: 13.8 us; 25 us while every substep tested eight cells a
// thread, divided by the row length and ended in a barrier of the whole cluster)
cudaError_t launch_thermal_step(const ThermalDev &t, DevState *state, int64_t *pending, unsigned long long *bin_row, int64_t dt_ns, int has_ext,
                                float *d_temps_out, int *cur, int generic_only, cudaStream_t st) {
    const float dt_sub_f = (float)((double)dt_ns * 1e-9 / (double)t.n_sub);
    size_t smem = 0;
    const int blocks = generic_only ? 0 : thermal_cluster_blocks(t, &smem);
    if (blocks) {
        const ThermalKernel k = thermal_cluster_kernel(t, blocks);
        { cudaError_t e = ensure_dyn_smem((const void *)k, smem); if (e != cudaSuccess) return e; }
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(blocks); cfg.blockDim = dim3(kThThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
        cudaLaunchAttribute at[2];
        at[0].id = cudaLaunchAttributeClusterDimension; at[0].val.clusterDim.x = blocks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
        at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[1].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at; cfg.numAttrs = 2;
        float *theta = t.theta[*cur];
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k, t, theta, state, pending, bin_row, dt_ns, has_ext, dt_sub_f, d_temps_out);
        if (e != cudaSuccess) return e;
        g_kernel_launches += 1;
        return cudaGetLastError();
    }
    if (bin_row) { const cudaError_t e = launch_take_bin(bin_row, pending, t.n_dies, st); if (e != cudaSuccess) return e; }
    return launch_thermal_generic(t, state, pending, dt_ns, has_ext, d_temps_out, cur, st);
}

}  // namespace hbf
