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
// band of rows of the field (both Jacobi buffers, with a halo row above and below) in shared memory and every cell's
// constants, power and compensation term in registers.  After each substep a block sends its first and last row into its
// neighbours' halo rows (st.async, counted in bytes by a barrier in the neighbour's shared memory): a block waits for its two
// neighbours only, not for the whole cluster.  A neighbour cannot run ahead into a buffer that is still read: it needs this
// block's rows of a substep before it starts the next.  The arithmetic of a cell is the same, in the same order, as in
// k_euler_substep (a missing neighbour has conductance 0, which adds nothing); the power map is formed by every block for its
// own cells and the hotspots are reduced through block 0.
// 16,384 cells are far too few to fill the device: a step lasts as long as its chain of substeps.  A thread holds pairs of cells,
// one above the other, and a buffer holds the two rows of a pair side by side, so that a pair's substep is three 8-byte and two
// 4-byte loads (its own, east, west; north, south) and one store, and the arithmetic is done on both cells at a time (f32x2): a substep
// without its exchange took 354 cycles cell by cell, the exchange with the neighbours takes some 500 more.  One warp polls for the
// neighbours' rows, the block's barrier holds the rest.  Coupled run of 48 windows 936 -> 886 us with these two.
// Whatever no kernel changes is read before the wait for the kernel before.
// ======================================================================================================
constexpr int kThClusterBlocks = 16;                       // blocks of the cluster when the device takes that many (not a portable size), else 8
constexpr int kThClusterPortable = 8;
constexpr int kThThreads = 512;
constexpr int kThPairsPerThread = 4;
constexpr int kThMaxRegions = 1024;
constexpr uint32_t kThTermDies = 1024;                     // dies whose power terms are formed a thread each

__device__ __forceinline__ void th_send(uint32_t addr, float v, uint32_t bar) { smem_send(addr, __float_as_uint(v), bar); }

// two cells at a time (the same roundings as one at a time)
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)));
    return reinterpret_cast<float2 &>(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(reinterpret_cast<unsigned long long &>(a)), "l"(reinterpret_cast<unsigned long long &>(b)), "l"(reinterpret_cast<unsigned long long &>(c)));
    return reinterpret_cast<float2 &>(r);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, make_float2(-1.0f, -1.0f), a); }   // (exact product: one rounding)

// floats as integers of the same order
__device__ __forceinline__ int th_order(float f) { const int k = __float_as_int(f); return k >= 0 ? k : k ^ 0x7fffffff; }
__device__ __forceinline__ float th_unorder(int k) { return __int_as_float(k >= 0 ? k : k ^ 0x7fffffff); }

template <int PPT>
__global__ void __launch_bounds__(kThThreads, 1)
k_thermal_cluster(const __grid_constant__ ThermalDev t, float *theta, DevState *state, int64_t *pending, unsigned long long *bin_row, int64_t dt_ns,
                  int has_ext, float dt_sub, float *temps_out) {
    extern __shared__ __align__(16) unsigned char th_smem_buf[];
    __shared__ double s_region_power[kThMaxRegions];
    __shared__ double s_term[kThTermDies];
    __shared__ uint16_t s_list[kThTermDies];
    __shared__ int s_hot[3][kThClusterBlocks];
    __shared__ int s_part[3][kThThreads / 32];
    __shared__ __align__(8) uint64_t s_bar[2];
    __shared__ __align__(8) uint64_t s_bar_hot;               // (first block) every block's hotspots have come
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), n_blocks = cluster.num_blocks();      // (the cluster's size is chosen at launch)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t H = t.H, W = t.W;
    const uint32_t rows = (H + n_blocks - 1) / n_blocks;
    const uint32_t y0 = min(H, rank * rows), y1 = min(H, y0 + rows), mine = y1 - y0;
    const uint32_t pairs = (mine + 1u) / 2u * W, pitch = ((rows + 1u) / 2u + 2u) * W;   // a buffer: pairs of rows (-2, -1), (0, 1), ... up to the one with the lower halo row
    float2 *buf0 = reinterpret_cast<float2 *>(th_smem_buf);
    const bool has_up = rank > 0u && mine > 0u, has_down = y1 < H && mine > 0u;
    if (tid < 3) {
        const uint32_t bar = smem_addr(tid < 2 ? &s_bar[tid] : &s_bar_hot);
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (tid == 2) asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n_blocks * 12u) : "memory");
    }
    // where row r of a block with `rows` rows lies in its buffer, in bytes
    auto row_at = [&](int32_t r, uint32_t x) { return ((((uint32_t)(r + 2) >> 1) * W + x) * 2u + ((uint32_t)r & 1u)) * 4u; };
    // what no kernel changes: the constants of this thread's cells, the regions' dies
    float kC[PPT][2], gE[PPT][2], gW_[PPT][2], gS[PPT][2], gN[PPT][2], gs[PPT][2], P[PPT][2], cmp[PPT][2], inv[PPT][2];
    uint32_t off[PPT], up[PPT], down[PPT];                    // place in a buffer; the boundary cell's place in the neighbours' halo rows (0: none)
    int32_t region[PPT][2], kind[PPT][2];
    bool live[PPT][2];
#pragma unroll
    for (int c = 0; c < PPT; ++c) {
        const uint32_t li = (uint32_t)c * kThThreads + tid, pr = li / W, x = li - pr * W;
        off[c] = W; up[c] = down[c] = 0u;
        if (li < pairs) {
            const uint32_t b0 = smem_addr(buf0);
            off[c] = (pr + 1u) * W + x;
            if (pr == 0u && has_up) up[c] = smem_remote(b0 + row_at((int32_t)rows, x), rank - 1u);          // (a block above another is full)
            if (pr == (mine - 1u) / 2u && has_down) down[c] = smem_remote(b0 + row_at(-1, x), rank + 1u);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t r = pr * 2u + h, y = y0 + r;
            live[c][h] = li < pairs && r < mine;
            region[c][h] = -1; kind[c][h] = HBF_KIND_NONE;
            kC[c][h] = gE[c][h] = gW_[c][h] = gS[c][h] = gN[c][h] = gs[c][h] = P[c][h] = cmp[c][h] = inv[c][h] = 0.0f;
            if (live[c][h]) {
                const uint64_t i = (uint64_t)y * W + x;
                kC[c][h] = dt_sub / t.C[i];
                if (x + 1 < W) gE[c][h] = t.Gx[i];
                if (x > 0) gW_[c][h] = t.Gx[i - 1];
                if (y + 1 < H) gS[c][h] = t.Gy[i];
                if (y > 0) gN[c][h] = t.Gy[i - W];
                gs[c][h] = -t.Gs[i];
                region[c][h] = t.cell_region[i];
                if (region[c][h] >= 0) { inv[c][h] = t.region_inv_cells[region[c][h]]; kind[c][h] = t.region_kind[region[c][h]]; }
            }
        }
    }
    const bool by_die = t.n_dies <= kThTermDies;
    if (by_die) for (uint32_t d = tid; d < t.n_dies; d += kThThreads) s_list[d] = (uint16_t)t.region_die_list[d];
    int32_t g0 = 0, g1 = 0;                                   // this thread's first region: its dies and its other power (the host writes ext_power between kernels only)
    double p_idle = 0.0, p_ext = 0.0;
    if ((uint32_t)tid < t.n_regions) { g0 = t.region_die_ptr[tid]; g1 = t.region_die_ptr[tid + 1]; p_idle = (double)t.region_idle_w[tid]; if (has_ext) p_ext = (double)t.ext_power[tid]; }
    for (uint32_t i = tid; i < 2u * pitch; i += kThThreads) buf0[i] = make_float2(0.0f, 0.0f);      // (rows outside the grid stay 0)
    const uint32_t bar0 = smem_addr(&s_bar[0]);
    const uint32_t up_bar = has_up ? smem_remote(bar0, rank - 1u) : 0u, down_bar = has_down ? smem_remote(bar0, rank + 1u) : 0u;
    const uint32_t expect = ((has_up ? 1u : 0u) + (has_down ? 1u : 0u)) * W * 4u;
    __syncthreads();
    pdl_wait();                                               // from here on: what the kernels before left
    pdl_trigger();
    // the energies, the cells' own state and the neighbours' boundary rows: all loads go out together
    const int32_t mode0 = state->mode;
    int64_t e0 = 0;
    auto energy = [&](uint32_t d) { return pending[d] + (bin_row ? (int64_t)bin_row[d] : 0); };
    if (by_die && (uint32_t)tid < t.n_dies) e0 = energy(tid);
    float own[PPT][2];
#pragma unroll
    for (int c = 0; c < PPT; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t li = (uint32_t)c * kThThreads + tid, pr = li / W, x = li - pr * W;
            own[c][h] = 0.0f;
            if (live[c][h]) { const uint64_t i = (uint64_t)(y0 + pr * 2u + h) * W + x; own[c][h] = theta[i]; cmp[c][h] = -t.comp[i]; }
        }
    for (uint32_t x = tid; x < W; x += kThThreads) {
        if (has_up) reinterpret_cast<float *>(buf0)[row_at(-1, x) / 4u] = theta[(uint64_t)(y0 - 1u) * W + x];
        if (has_down) reinterpret_cast<float *>(buf0)[row_at((int32_t)mine, x) / 4u] = theta[(uint64_t)y1 * W + x];
    }
    // power of every region over the window (every block forms the same values, summed in the order of the region's dies), then
    // of this block's cells.  The ledger's bin, when there is one, is taken with the pending totals.
    auto term = [&](int64_t e) { return ((double)e * 1e-12) / ((double)dt_ns * 1e-9); };
    if (by_die)
        for (uint32_t d = tid; d < t.n_dies; d += kThThreads) s_term[d] = term(d < (uint32_t)kThThreads ? e0 : energy(d));
#pragma unroll
    for (int c = 0; c < PPT; ++c) {
        if (live[c][1]) buf0[off[c]] = make_float2(own[c][0], own[c][1]);
        else if (live[c][0]) buf0[off[c]].x = own[c][0];      // (the other half of a last odd row's pair is the halo row)
    }
    __syncthreads();
    for (uint32_t g = tid; g < t.n_regions; g += kThThreads) {
        if (g >= (uint32_t)kThThreads) { g0 = t.region_die_ptr[g]; g1 = t.region_die_ptr[g + 1]; p_idle = (double)t.region_idle_w[g]; if (has_ext) p_ext = (double)t.ext_power[g]; }
        double p = 0.0;
        for (int32_t k = g0; k < g1; ++k) p += by_die ? s_term[s_list[k]] : term(energy((uint32_t)t.region_die_list[k]));
        p += p_idle;
        if (has_ext) p += p_ext;
        s_region_power[g] = p;
    }
    cluster.barrier_arrive();                                 // this block's buffers and barriers stand, and it has read the energies
    __syncthreads();
#pragma unroll
    for (int c = 0; c < PPT; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) if (region[c][h] >= 0) P[c][h] = (float)(s_region_power[region[c][h]] * (double)inv[c][h]);
    cluster.barrier_wait();
    if (rank == 0)
        for (uint32_t d = tid; d < t.n_dies; d += kThThreads) { pending[d] = 0; if (bin_row) bin_row[d] = 0ull; }

    bool lost = false;
    for (uint32_t k = 0; k < t.n_sub; ++k) {
        const uint32_t ob = (k + 1u) & 1u;                    // the buffer written
        const float2 *in = buf0 + (k & 1u) * pitch;
        float2 *out = buf0 + ob * pitch;
        const bool more = k + 1u < t.n_sub;
        if (more && expect && tid == 0)
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar0 + ob * 8u), "r"(expect) : "memory");
#pragma unroll
        for (int c = 0; c < PPT; ++c) {
            if (live[c][0]) {
                const uint32_t o = off[c];
                const float2 T = in[o], E = in[o + 1], Wt = in[o - 1];
                const float N = in[o - W].y, S = in[o + W].x;
                auto two = [&](const float (&v)[2]) { return make_float2(v[0], v[1]); };
                float2 flow = fma2(two(gE[c]), sub2(T, E), make_float2(0.0f, 0.0f));
                flow = fma2(two(gW_[c]), sub2(T, Wt), flow);
                flow = fma2(two(gS[c]), sub2(T, make_float2(T.y, S)), flow);
                flow = fma2(two(gN[c]), sub2(T, make_float2(N, T.x)), flow);
                const float2 yv = fma2(two(kC[c]), fma2(two(gs[c]), T, sub2(two(P[c]), flow)), two(cmp[c]));
                const float2 tn = add2(T, yv), left = sub2(yv, sub2(tn, T));
                cmp[c][0] = left.x; cmp[c][1] = left.y;
                const float a = tn.x, last = live[c][1] ? tn.y : tn.x;
                if (live[c][1]) out[o] = tn; else out[o].x = a;
                if (more) {
                    if (up[c]) th_send(up[c] + ob * pitch * 8u, a, up_bar + ob * 8u);
                    if (down[c]) th_send(down[c] + ob * pitch * 8u, last, down_bar + ob * 8u);
                }
            }
        }
        if (more && expect && !lost && warp == 0) {            // (the others are held by the barrier below)
            uint32_t polls = 0;
            while (!smem_poll(bar0 + ob * 8u, (k >> 1) & 1u)) if (++polls > kClusterPolls) { lost = true; break; }
        }
        __syncthreads();
    }
    if (lost) state->poisoned = 1;                            // a neighbour's rows never came: the context is given up
    // results: field and compensation back to global memory, hotspots to block 0
    const float2 *in = buf0 + (t.n_sub & 1u) * pitch;
    float hot[3] = {-INFINITY, -INFINITY, -INFINITY};
#pragma unroll
    for (int c = 0; c < PPT; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (live[c][h]) {
                const uint32_t li = (uint32_t)c * kThThreads + tid, pr = li / W, x = li - pr * W;
                const uint64_t i = (uint64_t)(y0 + pr * 2u + h) * W + x;
                const float th = h ? in[off[c]].y : in[off[c]].x;
                theta[i] = th; t.comp[i] = -cmp[c][h];
                const float T = t.ambient_c + th;
                if (temps_out) temps_out[i] = T;
                if (kind[c][h] == HBF_KIND_HBF) hot[0] = fmaxf(hot[0], T); else if (kind[c][h] == HBF_KIND_HBM) hot[1] = fmaxf(hot[1], T);
                else if (kind[c][h] == HBF_KIND_GPU) hot[2] = fmaxf(hot[2], T);
            }
    // (as ordered integers: one reduction instruction per warp and medium; the other blocks send theirs to the first and are done)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int v = __reduce_max_sync(0xffffffffu, th_order(hot[k]));
        if (lane == 0) s_part[k][warp] = v;
    }
    __syncthreads();
    if (warp < 3) {
        const int v = __reduce_max_sync(0xffffffffu, lane < kThThreads / 32 ? s_part[warp][lane] : th_order(-INFINITY));
        if (lane == 0) th_send(smem_remote(smem_addr(&s_hot[warp][rank]), 0u), __int_as_float(v), smem_remote(smem_addr(&s_bar_hot), 0u));
    }
    if (rank != 0u || warp != 0) return;
    {
        const uint32_t bar = smem_addr(&s_bar_hot);
        uint32_t polls = 0;
        while (!smem_poll(bar, 0u)) if (++polls > kClusterPolls) { state->poisoned = 1; break; }
    }
    float h[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float v = th_unorder(__reduce_max_sync(0xffffffffu, (uint32_t)lane < n_blocks ? s_hot[k][lane] : th_order(-INFINITY)));
        h[k] = v == -INFINITY ? t.ambient_c : v;
    }
    if (lane == 0) {
        t.hot[0] = h[0]; t.hot[1] = h[1]; t.hot[2] = h[2];
        const int mode = next_mode(t, mode0, quantise_mk(h[0]));
        state->mode = mode;
        if (mode == HBF_MODE_NORMAL) state->q_ppm = 1000000;
        else if (mode == HBF_MODE_LIGHT) state->q_ppm = t.q_light_ppm;
    }
}

using ThermalKernel = void (*)(const ThermalDev, float *, DevState *, int64_t *, unsigned long long *, int64_t, int, float, float *);
// the kernel whose threads hold just as many pairs of cells as the grid needs on a cluster of n_blocks
static ThermalKernel thermal_cluster_kernel(const ThermalDev &t, int n_blocks) {
    const uint64_t pairs = (uint64_t)((t.H + n_blocks - 1) / n_blocks + 1) / 2 * t.W;
    return pairs <= 1u * kThThreads ? k_thermal_cluster<1> : pairs <= 2u * kThThreads ? k_thermal_cluster<2> : k_thermal_cluster<kThPairsPerThread>;
}

static bool thermal_cluster_fits(const ThermalDev &t, int n_blocks, size_t *smem_bytes) {
    const uint32_t rows = (t.H + n_blocks - 1) / n_blocks;
    const size_t smem = (size_t)2 * ((rows + 1) / 2 + 2) * t.W * sizeof(float2);
    *smem_bytes = smem;
    return (size_t)((rows + 1) / 2) * t.W <= (size_t)kThThreads * kThPairsPerThread && smem <= 200u * 1024u && t.n_regions <= (uint32_t)kThMaxRegions;
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
                                float *d_temps_out, int *cur, int generic_only, bool *plain_next, cudaStream_t st) {
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
        cfg.attrs = at; cfg.numAttrs = *plain_next ? 1 : 2;   // (see launch_first)
        float *theta = t.theta[*cur];
        const cudaError_t e = cudaLaunchKernelEx(&cfg, k, t, theta, state, pending, bin_row, dt_ns, has_ext, dt_sub_f, d_temps_out);
        if (e != cudaSuccess) return e;
        *plain_next = false;
        g_kernel_launches += 1;
        return cudaGetLastError();
    }
    if (bin_row) { const cudaError_t e = launch_take_bin(bin_row, pending, t.n_dies, st); if (e != cudaSuccess) return e; }
    return launch_thermal_generic(t, state, pending, dt_ns, has_ext, d_temps_out, cur, st);
}

}  // namespace hbf
