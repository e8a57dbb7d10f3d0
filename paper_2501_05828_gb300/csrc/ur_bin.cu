// Binning of arrivals into the analytic channel data (Eq. 14, deposited at the
// exact arrival time).  Arrivals are counting-sorted by row (transmit x element)
// and cut into work items of at most `chunk` arrivals; one CTA accumulates an
// item's pulse taps for its whole row in shared memory (n_s complex samples)
// with shared-memory atomics and flushes the row with coalesced global
// reductions.  Rows of many arrivals accumulate them on interpolation nodes and
// apply the pulse once per row instead of once per arrival.
#include "ur_device.cuh"

#include <algorithm>
#include <cmath>

namespace ur {
namespace {

__device__ __forceinline__ uint32_t lanemask_lt() {
    return (1u << (threadIdx.x & 31)) - 1u;
}

// Arrivals are split into one contiguous range per CTA.  With few rows (one
// transmit has n_el rows) every arrival of a frame lands on one of a handful of
// counters, so the row histogram is kept per CTA in shared memory and added to
// the global counts once per (CTA, row); with more rows than fit, the counts go
// straight to global memory (warp-aggregated).
__device__ __forceinline__ void cta_range(uint64_t n, uint64_t &b, uint64_t &e) {
    const uint64_t per = (n + gridDim.x - 1) / gridDim.x;
    b = min(n, (uint64_t)blockIdx.x * per);
    e = min(n, b + per);
}

__global__ void k_bin_count(const BinP B) {
    extern __shared__ uint32_t hist[];   // [n_rows] when B.priv_rows
    const uint64_t n = min((uint64_t)*B.arr_count, B.arr_cap);
    const bool priv = B.priv_rows;
    if (priv) {
        for (int r = threadIdx.x; r < B.n_rows; r += blockDim.x) hist[r] = 0u;
        __syncthreads();
    }
    uint64_t b, e;
    cta_range(n, b, e);
    for (uint64_t idx = b + threadIdx.x; idx < e; idx += blockDim.x) {
        const uint32_t row = B.arr[idx].x;
        const unsigned peers = __match_any_sync(__activemask(), row);
        if ((threadIdx.x & 31) == __ffs(peers) - 1)
            atomicAdd(priv ? &hist[row] : &B.row_count[row], (uint32_t)__popc(peers));
    }
    if (priv) {
        __syncthreads();
        for (int r = threadIdx.x; r < B.n_rows; r += blockDim.x)
            if (hist[r]) atomicAdd(&B.row_count[r], hist[r]);
    }
}

// Single-CTA scan: row offsets (exclusive scan of counts) and the work-item list.
__global__ void __launch_bounds__(1024) k_bin_plan(const BinP B) {
    __shared__ uint32_t s_warp[3][32];
    __shared__ uint32_t s_carry[3];
    if (threadIdx.x < 3) s_carry[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // Work-item size: enough items for several waves of the deposit grid, within [chunk_min, chunk].
    const uint64_t total = min((uint64_t)*B.arr_count, B.arr_cap);
    const uint32_t chunk = (uint32_t)min((uint64_t)B.chunk,
                                         max((uint64_t)B.chunk_min, (total + B.target_items - 1) / B.target_items));
    for (int base = 0; base < B.n_rows; base += 1024) {
        const int row = base + (int)threadIdx.x;
        const uint32_t cnt = row < B.n_rows ? B.row_count[row] : 0u;
        const bool nodes = B.n_nodes > 0 && cnt >= B.node_min;
        const uint32_t per = nodes ? B.node_chunk : chunk;
        const uint32_t nit = (cnt + per - 1) / per;
        // inclusive warp scans of the arrivals, the tap-by-tap items and the node items
        uint32_t v[3] = {cnt, nodes ? 0u : nit, nodes ? nit : 0u};
#pragma unroll
        for (int off = 1; off < 32; off <<= 1)
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, v[q], off);
                if (lane >= off) v[q] += y;
            }
        if (lane == 31)
            for (int q = 0; q < 3; ++q) s_warp[q][wid] = v[q];
        __syncthreads();
        if (wid < 3) {
            uint32_t w = s_warp[wid][lane];
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, w, off);
                if (lane >= off) w += y;
            }
            s_warp[wid][lane] = w;
        }
        __syncthreads();
        uint32_t pre[3];   // exclusive over the rows so far
        for (int q = 0; q < 3; ++q) pre[q] = (wid ? s_warp[q][wid - 1] : 0u) + v[q] + s_carry[q];
        pre[0] -= cnt;
        pre[nodes ? 2 : 1] -= nit;
        if (row < B.n_rows) {
            B.row_off[row] = pre[0];
            for (uint32_t q = 0; q < nit; ++q) {
                const uint32_t b0 = pre[0] + q * per, b1 = min(pre[0] + cnt, b0 + per);
                const uint32_t it = nodes ? B.max_items - 1u - (pre[2] + q) : pre[1] + q;
                if (it < B.max_items) B.items[it] = make_uint4((uint32_t)row, b0, b1, 0u);
            }
        }
        __syncthreads();
        if (threadIdx.x < 3) s_carry[threadIdx.x] += s_warp[threadIdx.x][31];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        B.row_off[B.n_rows] = s_carry[0];
        B.n_items[0] = s_carry[1];
        B.n_items[1] = s_carry[2];
    }
}

// Counting-sort scatter.  With the shared histogram each CTA counts its range
// again, reserves one block of positions per row with a single global atomic,
// then hands out positions inside the block with shared-memory atomics.
__global__ void k_bin_scatter(const BinP B) {
    extern __shared__ uint32_t hist[];   // [n_rows]: local counts, then next free position
    const uint64_t n = min((uint64_t)*B.arr_count, B.arr_cap);
    const unsigned lt = lanemask_lt();
    uint64_t b, e;
    cta_range(n, b, e);
    if (!B.priv_rows) {
        for (uint64_t idx = b + threadIdx.x; idx < e; idx += blockDim.x) {
            const uint4 a = B.arr[idx];
            const uint32_t row = a.x;
            const unsigned peers = __match_any_sync(__activemask(), row);
            const int leader = __ffs(peers) - 1;
            uint32_t base = 0;
            if ((int)(threadIdx.x & 31) == leader) base = atomicAdd(&B.row_fill[row], (uint32_t)__popc(peers));
            base = __shfl_sync(peers, base, leader);
            const uint32_t pos = B.row_off[row] + base + (uint32_t)__popc(peers & lt);
            B.sorted[pos] = make_float4(__uint_as_float(a.y), __uint_as_float(a.z), __uint_as_float(a.w), 0.f);
        }
        return;
    }
    for (int r = threadIdx.x; r < B.n_rows; r += blockDim.x) hist[r] = 0u;
    __syncthreads();
    for (uint64_t idx = b + threadIdx.x; idx < e; idx += blockDim.x) {
        const uint32_t row = B.arr[idx].x;
        const unsigned peers = __match_any_sync(__activemask(), row);
        if ((threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&hist[row], (uint32_t)__popc(peers));
    }
    __syncthreads();
    for (int r = threadIdx.x; r < B.n_rows; r += blockDim.x) {
        const uint32_t c = hist[r];
        if (c) hist[r] = B.row_off[r] + atomicAdd(&B.row_fill[r], c);
    }
    __syncthreads();
    for (uint64_t idx = b + threadIdx.x; idx < e; idx += blockDim.x) {
        const uint4 a = B.arr[idx];
        const uint32_t row = a.x;
        const unsigned peers = __match_any_sync(__activemask(), row);
        const int leader = __ffs(peers) - 1;
        uint32_t base = 0;
        if ((int)(threadIdx.x & 31) == leader) base = atomicAdd(&hist[row], (uint32_t)__popc(peers));
        base = __shfl_sync(peers, base, leader);
        B.sorted[base + (uint32_t)__popc(peers & lt)] =
            make_float4(__uint_as_float(a.y), __uint_as_float(a.z), __uint_as_float(a.w), 0.f);
    }
}

// ceil / floor of a float-float value hi + lo
__device__ __forceinline__ int ff_ceil(float hi, float lo) {
    const float c = ceilf(hi);
    return (int)c + ((c == hi && lo > 0.f) ? 1 : 0);
}
__device__ __forceinline__ int ff_floor(float hi, float lo) {
    const float f = floorf(hi);
    return (int)f - ((f == hi && lo < 0.f) ? 1 : 0);
}

// One CTA per work item (a chunk of one row's arrivals): the row's complex
// samples accumulate in shared memory and are flushed with one global reduction
// each.  A warp loads 32 arrivals at once (one per lane, coalesced); each lane
// evaluates the carrier phase of its own arrival at that arrival's first tap,
// and the warp then deposits the 32 arrivals one after the other, lanes taking
// consecutive taps.  A lane's phase is the broadcast first-tap phase rotated by
// its lane offset, advanced by the exact rotation of 32 samples per step; the
// Gaussian envelope is evaluated per tap.
__global__ void __launch_bounds__(512) k_bin_deposit(const BinP B) {
    extern __shared__ float acc[];  // [2][n_s]: real, quadrature
    const uint32_t n_items = *B.n_items;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    float rl_s, rl_c;   // carrier rotation over `lane` samples
    sincospif((float)lane * B.phase_per_sample, &rl_s, &rl_c);
    for (uint32_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const uint4 item = B.items[it];
        for (int n = threadIdx.x; n < 2 * B.n_s; n += blockDim.x) acc[n] = 0.f;
        __syncthreads();
        for (uint32_t q0 = item.y + 32u * (uint32_t)wid; q0 < item.z; q0 += 32u * (uint32_t)nw) {
            const uint32_t q = q0 + (uint32_t)lane;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            int n0 = 0, n1 = -1;
            float bs = 0.f, bc = 1.f;
            if (q < item.z) {
                a = B.sorted[q];
                n0 = max(ff_ceil(a.x - B.K, a.y), 0);
                n1 = min(ff_floor(a.x + B.K, a.y), B.n_s - 1);
                sincospif((((float)n0 - a.x) - a.y) * B.phase_per_sample, &bs, &bc);
            }
            const int cnt = (int)min(32u, item.z - q0);
            for (int j = 0; j < cnt; ++j) {
                const int jn0 = __shfl_sync(0xffffffffu, n0, j);
                const int jn1 = __shfl_sync(0xffffffffu, n1, j);
                const float t_hi = __shfl_sync(0xffffffffu, a.x, j);
                const float t_lo = __shfl_sync(0xffffffffu, a.y, j);
                const float amp = __shfl_sync(0xffffffffu, a.z, j);
                const float js = __shfl_sync(0xffffffffu, bs, j);
                const float jc = __shfl_sync(0xffffffffu, bc, j);
                int n = jn0 + lane;
                if (n > jn1) continue;
                float sn = fmaf(js, rl_c, jc * rl_s);
                float cs = fmaf(jc, rl_c, -js * rl_s);
                float tau = ((float)n - t_hi) - t_lo;   // (n - t_hi) is exact
                for (;;) {
                    const float g = amp * exp2f(-tau * tau * B.inv_2s2_log2e);
                    atomicAdd(&acc[n], g * sn);
                    atomicAdd(&acc[B.n_s + n], -g * cs);
                    n += 32;
                    if (n > jn1) break;
                    tau += 32.f;
                    const float s2 = fmaf(sn, B.rot32_c, cs * B.rot32_s);
                    cs = fmaf(cs, B.rot32_c, -sn * B.rot32_s);
                    sn = s2;
                }
            }
        }
        __syncthreads();
        float *rf = B.rf + (size_t)item.x * B.n_s;
        float *qd = B.quad + (size_t)item.x * B.n_s;
        for (int n = threadIdx.x; n < B.n_s; n += blockDim.x) {
            const float vr = acc[n], vq = acc[B.n_s + n];
            if (vr != 0.f) atomicAdd(&rf[n], vr);
            if (vq != 0.f) atomicAdd(&qd[n], vq);
        }
        __syncthreads();
    }
}

// Rows of many arrivals: the pulse as a convolution.  With w(u) = g(u) e^(i omega u), g the Gaussian,
//   rf + j quad of an arrival (t, amp) at sample n:  sin / -cos of  omega (n - t), times amp g(n - t),
// so the row is e^(i omega n) times the sum of amp e^(-i omega t) g(n - t).  g is smooth on the scale of a
// few samples: within a cell of 4 samples around tc, g(n - t) is its interpolation from R Chebyshev
// nodes tc + x_k (R chosen so that the error stays below FP32's rounding of the peak, and below that
// of the tap itself at the pulse's weak ends, see kNodeRel), and an arrival
// adds amp e^(-i omega t) L_k(t - tc) to its cell's R complex node sums: 2 R shared atomics instead of 2 per
// tap (14 instead of 202).  Each sample then sums g over the nodes of the cells around it once.  Only
// taps inside the pulse's cut |n - t| <= K for every t of a cell go through the nodes; the up to 5 others
// of an arrival are deposited one by one, so the cut stays where it is.
// The Gaussian's values come from the kernel's constants.  Bound by issue on the layered frame (82 % of
// the slots of busy schedulers, 63 warp instructions per arrival; over the launch 47 %, as 640 work
// items on 456 CTAs end in a part wave; shared-memory latency next), and by the chains of
// shared-memory atomics where arrivals of other times crowd into the same cells: there tap by tap
// is faster, but the host does not know (one focused transmit of 2e6 rays 70 us tap by tap, 200 this
// way).  Layered frame (2.27M arrivals, 128 rows) 412 -> 240 us, 4096 rows of 1.8k arrivals 1239 -> 690 us;
// error of the layered frame's channel data against 64 bits 1.4e-6 -> 3.0e-7.  Tap by tap stays the
// better one below about 1000 arrivals per row (680 per row: 63 us against 89).
constexpr int kNodeThreads = 512;

// Samples before (and after) the row that its cells cover, a multiple of the cell; cells of a row.
__host__ __device__ __forceinline__ int node_margin(float K) { return ((int)ceilf(K) / kBinCell + 2) * kBinCell; }
__host__ __device__ __forceinline__ int node_cells(float K, int n_s) {
    return (n_s + 2 * node_margin(K) + kBinCell - 1) / kBinCell;
}

template <int R>
__global__ void __launch_bounds__(kNodeThreads) k_bin_nodes(const __grid_constant__ BinP B, const __grid_constant__ BinNodeG G) {
    extern __shared__ float node[];   // [R][2][cells]: node sums, real and imaginary; then [2][n_s]: edge taps
    const int off = node_margin(B.K);                                 // samples before the row that cells cover
    const int cells = node_cells(B.K, B.n_s);
    float *acc = node + 2 * R * cells;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int d_lo = G.d_lo, d_hi = G.d_hi;
    const int my_k = (lane & 15) >> 1;   // this lane's node
    const float my_w = my_k < R ? B.node_w[my_k] : 0.f;
    const uint32_t n_items = B.n_items[1];
    for (uint32_t it = blockIdx.x; it < n_items; it += gridDim.x) {
        const uint4 item = B.items[B.max_items - 1u - it];
        for (int n = threadIdx.x; n < 2 * R * cells; n += kNodeThreads) node[n] = 0.f;
        for (int n = threadIdx.x; n < 2 * B.n_s; n += kNodeThreads) acc[n] = 0.f;
        __syncthreads();
        for (uint32_t q0 = item.y + 32u * (uint32_t)wid; q0 < item.z; q0 += (uint32_t)kNodeThreads) {
            const bool valid = q0 + (uint32_t)lane < item.z;
            float4 a = valid ? B.sorted[q0 + (uint32_t)lane] : make_float4(0.f, 0.f, 0.f, 0.f);
            // Echoes of planes under a plane wave arrive at one time: equal times of a warp are added
            // up first and deposited once (their node sums would be contended, and grow one by one).
            unsigned same = __match_any_sync(0xffffffffu, __float_as_uint(a.x)) &
                            __match_any_sync(0xffffffffu, __float_as_uint(a.y)) & __ballot_sync(0xffffffffu, valid);
            const bool first = valid && lane == __ffs(same) - 1;
            float amp = 0.f;
            for (int n = (int)__reduce_max_sync(0xffffffffu, (unsigned)__popc(same)); n > 0; --n) {
                const float v = __shfl_sync(0xffffffffu, a.z, same ? __ffs(same) - 1 : 0);
                if (same) amp += v;
                same &= same - 1u;
            }
            a.z = amp;
            const int n0 = max(ff_ceil(a.x - B.K, a.y), 0), n1 = min(ff_floor(a.x + B.K, a.y), B.n_s - 1);
            const int c = (ff_floor(a.x, a.y) + off) >> 2;
            const int tc = kBinCell * c + kBinCell / 2 - off;
            const float dl = (a.x - (float)tc) + a.y;   // in [-2, 2)
            // carrier phase at t in half-cycles, its whole periods taken off before the tail is added
            const float p = a.x * B.phase_per_sample;
            const float pl = fmaf(a.x, B.phase_per_sample, -p) + a.y * B.phase_per_sample;
            float sn, cs;
            sincospif((p - 2.f * rintf(0.5f * p)) + pl, &sn, &cs);
            const float re = a.z * cs, im = -a.z * sn;
            // a cell outside the row's has no taps in it (no arrival is that early or late)
            const bool use = first && n0 <= n1 && c >= 0 && c < cells;
            // amplitudes that are not finite (or nearly overflow) would spoil every sample of their nodes:
            // all their taps are left to the loop below
            const bool smooth = use && fabsf(a.z) < 1e37f && dl == dl;
            // The warp adds its arrivals two at a time, half a warp per arrival and a lane per (node,
            // component): echoes of one scatterer arrive within a cell, and a lane per arrival would
            // leave the lanes of a warp waiting for one another's sums.
            unsigned todo = __ballot_sync(0xffffffffu, smooth);
            while (todo) {
                const int j0 = __ffs(todo) - 1;
                todo &= todo - 1u;
                const int j1 = todo ? __ffs(todo) - 1 : -1;
                todo &= todo - 1u;
                const int src = lane < 16 ? j0 : j1;
                const float jd = __shfl_sync(0xffffffffu, dl, src & 31), jr = __shfl_sync(0xffffffffu, re, src & 31);
                const float ji = __shfl_sync(0xffffffffu, im, src & 31);
                const int jc = __shfl_sync(0xffffffffu, c, src & 31);
                if (src >= 0 && my_k < R) {
                    float w = my_w;
#pragma unroll
                    for (int m = 0; m < R; ++m) w *= m == my_k ? 1.f : jd - B.node[m];
                    atomicAdd(&node[(2 * my_k + (lane & 1)) * cells + jc], w * ((lane & 1) ? ji : jr));
                }
            }
            if (!use) continue;
            // taps the nodes leave out
            const int l1 = smooth ? min(n1, tc + d_lo - 1) : n1, r0 = max(n0, tc + d_hi + 1);
            for (int n = n0 <= l1 ? n0 : r0; n <= n1; n = n == l1 ? max(r0, l1 + 1) : n + 1) {
                const float tau = ((float)n - a.x) - a.y;
                const float g = a.z * exp2f(-tau * tau * B.inv_2s2_log2e);
                sincospif(tau * B.phase_per_sample, &sn, &cs);
                atomicAdd(&acc[n], g * sn);
                atomicAdd(&acc[B.n_s + n], -g * cs);
            }
        }
        __syncthreads();
        float *rf = B.rf + (size_t)item.x * B.n_s;
        float *qd = B.quad + (size_t)item.x * B.n_s;
        for (int a = threadIdx.x; kBinCell * a < B.n_s; a += kNodeThreads) {
            float re[kBinCell] = {0.f, 0.f, 0.f, 0.f}, im[kBinCell] = {0.f, 0.f, 0.f, 0.f};
            for (int j = 0; j < G.n_j; ++j) {
                // sample 4 a + b lies d = 4 (a - c) + b - 2 from the centre of cell c (counted from sample 0)
                const float *m = node + (a - (j + G.j_lo) + off / kBinCell);   // cells are stored from -off
                const float4 *g = G.g + j * R;
#pragma unroll
                for (int k = 0; k < R; ++k) {
                    const float2 v = make_float2(m[2 * k * cells], m[(2 * k + 1) * cells]);
                    const float4 w = g[k];
                    re[0] = fmaf(w.x, v.x, re[0]);
                    im[0] = fmaf(w.x, v.y, im[0]);
                    re[1] = fmaf(w.y, v.x, re[1]);
                    im[1] = fmaf(w.y, v.y, im[1]);
                    re[2] = fmaf(w.z, v.x, re[2]);
                    im[2] = fmaf(w.z, v.y, im[2]);
                    re[3] = fmaf(w.w, v.x, re[3]);
                    im[3] = fmaf(w.w, v.y, im[3]);
                }
            }
#pragma unroll
            for (int b = 0; b < kBinCell; ++b) {
                const int n = kBinCell * a + b;
                if (n >= B.n_s) break;
                const float p = (float)n * B.phase_per_sample;
                const float pl = fmaf((float)n, B.phase_per_sample, -p);
                float sn, cs;
                sincospif((p - 2.f * rintf(0.5f * p)) + pl, &sn, &cs);
                const float vr = fmaf(sn, re[b], fmaf(cs, im[b], acc[n]));
                const float vq = fmaf(sn, im[b], fmaf(-cs, re[b], acc[B.n_s + n]));
                if (vr != 0.f) atomicAdd(&rf[n], vr);
                if (vq != 0.f) atomicAdd(&qd[n], vq);
            }
        }
        __syncthreads();
    }
}

// Interpolation error of a tap relative to its envelope.  FP32's own, tap by tap (rounded arguments of
// the Gaussian and of the carrier), is 1e-6 RMS and 2.6e-6 to 6e-6 at most for pulses of 3 to 9 cycles at
// 25 to 50 MHz; the bound takes 50 MHz x 5 cycles from 6 nodes (7.9e-6) to 7 (2.8e-7).
constexpr double kNodeRel = 2.5e-6;
constexpr double kNodeWeak = 3.7e-6;   // taps weaker than this (5 sigma) count as this strong

constexpr int kNodeSmem = 226 << 10;   // most shared memory of a CTA

int node_smem(const BinP &B) {
    return (2 * B.n_nodes * node_cells(B.K, B.n_s) + 2 * B.n_s) * (int)sizeof(float);
}

template <int R>
void launch_nodes(const BinP &B, const BinNodeG &G, uint64_t most_items, int sms, cudaStream_t s) {
    const int smem = node_smem(B);
    // one value for every caller: the attribute belongs to the process, and a context of shorter rows in
    // another thread must not lower it between this call's attribute and its launch
    cudaFuncSetAttribute(k_bin_nodes<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, kNodeSmem);
    uint64_t grid = (uint64_t)sms * std::max(1, std::min(4, kNodeSmem / (smem + 1024)));
    if (most_items) grid = std::min(grid, most_items);
    k_bin_nodes<R><<<(int)grid, kNodeThreads, smem, s>>>(B, G);
}

__global__ void k_unpack_debug(const uint4 *arr, const uint2 *dbg, const unsigned long long *count, uint64_t cap_in,
                               const DebugOut D) {
    const uint64_t n = min(min((uint64_t)*count, cap_in), D.cap);
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint4 a = arr[i];
        const uint2 b = dbg[i];
        D.row[i] = a.x;
        D.t_hi[i] = __uint_as_float(a.y);
        D.t_lo[i] = __uint_as_float(a.z);
        D.amp[i] = __uint_as_float(a.w);
        D.ray[i] = b.x;
        D.event[i] = b.y;
    }
}

}  // namespace

void launch_unpack_debug(const uint4 *arr, const uint2 *dbg, const unsigned long long *count, uint64_t cap_in,
                         const DebugOut &D, cudaStream_t s) {
    k_unpack_debug<<<1024, 256, 0, s>>>(arr, dbg, count, cap_in, D);
}

int bin_sort_smem(int n_rows) {
    return n_rows <= kBinPrivRows ? n_rows * (int)sizeof(uint32_t) : 0;
}

void launch_bin_sort(const BinP &B, int sms, cudaStream_t s) {
    const int smem = B.priv_rows ? bin_sort_smem(B.n_rows) : 0;
    // CTAs per SM: up to 4 x 512 threads, fewer when the histogram is large
    const int per_sm = smem ? std::max(1, std::min(4, (200 << 10) / (smem + 1024))) : 4;
    const int grid = sms * per_sm;
    if (smem > 48 * 1024) {
        cudaFuncSetAttribute(k_bin_count, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        cudaFuncSetAttribute(k_bin_scatter, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    }
    k_bin_count<<<grid, 512, smem, s>>>(B);
    k_bin_plan<<<1, 1024, 0, s>>>(B);
    k_bin_scatter<<<grid, 512, smem, s>>>(B);
}

void plan_bin_nodes(BinP &B, BinNodeG &G, double s) {
    B.n_nodes = 0;
    if (!(B.K >= 8.f)) return;   // short pulses: hardly a tap that every arrival of a cell has
    const int half = (int)std::floor(B.K);
    G.d_lo = kBinCell / 2 - half;
    G.d_hi = half - kBinCell / 2;
    G.j_lo = (G.d_lo + kBinCell / 2 - (kBinCell - 1)) >> 2;
    G.n_j = ((G.d_hi + kBinCell / 2) >> 2) - G.j_lo + 1;
    if (G.n_j > kBinDist) return;
    // The Gaussian at the taps -half .. half around x, outward from its peak by its ratios: two
    // multiplications a tap (relative error below 1e-11).  A plan of fresh exponentials took 0.25 ms of
    // a frame's host time.
    constexpr int most = 4 * kBinDist;   // taps (half is below 2 kBinDist, see n_j above)
    const int taps = 2 * half + 1;
    const double step = std::exp(-1.0 / (s * s));
    const auto gaussian = [&](double x, double *g) {
        const double u = std::lround(x) - x, peak = std::exp(-u * u / (2.0 * s * s));
        double *mid = g + half + std::lround(x);
        double v = peak, ratio = std::exp(-(2.0 * u + 1.0) / (2.0 * s * s));
        for (double *p = mid; p < g + taps; ++p, v *= ratio, ratio *= step) *p = v;
        v = peak, ratio = std::exp((2.0 * u - 1.0) / (2.0 * s * s));
        for (double *p = mid; p >= g; --p, v *= ratio, ratio *= step) *p = v;
    };
    constexpr int kOffsets = 17;   // arrival times over half a cell (the nodes are symmetric)
    double at_t[kOffsets][most], at_x[kBinNodes][most];
    for (int q = 0; q < kOffsets; ++q) gaussian(kBinCell / 2 * q / (kOffsets - 1.0), at_t[q]);
    for (int R = 5; R <= kBinNodes && !B.n_nodes; ++R) {
        double x[kBinNodes], w[kBinNodes];
        for (int k = 0; k < R; ++k) x[k] = kBinCell / 2 * std::cos((2 * k + 1) * 3.14159265358979323846 / (2 * R));
        for (int k = 0; k < R; ++k) {
            w[k] = 1.0;
            for (int m = 0; m < R; ++m)
                if (m != k) w[k] /= x[k] - x[m];
            gaussian(x[k], at_x[k]);
        }
        // the interpolation error of the unit-peak Gaussian over a cell and the pulse, and relative to the tap
        // itself where the nodes serve it
        bool good = true;
        for (int q = 0; q < kOffsets && good; ++q) {
            const double t = kBinCell / 2 * q / (kOffsets - 1.0);
            double err[most];
            for (int d = 0; d < taps; ++d) err[d] = -at_t[q][d];
            for (int k = 0; k < R; ++k) {
                double L = w[k];
                for (int m = 0; m < R; ++m)
                    if (m != k) L *= t - x[m];
                for (int d = 0; d < taps; ++d) err[d] += L * at_x[k][d];
            }
            for (int d = 0; d < taps; ++d) {
                const bool served = d >= G.d_lo + half && d <= G.d_hi + half;
                good = good && std::fabs(err[d]) <= 2e-8 && (!served || std::fabs(err[d]) <= kNodeRel * std::max(at_t[q][d], kNodeWeak));
            }
        }
        if (!good) continue;
        B.n_nodes = R;
        for (int k = 0; k < R; ++k) {
            B.node[k] = (float)x[k];
            B.node_w[k] = (float)w[k];
        }
        if (node_smem(B) > kNodeSmem) {
            B.n_nodes = 0;
            return;
        }
        for (int q = 0; q < G.n_j * R; ++q) {
            float g[kBinCell];
            for (int b = 0; b < kBinCell; ++b) {
                const int d = kBinCell * (q / R + G.j_lo) + b - kBinCell / 2;
                const double u = d - x[q % R];
                g[b] = d >= G.d_lo && d <= G.d_hi ? (float)std::exp(-u * u / (2.0 * s * s)) : 0.f;
            }
            G.g[q] = make_float4(g[0], g[1], g[2], g[3]);
        }
    }
}

int launch_bin_deposit(const BinP &B, const BinNodeG &G, uint64_t most_items, int sms, cudaStream_t s) {
    const int smem = 2 * B.n_s * (int)sizeof(float);
    cudaFuncSetAttribute(k_bin_deposit, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kMaxNs * (int)sizeof(float));
    k_bin_deposit<<<sms * 4, 512, smem, s>>>(B);
    if (!B.n_nodes) return 1;
    switch (B.n_nodes) {
        case 5: launch_nodes<5>(B, G, most_items, sms, s); break;
        case 6: launch_nodes<6>(B, G, most_items, sms, s); break;
        case 7: launch_nodes<7>(B, G, most_items, sms, s); break;
        default: launch_nodes<8>(B, G, most_items, sms, s);
    }
    return 2;
}

}  // namespace ur
