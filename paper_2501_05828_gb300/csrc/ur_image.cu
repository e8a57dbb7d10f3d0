// Image formation: delay-and-sum of the analytic channel data with
// coherent compounding over transmits, envelope, global maximum and log
// compression.  Transmit delays are evaluated in float-float, receive delays by a
// square root corrected from its exact residual; both are held in 32.32 fixed point,
// so that only the interpolation weight is rounded to FP32 (2^-25 samples).
#include "ur_device.cuh"

namespace ur {
namespace {

__device__ __forceinline__ ff ff_neg(ff a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ int ff_floor_i(ff a) {
    const float f = floorf(a.hi);
    return (int)f - ((f == a.hi && a.lo < 0.f) ? 1 : 0);
}

// Delays in samples as 32.32 fixed point: a sum is two integer adds, the sample index is the
// high word and the interpolation weight the low one.  hi + lo is a float-float (lo the tail, below
// one half): hi's distance to the nearest integer is exact, and it and the tail are rounded to 2^-31
// each, so a delay is off by 2^-32 and only the weight by FP32's 2^-25 (with the fraction rounded to 24
// bits as well, in units of 2^-30, the weight was off by up to 6e-8).  Valid for |hi| < kFixedMax.
constexpr float kFixedMax = 2097152.f;   // 2^21 samples

__device__ __forceinline__ long long to_fixed(float hi, float lo) {
    const float b = __fadd_rn(hi, 12582912.f);   // 1.5 x 2^23: the mantissa holds round(hi)
    const float fr = __fsub_rn(hi, __fsub_rn(b, 12582912.f));   // exact
    const int a = __float2int_rn(__fmul_rn(fr, 0x1p31f)) + __float2int_rn(__fmul_rn(lo, 0x1p31f));
    const int i = __float_as_int(b) - 0x4B400000 + (a >> 31);
    return (long long)(((unsigned long long)(unsigned)i << 32) | ((unsigned)a << 1));
}

__device__ __forceinline__ float rsqrt_approx(float a) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(a));
    return y;
}

// Transmit delay to (x, z) in samples: plane wave; distance from a virtual source; through a focus.
__device__ __forceinline__ ff transmit_delay(const ImageP &I, int k, float x, float z) {
    const int kind = I.tx_kind ? I.tx_kind[k] : UR_TX_PLANE;
    if (kind == UR_TX_PLANE) {
        const ff T = ff_add(ff_mul_f(x, I.tx_sin[k]), ff_mul_f(z, I.tx_cos[k]));
        return ff_mul(ff_add(T, ff_neg(I.tx_m[k])), I.q);
    }
    const ff ddx = ff_add_f(ff_neg(I.tx_sin[k]), x), ddz = ff_add_f(ff_neg(I.tx_cos[k]), z);
    const ff r = ff_sqrt(ff_add(ff_mul(ddx, ddx), ff_mul(ddz, ddz)));
    if (kind == UR_TX_DIVERGING) return ff_mul(ff_add(r, ff_neg(I.tx_m[k])), I.q);
    return ff_mul(ff_add(I.tx_m[k], (z >= I.tx_cos[k].hi) ? r : ff_neg(r)), I.q);
}

// Element centre: from the table of a convex array, else on z = 0 at x_first + e pitch.
template <bool CONVEX>
__device__ __forceinline__ void element_centre(const ImageP &I, int e, ff &x, ff &z) {
    if (CONVEX) {
        x = I.elem_xz[2 * e];
        z = I.elem_xz[2 * e + 1];
    } else {
        const float pe = (float)e * I.pitch;
        const ff ep = {pe, __fmaf_rn((float)e, I.pitch, -pe)};
        x = ff_add(I.x_first, ep);
        z = {0.f, 0.f};
    }
}

// Elements [e0, e1) of transmit k (item `item`) for a pixel whose delays leave the fixed-point
// range (non-finite coordinates, or kilometres away): float-float throughout, one term at a time.
template <bool CONVEX>
__device__ __noinline__ float2 das_wide(const ImageP &I, int item, int k, int e0, int e1, float x, float z) {
    const ff T = transmit_delay(I, k, x, z);
    const float top = (float)(I.n_s - 1);
    float sr = 0.f, si = 0.f;
    for (int e = e0; e < e1; ++e) {
        ff ex, ez;
        element_centre<CONVEX>(I, e, ex, ez);
        const ff dx = ff_add_f(ff_neg(ex), x);
        ff r2;
        if (CONVEX) {
            const ff dz = ff_add_f(ff_neg(ez), z);
            r2 = ff_add(ff_mul(dz, dz), ff_mul(dx, dx));
        } else {
            r2 = ff_add(ff_sqr_f(z), ff_mul(dx, dx));
        }
        const ff tau = ff_add(T, ff_mul(ff_sqrt(r2), I.q));
        if (tau.hi < 0.f || (tau.hi == 0.f && tau.lo < 0.f) || ff_gt(tau, top)) continue;
        const int i0 = ff_floor_i(tau);
        const float f = ((tau.hi - (float)i0) + tau.lo);
        const int i1 = min(i0 + 1, I.n_s - 1);
        const size_t row = ((size_t)item * I.n_el + e) * I.n_s;
        sr += I.rf[row + i0] * (1.f - f) + I.rf[row + i1] * f;
        si += I.quad[row + i0] * (1.f - f) + I.quad[row + i1] * f;
    }
    return make_float2(sr, si);
}

// Warps below which small images share a pixel's elements: two residencies of the chip at 32 warps
// per SM; 5120 and 20480 gave 31 transmits 1042 and 891 us against 933 us at this value (4 CTAs per
// SM), single transmits 51 and 55 against 52 us.
constexpr long long kDasWarps = 10240;

// Pixels along x of a warp: 16 in images of this width, else 8 (fewer in narrower images).  A warp of
// 32 wastes up to half its lanes on the edge (33 columns of 64 elements x 8192 samples over 0.2 m, 7
// transmits: slower than lanes along depth), and columns far apart share no cache lines along x.
// Measured (us) at 32, 16, 8, 4: 31 transmits of 128 elements, 512 x 256 710, 705, 709, 730; 512 x 96
// 326, 328, 389, 561; 383 x 301 645, 643, 643, 647; 128 x 1600 1179, 1068, 1025, 1019; 161 x 300 383, 358,
// 338, 345; 97 x 700 621, 500, 459, 442; 33 x 2000 1065, 683, 524, 456; one transmit alike within 5 %.
constexpr int kWideImage = 192;

constexpr long long kNoTransmit = -(1ll << 62);   // with any receive delay: outside every recording

// Samples a[0], b[0] if tau <= top, a[1], b[1] if tau's sample is not the last, else 0: predicated
// loads in straight-line code, so that the loads of all transmits of a chunk are in flight at once
// (with a branch around each term's loads the 31-transmit image took 1190 us, one term at a time).
__device__ __forceinline__ void gather(const float *a, const float *b, unsigned long long tau, unsigned long long top,
                                       float &a0, float &a1, float &b0, float &b1) {
    asm("{\n\t"
        ".reg .pred p, q;\n\t"
        "setp.le.u64 p, %6, %7;\n\t"
        "setp.lt.u64 q, %6, %7;\n\t"
        "mov.f32 %0, 0f00000000;\n\t"
        "mov.f32 %1, 0f00000000;\n\t"
        "mov.f32 %2, 0f00000000;\n\t"
        "mov.f32 %3, 0f00000000;\n\t"
        "@p ld.global.nc.f32 %0, [%4];\n\t"
        "@q ld.global.nc.f32 %1, [%4+4];\n\t"
        "@p ld.global.nc.f32 %2, [%5];\n\t"
        "@q ld.global.nc.f32 %3, [%5+4];\n\t"
        "}"
        : "=&f"(a0), "=&f"(a1), "=&f"(b0), "=&f"(b1)
        : "l"(a), "l"(b), "l"(tau), "l"(top));
}

// How the image is cut up: a warp holds 1 << wx_log2 pixels along x and 32 >> wx_log2 along z,
// and `split` warps of a CTA share a group of pixels, each summing its part of the elements.
struct DasTile {
    int wx_log2, split, tiles_x;
};

// One thread per pixel (and part of the elements), KT transmits at a time.
//
// Bound by issue slots (67 % for 31 transmits, 80 % for one) and, next, by the latency of the four gathers
// per (pixel, element, transmit) term.  Lanes run along x: neighbouring pixels of a row read samples at most a lateral
// step apart (0.5 on average on the 512 x 256 image of 128 elements), so a row's gather touches one
// or two cache lines, where lanes along depth are 2 dz fs / c = 12 samples apart and touch one sector
// each.  A CTA's warps take consecutive rows of one x range, which share lines the same way.  The
// receive delay is formed once per (pixel, element) and serves KT transmits; times are 32.32 fixed
// point, so a term adds, splits and compares integers.  512 x 256 image of 128 elements x 3200 samples,
// before (lanes along depth; float-float add, floor, IEEE square root and divide per term) and now:
// 31 transmits 3044 -> 682 us, one transmit 98 -> 48 us; 25 transmits x 4096 samples 2451 -> 541 us.
// Registers for the loads of a whole chunk pay more than warps once a chunk is long (31 transmits:
// 680 us at 2 CTAs per SM, 760 at 3, 940 at 4), and the other way round for single transmits.
template <int KT>
constexpr int das_ctas_per_sm() { return KT >= 5 ? 2 : KT >= 3 ? 3 : 4; }

template <bool CONVEX, int KT>
__global__ void __launch_bounds__(256, das_ctas_per_sm<KT>()) k_das(const ImageP I, const DasTile D) {
    extern __shared__ ff s_xe[];  // element centres in samples: x [n_el] (then z [n_el] if CONVEX); partial sums later
    for (int e = threadIdx.x; e < I.n_el; e += blockDim.x) {
        ff x, z;
        element_centre<CONVEX>(I, e, x, z);
        s_xe[e] = ff_mul(x, I.q);
        if (CONVEX) s_xe[I.n_el + e] = ff_mul(z, I.q);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int part = warp % D.split, group = warp / D.split;
    const int rows = 32 >> D.wx_log2;
    const int ix = ((blockIdx.x % D.tiles_x) << D.wx_log2) + (lane & ((1 << D.wx_log2) - 1));
    const int iz = ((int)(blockIdx.x / D.tiles_x) * (8 / D.split) + group) * rows + (lane >> D.wx_log2);
    const bool in = ix < I.nx && iz < I.nz;
    const int img = blockIdx.z;
    const int q0 = I.img_items ? I.img_begin[img] : 0;
    const int q1 = I.img_items ? I.img_begin[img + 1] : I.n_tx;
    const int e0 = I.n_el * part / D.split, e1 = I.n_el * (part + 1) / D.split;
    // lanes past the image's edge repeat its last pixel
    const float x = I.x_px[min(ix, I.nx - 1)], z = I.z_px[min(iz, I.nz - 1)];
    const ff xs = ff_mul_f(x, I.q), zs = ff_mul_f(z, I.q);
    const ff zz = ff_mul(zs, zs);
    // no receive delay exceeds the distance to element 0 plus the aperture's length (false for NaN)
    const float far = fabsf(xs.hi - s_xe[0].hi) + fabsf(zs.hi - (CONVEX ? s_xe[I.n_el].hi : 0.f)) +
                      (float)I.n_el * I.pitch * I.q.hi;
    const bool near_px = far < kFixedMax;
    const unsigned long long top = (unsigned long long)(I.n_s - 1) << 32;
    const long long to_quad = (const char *)I.quad - (const char *)I.rf;
    float sr = 0.f, si = 0.f;
    const int n_chunks = (q1 - q0 + KT - 1) / KT;
    for (int c = 0; c < n_chunks; ++c) {
        const int qa = q0 + (int)((long long)(q1 - q0) * c / n_chunks);
        const int nk = q0 + (int)((long long)(q1 - q0) * (c + 1) / n_chunks) - qa;
        long long T[KT];
        const float *base[KT];
        bool fixed = near_px;
#pragma unroll
        for (int j = 0; j < KT; ++j) {
            T[j] = kNoTransmit;
            base[j] = I.rf;
            if (j < nk) {
                const int item = I.img_items ? I.img_items[qa + j] : qa + j;
                const ff t = transmit_delay(I, I.img_items ? I.item_angle[item] : item, x, z);
                fixed = fixed && fabsf(t.hi) < kFixedMax;
                T[j] = to_fixed(t.hi, t.lo);
                base[j] = I.rf + (size_t)item * I.n_el * I.n_s;
            }
        }
        if (!fixed) {
            for (int j = 0; j < nk; ++j) {
                const int item = I.img_items ? I.img_items[qa + j] : qa + j;
                const float2 v = das_wide<CONVEX>(I, item, I.img_items ? I.item_angle[item] : item, e0, e1, x, z);
                sr += v.x;
                si += v.y;
            }
            continue;
        }
#pragma unroll (KT == 1 ? 4 : 1)   // a single transmit's loads: four elements in flight (52 -> 48 us)
        for (int e = e0; e < e1; ++e) {
            const ff xe = s_xe[e];
            const ff d = ff_two_sum(xs.hi, -xe.hi);
            const float dl = d.lo + (xs.lo - xe.lo);
            const float p = __fmul_rn(d.hi, d.hi);
            float pl = __fmaf_rn(2.f * d.hi, dl, __fmaf_rn(d.hi, d.hi, -p));
            ff r;
            if (CONVEX) {
                const ff ze = s_xe[I.n_el + e];
                const ff v = ff_two_sum(zs.hi, -ze.hi);
                const float vl = v.lo + (zs.lo - ze.lo);
                const float w = __fmul_rn(v.hi, v.hi);
                pl += __fmaf_rn(2.f * v.hi, vl, __fmaf_rn(v.hi, v.hi, -w));
                r = ff_two_sum(w, p);
                r.lo += pl;
            } else {
                r = ff_two_sum(zz.hi, p);
                r.lo += pl + zz.lo;
            }
            // square root: the approximate one and a Newton correction from the exact residual
            const float y = rsqrt_approx(fmaxf(r.hi, 1e-30f));
            const float s = __fmul_rn(r.hi, y);
            const long long R = to_fixed(s, (__fmaf_rn(-s, s, r.hi) + r.lo) * (0.5f * y));
            const int row = e * I.n_s;
            float pr = 0.f, pi = 0.f;
#pragma unroll
            for (int j = 0; j < KT; ++j) {
                const unsigned long long tau = (unsigned long long)(T[j] + R);
                const unsigned i0 = (unsigned)(tau >> 32);
                const float f = __uint2float_rn((unsigned)tau) * 0x1p-32f;
                const float *a = base[j] + (row + (int)i0);
                float a0, a1, b0, b1;
                gather(a, (const float *)((const char *)a + to_quad), tau, top, a0, a1, b0, b1);
                const float g = 1.f - f;
                pr = fmaf(a1, f, fmaf(a0, g, pr));
                pi = fmaf(b1, f, fmaf(b0, g, pi));
            }
            sr += pr;
            si += pi;
        }
    }
    if (D.split > 1) {   // the parts of a pixel's elements are summed by the first of its warps
        float2 *s_sum = (float2 *)s_xe;
        __syncthreads();
        s_sum[threadIdx.x] = make_float2(sr, si);
        __syncthreads();
        if (part != 0) return;
        for (int q = 1; q < D.split; ++q) {
            const float2 v = s_sum[threadIdx.x + 32 * q];
            sr += v.x;
            si += v.y;
        }
    }
    float env = 0.f;
    if (in) {
        const size_t px = ((size_t)img * I.nz + iz) * I.nx + ix;
        if (I.iq) I.iq[px] = make_float2(sr, si);
        env = sqrtf(sr * sr + si * si);
        if (I.env) I.env[px] = env;
    }
    const unsigned int m = __reduce_max_sync(0xffffffffu, __float_as_uint(env));
    if (lane == 0 && m) atomicMax(&I.env_max[img], m);
}

__global__ void k_log(const ImageP I) {
    const int n = I.nx * I.nz;
    const int img = blockIdx.y;
    const float mx = __uint_as_float(I.env_max[img]);
    const float *env = I.env + (size_t)img * n;
    float *db = I.db + (size_t)img * n;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        const float e = env[p];
        float v = (mx > 0.f && e > 0.f) ? 20.f * log10f(e / mx) : -I.dyn_range_db;
        db[p] = fmaxf(v, -I.dyn_range_db);
    }
}

}  // namespace

namespace {

template <int KT>
void launch_das_kt(const ImageP &I, const DasTile &D, dim3 grid, cudaStream_t s) {
    const size_t elems = (size_t)I.n_el * sizeof(ff) * (I.elem_xz ? 2 : 1);
    const size_t smem = elems > 256 * sizeof(float2) ? elems : 256 * sizeof(float2);
    if (smem > 48 * 1024)   // convex arrays of more than 3072 elements; one value for every caller, up to 4096
        cudaFuncSetAttribute(k_das<true, KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 4096 * 2 * (int)sizeof(ff));
    if (I.elem_xz)
        k_das<true, KT><<<grid, 256, smem, s>>>(I, D);
    else
        k_das<false, KT><<<grid, 256, smem, s>>>(I, D);
}

}  // namespace

void launch_das(const ImageP &I, cudaStream_t s) {
    const int images = I.img_items ? I.n_images : 1;
    DasTile D;
    D.wx_log2 = 0;   // narrow images: as many pixels along x as there are, the warp's other lanes along z
    while (D.wx_log2 < (I.nx >= kWideImage ? 4 : 3) && (1 << D.wx_log2) < I.nx) ++D.wx_log2;
    D.tiles_x = (I.nx + (1 << D.wx_log2) - 1) >> D.wx_log2;
    // small images: warps share a pixel's elements until there are about kDasWarps of them
    const long long warps = (((long long)I.nx * I.nz + 31) >> 5) * images;
    D.split = 1;
    while (D.split < 8 && warps * D.split < kDasWarps && I.n_el >= 16 * D.split) D.split *= 2;
    const int tile_z = (8 / D.split) * (32 >> D.wx_log2);
    const dim3 grid(D.tiles_x * ((I.nz + tile_z - 1) / tile_z), 1, images);
    // transmits per chunk: the fewest (chunk, slot) steps, a chunk's receive delays costing about two slots' terms
    const int n = I.img_items ? (I.n_tx + images - 1) / images : I.n_tx;   // transmits of an image (on average)
    int kt = 1, best = n * 3;
    for (int k = 2; k <= 8; ++k) {
        const int cost = (n + k - 1) / k * (k + 2);
        if (k != 7 && cost <= best) {
            best = cost;
            kt = k;
        }
    }
    switch (kt) {
        case 1: launch_das_kt<1>(I, D, grid, s); break;
        case 2: launch_das_kt<2>(I, D, grid, s); break;
        case 3: launch_das_kt<3>(I, D, grid, s); break;
        case 4: launch_das_kt<4>(I, D, grid, s); break;
        case 5: launch_das_kt<5>(I, D, grid, s); break;
        case 6: launch_das_kt<6>(I, D, grid, s); break;
        default: launch_das_kt<8>(I, D, grid, s);
    }
}

void launch_log(const ImageP &I, cudaStream_t s) {
    const int n = I.nx * I.nz;
    dim3 grid(min(4096, (n + 255) / 256), I.img_items ? I.n_images : 1);
    k_log<<<grid, 256, 0, s>>>(I);
}

}  // namespace ur
