// Forward march kernels (Sec. 4.1-4.2): one thread per ray, warps on 8 x 4
// pixel tiles (several lanes per ray in small launches), bricked volume gathers
// through the read-only path, transfer function in shared memory (1-D) or global
// memory (2-D), exact empty-space skipping by one empty level per 4^3 sub-block
// and early ray termination lane by lane. The instances are spread over several translation units
// (rc_march.cu, rc_march_cubic.cu, rc_march_tf2.cu) so they compile in parallel.
#pragma once

#include "rc_device.cuh"

namespace rc {

constexpr unsigned kFull = 0xffffffffu;

// A CTA renders a tile of kTileW x kTileH pixels, each warp an 8 x 4 block
// of it.
constexpr int kWarpsX = 2, kWarpsY = 2;
constexpr int kTileW = 8 * kWarpsX, kTileH = 4 * kWarpsY, kMarchThreads = 32 * kWarpsX * kWarpsY;

__device__ __forceinline__ void pixel_of_thread(int &x, int &y) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    x = blockIdx.x * kTileW + (warp % kWarpsX) * 8 + (lane & 7);
    y = blockIdx.y * kTileH + (warp / kWarpsX) * 4 + (lane >> 3);
}

__device__ __forceinline__ void add_stats(unsigned long long *stats, unsigned dense, unsigned evald,
                                          unsigned hit, unsigned inimg) {
    dense = __reduce_add_sync(kFull, dense);
    evald = __reduce_add_sync(kFull, evald);
    hit = __reduce_add_sync(kFull, hit);
    inimg = __reduce_add_sync(kFull, inimg);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(stats + 0, (unsigned long long)dense);
        atomicAdd(stats + 1, (unsigned long long)evald);
        atomicAdd(stats + 2, (unsigned long long)hit);
        atomicAdd(stats + 3, (unsigned long long)inimg);
    }
}

// Compositing ray function (Sec. 4.2, Eq. 4): C += T a' c, T *= (1 - a'),
// front to back from the eye; stop after the sample where 1 - T >= term.
// F selects the sample form (kShade, kCubic, kTF2).
//
// Instruction issue and the L1 data path bound it, with the latency of one
// sample's chain (level, voxels, table) behind both. One turn of the loop is
// - two samples for the plain trilinear form, whose 8 loads leave registers
//   for a second sample in flight (4 FP16 views of 181x217x157 at 901x703:
//   0.342 -> 0.327 ms; 4 shaded views of 256x256x180 at 1024^2 0.875 -> 0.905:
//   there the registers cost more warps than the overlap gains);
// - one sample with the next one's cell and level fetched under it for the
//   forms that read gradients from FP32 and uint16 volumes (shaded 0.916 ->
//   0.875, 512x512x256 at 2048^2, step 1/4, 1.320 -> 1.283, 2-D table 1.813 ->
//   1.774; FP16, with its longer decode, 0.892 -> 0.898 and 1.283 -> 1.310);
// - one sample at a time else (B-spline 1.725 -> 1.762 with the fetch).
// Lanes leave the loop one by one: holding the warp together by a vote per
// turn took uint16 at 512x512x256, 2048^2, from 1.37 to 1.45 ms.
constexpr bool reads_gradients(int F) { return (F & (kShade | kTF2)) != 0 && !(F & kCubic); }

enum : int { kTurnOne = 0, kTurnPair = 1, kTurnAhead = 2 };

template <int ST, int F, int RM>
__global__ void __launch_bounds__(kMarchThreads) composite_kernel(const MarchArgs a) {
    constexpr int kTurn = F == 0 ? kTurnPair
                          : reads_gradients(F) && (ST & 3) != RC_STORE_F16 ? kTurnAhead : kTurnOne;
    extern __shared__ float4 s_tf[];
    if (!(F & kTF2)) {
        load_tf(a.tf, s_tf);
        __syncthreads();
    }
    // a batch of volumes: the volume's own data and masks, the shared record
    VolDev vol = a.vol;
    const uint8_t *lvl = a.lvl;
    int view = blockIdx.z;
    if (a.batch) {
        const int vi = blockIdx.z / a.views;
        view = blockIdx.z - vi * a.views;
        const BatchVol bv = a.batch[vi];
        vol.data = bv.data;
        vol.vg = bv.vg;
        vol.pairs = bv.pairs;
        lvl = bv.lvl;
    }
    const CamRec cam = a.cams ? a.cams[view] : a.cam;
    float4 *out = a.out + (size_t)blockIdx.z * cam.W * cam.H;
    int x, y;
    pixel_of_thread(x, y);
    const bool inimg = x < cam.W && y < cam.H;
    Ray R;
    const bool hit = inimg && setup_ray(cam, vol, a.p.step_vox, x, y, R);
    const int nsamp = hit ? R.nsamp : 0;
    float C0 = 0.0f, C1 = 0.0f, C2 = 0.0f, T = 1.0f;
    float k = 0.0f;               // sample counter: a float (exact, below 2^24) needs no conversion per sample
    const float n = (float)nsamp;
    unsigned evald = 0;
    bool active = nsamp > 0;
    auto cell_at = [&](float i, Cell &c) {
        float p[3];
        position_at(R, __fmaf_rn(i, R.ds, R.tn), p);
        cell_of(vol, p, c);
    };
    auto level = [&](const Cell &c) { return a.p.skip ? empty_level(a, lvl, c) : 0; };
    auto sample = [&](const Cell &c) {
        return eval_sample_x<ST, F, RM>(vol, a.p, s_tf, a.tf, R.dir, c, a.p.rmode, a.p.ratio);
    };
    auto add = [&](const float4 &e) {
        composite_add(e, C0, C1, C2, T);
        evald++;
        k += 1.0f;
        active = k < n && (1.0f - T) < a.p.term;
    };
    // past the largest empty block around the sample: its cell-brick, octant
    // or 4^3 sub-block
    auto jump = [&](const Cell &c, int s) {
        k = (float)jump_block(R, vol, c, (int)k, s);
        active = k < n;
    };
    if constexpr (kTurn == kTurnPair) {
        while (active) {
            Cell c, cn;
            cell_at(k, c);
            cell_at(k + 1.0f, cn);                 // past the end: clamped into the volume, not used
            const int s = level(c), sn = level(cn);
            if (s) {
                jump(c, s);
                continue;
            }
            const float4 e = sample(c), en = sample(cn);
            add(e);
            if (active && !sn) add(en);
        }
    } else if constexpr (kTurn == kTurnAhead) {
        Cell c;
        int s = 0;
        if (active) {
            cell_at(0.0f, c);
            s = level(c);
        }
        while (active) {
            if (s) {
                jump(c, s);
                cell_at(k, c);
                s = level(c);
                continue;
            }
            Cell cn;
            cell_at(k + 1.0f, cn);
            s = level(cn);
            add(sample(c));
            c = cn;
        }
    } else {
        while (active) {
            Cell c;
            cell_at(k, c);
            const int s = level(c);
            if (s) jump(c, s);
            else add(sample(c));
        }
    }
    __syncwarp();
    if (inimg) out[(size_t)y * cam.W + x] = make_float4(C0, C1, C2, 1.0f - T);
    if (a.stats) add_stats(a.stats, (unsigned)min((int)k, nsamp), evald, hit ? 1u : 0u, inimg ? 1u : 0u);
}

// The compositing march with L lanes per ray, for launches too small to fill
// the GPU with one: lane j of a ray's group evaluates sample k + j, then every
// lane of the group composites the L samples in order from shuffles, so the
// image is composite_kernel's bit for bit and a ray's chain of dependent
// sample latencies is L times shorter. Samples past a termination are
// evaluated in vain and the shuffles cost issue slots: lanes_per_ray says
// where that pays.
template <int L> struct WideTile { static constexpr int X = 8, Y = 4; };
template <> struct WideTile<2> { static constexpr int X = 4, Y = 4; };
template <> struct WideTile<4> { static constexpr int X = 4, Y = 2; };
template <> struct WideTile<8> { static constexpr int X = 2, Y = 2; };

template <int ST, int F, int L>
__global__ void __launch_bounds__(kMarchThreads) wide_kernel(const MarchArgs a) {
    extern __shared__ float4 s_tf[];
    if (!(F & kTF2)) {
        load_tf(a.tf, s_tf);
        __syncthreads();
    }
    VolDev vol = a.vol;
    const uint8_t *lvl = a.lvl;
    int view = blockIdx.z;
    if (a.batch) {
        const int vi = blockIdx.z / a.views;
        view = blockIdx.z - vi * a.views;
        const BatchVol bv = a.batch[vi];
        vol.data = bv.data;
        vol.vg = bv.vg;
        vol.pairs = bv.pairs;
        lvl = bv.lvl;
    }
    const CamRec cam = a.cams ? a.cams[view] : a.cam;
    float4 *out = a.out + (size_t)blockIdx.z * cam.W * cam.H;
    constexpr int TX = WideTile<L>::X, TY = WideTile<L>::Y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = lane % L, ray = lane / L, first = lane - j;
    const int x = blockIdx.x * (kWarpsX * TX) + (warp % kWarpsX) * TX + ray % TX;
    const int y = blockIdx.y * (kWarpsY * TY) + (warp / kWarpsX) * TY + ray / TX;
    const bool inimg = x < cam.W && y < cam.H;
    Ray R;
    const bool hit = inimg && setup_ray(cam, vol, a.p.step_vox, x, y, R);
    const int nsamp = hit ? R.nsamp : 0;
    float C0 = 0.0f, C1 = 0.0f, C2 = 0.0f, T = 1.0f;
    int k = 0;
    unsigned evald = 0;
    bool active = nsamp > 0;
    while (__any_sync(kFull, active)) {
        // every lane of a group has the same k, active, C and T
        const bool turn = active, in = turn && k + j < nsamp;
        Cell c;
        int s = 0;
        if (in) {
            float p[3];
            position_at(R, sample_t(R, k + j), p);
            cell_of(vol, p, c);
            if (a.p.skip) s = empty_level(a, lvl, c);
        }
        const unsigned vis = (__ballot_sync(kFull, in && s == 0) >> first) & ((1u << L) - 1u);
        float4 e = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        int next = k + j + 1;
        if (in && s == 0) e = eval_sample_x<ST, F>(vol, a.p, s_tf, a.tf, R.dir, c, a.p.rmode, a.p.ratio);
        else if (in && vis == 0) next = jump_block(R, vol, c, k + j, s);
        // all L samples empty: on from the last one's block
        next = __shfl_sync(kFull, next, first + max(min(nsamp - 1 - k, L - 1), 0));
#pragma unroll
        for (int i = 0; i < L; i++) {
            const float4 q = make_float4(__shfl_sync(kFull, e.x, first + i), __shfl_sync(kFull, e.y, first + i),
                                         __shfl_sync(kFull, e.z, first + i), __shfl_sync(kFull, e.w, first + i));
            if (active && ((vis >> i) & 1u)) {
                composite_add(q, C0, C1, C2, T);
                evald++;
                active = (1.0f - T) < a.p.term;
                if (!active) next = k + i + 1;
            }
        }
        if (turn) k = next;
        active = active && k < nsamp;
    }
    if (inimg && j == 0) out[(size_t)y * cam.W + x] = make_float4(C0, C1, C2, 1.0f - T);
    if (a.stats) {
        const bool one = j == 0;
        add_stats(a.stats, one ? (unsigned)min(k, nsamp) : 0u, one ? evald : 0u, one && hit ? 1u : 0u, one && inimg ? 1u : 0u);
    }
}

// The largest block around cell c (brick b) whose codes cannot matter, none of
// them above `need`: 4 for the cell-brick, 2 for the 4^3 sub-block, -1 when the
// sample has to be evaluated. need is a threshold in code units less a.slack,
// rounded down (the conversion takes infinities to the ends of int). A block's maximum
// code bounds every value reconstructed in it up to FP32 rounding (and, for
// FP16 storage of more than 12 bits, the rounding of the stored values);
// a.slack covers both many times over, so a skipped sample is strictly below
// `need`.
__device__ __forceinline__ int low_block(const MarchArgs &a, const Cell &c, int b, int need) {
    const int j = ((c.i[2] >> 2) * a.c4[1] + (c.i[1] >> 2)) * a.c4[0] + (c.i[0] >> 2);
    if ((int)__ldg(a.mx4 + j) > need) return -1;
    return (int)__ldg(a.mx + b) > need ? 2 : 4;
}

// The first-hit functions of Sec. 4.1 (isosurface, threshold); output channels
// as documented in rc.h. CUBIC: B-spline values and analytic gradient instead
// of trilinear values and central differences.
//
// They march the block maxima instead of every sample: a sample in a 4^3
// sub-block or cell-brick whose largest code cannot reach the iso-value changes
// nothing, so the ray jumps over the block (the compositing march's exact jump,
// verified on the sample grid). A warp jumps only when none of its lanes has to
// evaluate: in noise the lanes' blocks alternate, and a jump costs more than
// the sample it saves. The value before a hit is reconstructed once, when the
// hit is found. Instruction issue bounds it. 256x256x180 phantom at 1024^2, 4
// isosurface views: 0.725 -> 0.253 ms.
template <int ST, bool CUBIC>
__global__ void __launch_bounds__(kMarchThreads) function_kernel(const MarchArgs a) {
    extern __shared__ float4 s_tf[];
    const int func = a.p.func;
    if (func == RC_FUNC_THRESHOLD) {   // the only one that classifies (1-D table)
        load_tf(a.tf, s_tf);
        __syncthreads();
    }
    const CamRec cam = a.cams ? a.cams[blockIdx.z] : a.cam;
    float4 *outp = a.out + (size_t)blockIdx.z * cam.W * cam.H;
    int x, y;
    pixel_of_thread(x, y);
    const bool inimg = x < cam.W && y < cam.H;
    Ray R;
    const bool hit = inimg && setup_ray(cam, a.vol, a.p.step_vox, x, y, R);
    const int nsamp = hit ? R.nsamp : 0;
    float4 out = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    int k = 0;
    unsigned evald = 0;
    int hit_k = -1;
    auto value = [&](const Cell &c) { return CUBIC ? bspline<ST>(a.vol, c) : trilinear<ST>(a.vol, c); };
    // the threshold in code units (FP16 storage holds h = code / o - 1)
    const int need = __float2int_rd((ST == RC_STORE_F16 ? (a.p.iso + 1.0f) * a.vol.f16o : a.p.iso) - a.slack);
    auto cell_at = [&](int j, Cell &c) {
        float p[3];
        position_at(R, sample_t(R, j), p);
        cell_of(a.vol, p, c);
    };
    bool active = nsamp > 0;
    while (__any_sync(kFull, active)) {
        Cell c0, c1;
        if (active) cell_at(k, c0);
        if (a.p.skip) {
            const int s = active ? low_block(a, c0, brick_of(a.vol, c0), need) : 4;
            if (!__any_sync(kFull, s < 0)) {
                if (active) {
                    k = jump_block(R, a.vol, c0, k, s);
                    active = k < nsamp;
                }
                continue;
            }
        }
        if (!active) continue;
        // two samples per turn; a second one past the end is clamped into the
        // volume and ignored
        cell_at(k + 1, c1);
        const float v0 = value(c0), v1 = value(c1);
        const bool two = k + 1 < nsamp;
        if (v0 >= a.p.iso || (two && v1 >= a.p.iso)) {
            if (!(v0 >= a.p.iso)) {
                k++;
                evald++;
            }
            evald++;
            hit_k = k++;
            active = false;
            continue;
        }
        k += 2;
        evald += two ? 2 : 1;
        active = k < nsamp;
    }
    if (hit_k >= 0) {
        // the hit's value again, and for an isosurface the value before it
        const float t = sample_t(R, hit_k);
        Cell c;
        cell_at(hit_k, c);
        const float v = value(c);
        if (func == RC_FUNC_THRESHOLD) {
            float4 e = classify(s_tf, a.tf.K, tf_coord<ST>(v, a.tf.ucoef), nullptr, nullptr, RC_DBG_ERR(a.vol));
            out = make_float4(e.x, e.y, e.z, 1.0f);
        } else {
            float ts = t;
            if (hit_k > 0) {
                const float prev_t = sample_t(R, hit_k - 1);
                Cell cp;
                cell_at(hit_k - 1, cp);
                const float prev_v = value(cp);
                ts = prev_t + (t - prev_t) * ((a.p.iso - prev_v) / (v - prev_v));
            }
            float g[3], sf, spec;
            if (CUBIC) bspline_grad<ST>(a.vol, c, g);
            else value_grad_any<ST>(a.vol, c, g);
            shade_factor(a.p, a.vol, g, R.dir, sf, spec);
            out = make_float4(ts, fminf(1.0f, sf + spec), (float)hit_k, 1.0f);
        }
    }
    k = min(k, nsamp);
    if (inimg) outp[(size_t)y * cam.W + x] = out;
    if (a.stats) add_stats(a.stats, (unsigned)k, evald, hit ? 1u : 0u, inimg ? 1u : 0u);
}

// Average, x-ray and (MAX) MIP: the sum or the maximum of every sample. L lanes
// per ray as in wide_kernel: lane j reconstructs sample k + j and the group adds
// the L values in sample order from shuffles (the same sum bit for bit); a
// maximum does not depend on the order, so each lane keeps its own to the end.
// The measured times stand at lanes_per_sum and lanes_per_max. Bound by
// instruction issue, for the B-spline by its chain of gathers.
// MIP takes every sample: in noise the maxima of 4^3 blocks lie above any value
// reconstructed in them, so skipping by them (as function_kernel does) left 60%
// of the samples of a head phantom and a longer chain per sample. One 128^2 view
// of 256x256x180, us: 304 with skipping, 171 with one lane and every sample, 65
// with the lanes; eight 1024^2 views 1992, 2188 and 1984.
template <int ST, bool CUBIC, int L, bool MAX>
__global__ void __launch_bounds__(kMarchThreads) reduce_kernel(const MarchArgs a) {
    const CamRec cam = a.cams ? a.cams[blockIdx.z] : a.cam;
    float4 *outp = a.out + (size_t)blockIdx.z * cam.W * cam.H;
    constexpr int TX = WideTile<L>::X, TY = WideTile<L>::Y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = lane % L, ray = lane / L, first = lane - j;
    const int x = blockIdx.x * (kWarpsX * TX) + (warp % kWarpsX) * TX + ray % TX;
    const int y = blockIdx.y * (kWarpsY * TY) + (warp / kWarpsX) * TY + ray / TX;
    const bool inimg = x < cam.W && y < cam.H;
    Ray R;
    const bool hit = inimg && setup_ray(cam, a.vol, a.p.step_vox, x, y, R);
    const int nsamp = hit ? R.nsamp : 0;
    float acc = MAX ? -__int_as_float(0x7f800000) : 0.0f;
    auto value = [&](int k) {
        float p[3];
        position_at(R, sample_t(R, k), p);
        Cell c;
        cell_of(a.vol, p, c);
        return CUBIC ? bspline<ST>(a.vol, c) : trilinear<ST>(a.vol, c);
    };
    if constexpr (MAX) {
#pragma unroll 1
        for (int k = j; k < nsamp; k += L) acc = fmaxf(acc, value(k));
        __syncwarp();
#pragma unroll
        for (int i = 1; i < L; i <<= 1) acc = fmaxf(acc, __shfl_xor_sync(kFull, acc, i));
    } else if constexpr (L == 1) {
#pragma unroll 1
        for (int k = 0; k < nsamp; k++) acc += value(k);
    } else {
#pragma unroll 1
        for (int k = 0; __any_sync(kFull, k < nsamp); k += L) {
            const float v = k + j < nsamp ? value(k + j) : 0.0f;
#pragma unroll
            for (int i = 0; i < L; i++) {
                const float q = __shfl_sync(kFull, v, first + i);
                if (k + i < nsamp) acc += q;
            }
        }
    }
    // over full scale; FP16 values h = code / o - 1 are shifted by 1 (a sum's by 1
    // per sample) first
    float4 out = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (nsamp > 0) {
        const float n = (float)nsamp;
        float m;
        if (MAX)
            m = (ST == RC_STORE_F16 ? acc + 1.0f : acc) / a.vol.vscale;
        else if (ST == RC_STORE_F16)
            m = a.p.func == RC_FUNC_AVERAGE ? (acc / n + 1.0f) / a.vol.vscale : (acc + n) * R.ds / a.vol.vscale;
        else
            m = a.p.func == RC_FUNC_AVERAGE ? acc / n / a.vol.vscale : acc * R.ds / a.vol.vscale;
        out = make_float4(m, m, m, 1.0f);
    }
    const bool one = j == 0;
    if (inimg && one) outp[(size_t)y * cam.W + x] = out;
    if (a.stats) {
        const unsigned n = one ? (unsigned)nsamp : 0u;
        add_stats(a.stats, n, n, one && hit ? 1u : 0u, one && inimg ? 1u : 0u);
    }
}

template <typename K>
static cudaError_t launch_kernel(K kern, const MarchArgs &a, int nviews, bool table_in_smem, cudaStream_t s,
                                 int tile_w = kTileW, int tile_h = kTileH) {
    size_t smem = table_in_smem ? (size_t)a.tf.K * sizeof(float4) : 0;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((a.cam.W + tile_w - 1) / tile_w, (a.cam.H + tile_h - 1) / tile_h, nviews);
    kern<<<grid, kMarchThreads, smem, s>>>(a);
    return cudaGetLastError();
}

static int lanes_per_ray(const MarchArgs &a) {
    if (a.cam.H > 4 * 65535) return 1;     // the grid's y limit at 4 rows per CTA
    return lanes_per_ray(a.size, (a.p.shade && !a.vol.vg16) || a.p.filter == RC_FILTER_BSPLINE || a.tf.M >= 2);
}

template <int F, int L>
static cudaError_t launch_wide(const MarchArgs &a, int nviews, cudaStream_t s) {
    const bool smem = !(F & kTF2);
    constexpr int W = kWarpsX * WideTile<L>::X, H = kWarpsY * WideTile<L>::Y;
    return by_storage<reads_gradients(F)>(a.vol, [&](auto st) {
        return launch_kernel(wide_kernel<decltype(st)::value, F, L>, a, nviews, smem, s, W, H);
    });
}

// Composite march with sample form F and opacity-correction mode RM for the
// volume's storage type.
template <int F, int RM>
static cudaError_t launch_composite_rm(const MarchArgs &a, int nviews, cudaStream_t s) {
    const bool smem = !(F & kTF2);
    return by_storage<reads_gradients(F)>(a.vol, [&](auto st) {
        return launch_kernel(composite_kernel<decltype(st)::value, F, RM>, a, nviews, smem, s);
    });
}

// The step ratios of the fixed modes (1, 1/2, 1/4) get their own instances.
template <int F>
static cudaError_t launch_composite(const MarchArgs &a, int nviews, cudaStream_t s) {
    switch (lanes_per_ray(a)) {
        case 8: return launch_wide<F, 8>(a, nviews, s);
        case 4: return launch_wide<F, 4>(a, nviews, s);
        case 2: return launch_wide<F, 2>(a, nviews, s);
    }
    switch (a.p.rmode) {
        case 0: return launch_composite_rm<F, 0>(a, nviews, s);
        case 1: return launch_composite_rm<F, 1>(a, nviews, s);
        case 2: return launch_composite_rm<F, 2>(a, nviews, s);
        default: return launch_composite_rm<F, 3>(a, nviews, s);
    }
}

template <bool CUBIC, bool MAX, int L>
static cudaError_t launch_reduce_lanes(const MarchArgs &a, int nviews, cudaStream_t s) {
    constexpr int TX = WideTile<L>::X, TY = WideTile<L>::Y;
    return by_storage<false>(a.vol, [&](auto st) {
        return launch_kernel(reduce_kernel<decltype(st)::value, CUBIC, L, MAX>, a, nviews, false, s, kWarpsX * TX,
                             kWarpsY * TY);
    });
}

template <bool CUBIC, bool MAX>
static cudaError_t launch_reduce(const MarchArgs &a, int nviews, cudaStream_t s) {
    int lanes = MAX ? lanes_per_max(a.size, CUBIC) : lanes_per_sum(a.size, CUBIC);
    if (lanes == 4 && a.cam.H > 4 * 65535) lanes = 2;      // the grid's y limit at 4 rows per CTA
    switch (lanes) {
        case 4: return launch_reduce_lanes<CUBIC, MAX, 4>(a, nviews, s);
        case 2: return launch_reduce_lanes<CUBIC, MAX, 2>(a, nviews, s);
        default: return launch_reduce_lanes<CUBIC, MAX, 1>(a, nviews, s);
    }
}

template <bool CUBIC>
static cudaError_t launch_function(const MarchArgs &a, int nviews, cudaStream_t s) {
    switch (a.p.func) {
        case RC_FUNC_MIP: return launch_reduce<CUBIC, true>(a, nviews, s);
        case RC_FUNC_AVERAGE:
        case RC_FUNC_XRAY: return launch_reduce<CUBIC, false>(a, nviews, s);
        default:
            return by_storage<false>(a.vol, [&](auto st) {
                return launch_kernel(function_kernel<decltype(st)::value, CUBIC>, a, nviews,
                                     a.p.func == RC_FUNC_THRESHOLD, s);
            });
    }
}

}  // namespace rc
