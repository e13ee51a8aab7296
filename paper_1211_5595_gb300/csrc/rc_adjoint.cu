// Adjoint of the compositing ray function with respect to the transfer-function
// table (Eq. 4-5 are differentiable in the table entries).
//
// Per ray, pass 1 recomputes the forward march (with exact empty-space
// skipping) to get C_final, T_final and the number n of samples up to
// termination; when the caller gives the forward images, C_final and T_final
// are read from them instead and pass 2 stops at the termination sample by
// itself (it rebuilds T sample by sample, and the skipped samples of the
// forward have zero opacity, so its stop decisions are the forward's). Pass 2
// marches again front to back, rebuilding T_k and the prefix C_{<=k}, so that
// the suffix S_k = C_final - C_{<=k} is known without storing samples or
// dividing transmittance backwards:
//   dI_c/da'_k = T_k col_kc - S_kc / (1 - a'_k),  dI_a/da'_k = T_k - (T_{k+1} - T_n) / (1 - a'_k)
//   dI_c/dcol_kc = T_k a'_k,  da'/da = r (1 - min(a, 1 - 1e-6))^(r - 1)
// and the two table entries of the sample's lerp receive weights (1 - w, w).
// Lanes of a warp that hit the same entries are summed first (a fixed tree
// order). A 1-D table of at most kWarpAccK entries then keeps one FP32 copy
// per warp in shared memory, which only that warp's group leaders update, in
// its own program order; at the end each CTA adds its warps' copies in warp
// order and converts the sums to 64-bit fixed point (scale 2^32 / max|dL/dI|)
// for the global sums. Larger 1-D tables add each group's sums as 64-bit fixed
// point to the CTA's shared accumulators directly, 2-D tables as 32-bit words
// with the overflows sent on (Acc2). Integer sums do not depend
// on the order of the atomics, and no other sum depends on thread scheduling,
// so the result is deterministic.
#include "rc_device.cuh"
#include "rc_rules.h"

namespace rc {

__global__ void absmax_kernel(const float *__restrict__ x, long long n, unsigned *out) {
    float m = 0.0f;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(x[i]));
    unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0) atomicMax(out, u);
}

cudaError_t launch_absmax(const float *x, long long n, float *out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(float), s);
    if (e != cudaSuccess) return e;
    absmax_kernel<<<1216, 256, 0, s>>>(x, n, (unsigned *)out);
    return cudaGetLastError();
}

// Fixed-point units per unit of gradient, finite for every dL/dI: the floor is
// the smallest maximum whose scale does not overflow FP32 (2^32 / 1.3e-29 =
// 3.30e38), so zeros stay zeros when they are scaled.
__device__ __forceinline__ float fixed_scale(const float *absmax) {
    return 4294967296.0f / fmaxf(*absmax, 1.3e-29f);
}

__device__ __forceinline__ void acc_add(unsigned long long *acc, int idx, float v, float scale) {
    long long q = __float2ll_rn(v * scale);
    if (q != 0) atomicAdd(acc + idx, (unsigned long long)q);
}

// 1-D tables of up to this many entries take the per-warp FP32 accumulators
// (16 B per entry and warp; with the FP32 table 80 B per entry and CTA: 40 KB
// at 512 entries). Measured on the 128x128x96 workload (256 entries, 8 views
// at 512^2, ms per view given the forward images): 0.231 with the CTA's 64-bit
// fixed-point atomics, 0.151 per warp: no conversion and no atomic per group.
constexpr int kWarpAccK = 512;
constexpr int kAdjWarps = 4;                     // warps of a 1-D table's CTA

// Whether a 1-D table's gradient takes the per-warp accumulators: up to
// kWarpAccK entries, except with the cubic B-spline when the forward is
// recomputed: that march's 64-voxel gathers need the L1 capacity the larger
// shared-memory footprint takes (same workload, B-spline, ms per view:
// recomputing 0.529 with the CTA's accumulators, 0.575 per warp; given the
// forward images 0.340 and 0.315).
__host__ __device__ constexpr bool warp_acc(int K, bool cubic, bool given) {
    return K <= kWarpAccK && (!cubic || given);
}

// 2-D table accumulators. The M x K x 4 sums are 64-bit fixed point in global
// memory; each CTA keeps the low 32 bits of its own part in shared memory (and
// 32 high bits of the opacity channel), added with native 32-bit atomics, and
// sends the overflows of the colour channels to global memory. The sums are the
// same integers in any order. A table of up to kDirectSlots
// slots has one per entry, its rows kRowSkew slots further apart than their K
// entries: the entries a warp adds to at once lie in a few adjacent columns
// and rows, and the skew keeps those in different banks. A larger table gets a
// direct-mapped cache of kTagSlots slots with tags: a slot is claimed by the
// first entry that maps to it (compare-and-swap on its tag) and keeps it for the
// CTA's lifetime, and an entry whose slot another entry holds adds to global
// memory. Either takes most of an SM's shared memory, so one CTA of many warps
// runs per SM for the whole launch and the sums are flushed once.
// Measured on 128x128x96, 4 views at 512^2, forward included, ms: 32 x 256
// table 4.12 with a tagged cache of 2048 slots of 64-bit sums per 8 warps, 2.43
// in this form; 16 x 200 6.6 and 2.4 (there the old cache's collisions sent hot
// entries to global memory), 32 x 512 8.8 and 5.3. Taken out one at a time: the
// lanes' grouping by cell 0.62, the 16 conversions to integers 0.45, the atomics
// 0.25. Adding every lane's values without grouping took 0.24 more, one value at
// a time with a test for zero 0.15 more, no high word for opacity up to 1.9 more
// (when dL/dI is steady), 32 warps per SM instead of 24 0.03 more.
constexpr int kRowSkew = 4;
constexpr int kSlotWords = 5, kTagWords = 6;   // 4 low words, opacity's high word, the tag
constexpr int kDirectSlots = 10240;            // 200 KB
constexpr int kTagBits = 13;
constexpr int kTagSlots = 1 << kTagBits;       // 192 KB
// Groups of 8 warps take 16 x 16 pixel chunks from a queue; the number of
// groups per CTA is set by the registers of a thread.
constexpr int kGroupWarps = 8;
constexpr int group_count(bool cubic) { return cubic ? 2 : 3; }

struct Acc2 {
    int *words;                                // kSlotWords (tagged: kTagWords) per slot
    bool tagged;
    int row;                                   // distance of two rows in cell indices: K (tagged) or K + kRowSkew
    int K;
    unsigned long long *g;                     // global sums
    __device__ __forceinline__ unsigned long long *global(int e) const {
        return g + 4 * (size_t)(e - (e / row) * (row - K));
    }
};

// Adds v (fixed-point units) to entry e (row * A.row + column). Colour channels:
// the low word, with the rare wraps and the rare value beyond 31 bits (at most a
// sample or two of a ray: their weights T a' add up to 1 along it) sent to the
// global sum. Opacity: low and high word, since with a steady dL/dI near its
// maximum every sample in front of the tissue is beyond 31 bits.
__device__ __forceinline__ void acc2_add4(const Acc2 &A, int e, const float *f) {
    int *slot = A.words + kSlotWords * e;
    bool own = fabsf(f[3]) < 1099511627776.0f;             // 2^40: the high word sums 2^23 of them
    if (A.tagged) {
        slot = A.words + kTagWords * (((unsigned)e * 2654435761u) >> (32 - kTagBits));
        int t = *reinterpret_cast<volatile int *>(slot + 5);
        if (t == -1) {
            t = atomicCAS(slot + 5, -1, e);
            if (t == -1) t = e;                // claimed here
        }
        own = own && t == e;
    }
    if (!own) {
        unsigned long long *g = A.global(e);
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const long long q = __float2ll_rn(f[c]);
            if (q != 0) atomicAdd(g + c, (unsigned long long)q);
        }
        return;
    }
    int old[4], q[4];
    const float big = fmaxf(fmaxf(fabsf(f[0]), fabsf(f[1])), fmaxf(fabsf(f[2]), fabsf(f[3])));
    if (big < 2147483648.0f) {
#pragma unroll
        for (int c = 0; c < 4; c++) {
            q[c] = __float2int_rn(f[c]);
            old[c] = atomicAdd(slot + c, q[c]);
        }
        // opacity: the sign of the 32-bit add's wrap is the carry into the high word
        int over[4];
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const int now = (int)((unsigned)old[c] + (unsigned)q[c]);
            over[c] = (old[c] ^ now) & (q[c] ^ now);       // sign bit: the add wrapped
        }
        if ((over[0] | over[1] | over[2] | over[3]) < 0) {
            unsigned long long *g = A.global(e);
#pragma unroll
            for (int c = 0; c < 3; c++)
                if (over[c] < 0) atomicAdd(g + c, q[c] > 0 ? 1ull << 32 : ~0ull << 32);
            if (over[3] < 0) atomicAdd(slot + 4, q[3] > 0 ? 1 : -1);
        }
        return;
    }
#pragma unroll
    for (int c = 0; c < 4; c++) {
        // the value as a signed low word and the multiple of 2^32 beside it
        const long long v = __float2ll_rn(f[c]);
        const int lo = (int)(unsigned)v;
        long long hi = (v - lo) >> 32;
        const int o = atomicAdd(slot + c, lo), now = (int)((unsigned)o + (unsigned)lo);
        if (((o ^ now) & (lo ^ now)) < 0) hi += lo > 0 ? 1 : -1;
        if (hi == 0) continue;
        if (c == 3) atomicAdd(slot + 4, (int)hi);
        else atomicAdd(A.global(e) + c, (unsigned long long)hi << 32);
    }
}

// Sum of v (N values) over the lanes of this lane's group (lanes with the same key), in a
// fixed pairwise-tree order over the group's lanes sorted by lane id; the sum
// ends in the group's lowest lane (rank 0). Deterministic for a given key set.
template <int N>
__device__ __forceinline__ void group_sum(unsigned peers, float (&v)[N]) {
    const int lane = threadIdx.x & 31;
    const int cnt = __popc(peers);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    // the lane of rank + s, by pointer jumping: first the next member above
    // this lane (or this lane itself when there is none)
    const unsigned above = peers & ~((2u << lane) - 1u);
    int nxt = above ? __ffs(above) - 1 : lane;
#pragma unroll 1
    for (int s = 1; __any_sync(0xffffffffu, s < cnt); s <<= 1) {
        const bool take = (rank % (2 * s)) == 0 && rank + s < cnt;
        const int src = take ? nxt : lane;
#pragma unroll
        for (int c = 0; c < N; c++) {
            const float o = __shfl_sync(0xffffffffu, v[c], src);
            if (take) v[c] += o;
        }
        nxt = __shfl_sync(0xffffffffu, nxt, nxt);          // rank + 2s
    }
}

// d a' / d a = r (1 - a)^(r - 1) for the step ratio r of mode RM, with
// x = 1 - a >= 1e-6: r = 1/2 and 1/4 as reciprocal square roots, else
// through log2 / exp2.
template <int RM>
__device__ __forceinline__ float dalpha_factor(float x, float ratio, int rmode) {
    const int m = RM >= 0 ? RM : rmode;
    if (m == 1) return 0.5f * rsqrtf(x);
    if (m == 2) {
        const float q = rsqrtf(x);
        return 0.25f * q * sqrtf(q);
    }
    return ratio * exp2f((ratio - 1.0f) * __log2f(x));
}

// The gradient of one warp's 8 x 4 pixels: pixel (x, y) of view `view` per
// lane, with dL/dI times gscale. scatter(i, v, leader) receives each sample's
// sums per table cell i (column + row * row_stride), in the lanes marked
// leader, for the whole warp at once.
// CUBIC: cubic B-spline reconstruction (value and analytic gradient) instead
// of trilinear values and central differences; the table scatter is the same.
// TF2: a 2-D table over (value, gradient magnitude) in global memory; each
// sample scatters into the four entries of its bilinear cell.
template <int ST, bool SHADE, int RM, bool CUBIC, bool TF2, typename Scatter>
__device__ __forceinline__ void gradient_tile(const AdjointArgs &A, const float4 *s_tf, const CamRec &cam, int view,
                                              int x, int y, float gscale, int row_stride, Scatter scatter) {
    const MarchArgs &a = A.m;
    const int K = a.tf.K;
    constexpr bool GRAD = SHADE || TF2;
    constexpr int NV = TF2 ? 16 : 8;                  // contributions per sample
    const int lane = threadIdx.x & 31;
    const bool inimg = x < cam.W && y < cam.H;
    Ray R;
    bool hit = inimg && setup_ray(cam, a.vol, a.p.step_vox, x, y, R);
    float4 g = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (hit) g = A.dimg[((size_t)view * cam.H + y) * cam.W + x];
    const bool has_g = hit && (g.x != 0.0f || g.y != 0.0f || g.z != 0.0f || g.w != 0.0f);
    if (TF2) g = make_float4(g.x * gscale, g.y * gscale, g.z * gscale, g.w * gscale);
    // pass 1: the forward march, with exact empty-space skipping over empty
    // bricks, octants and 4^3 sub-blocks (identical result), for C_final,
    // T_final and the sample count n up to termination
    float Cf0 = 0.0f, Cf1 = 0.0f, Cf2 = 0.0f, Tf = 1.0f;
    int n = 0;
    const bool given = A.fimg != nullptr;
    if (given) {
        if (has_g) {
            const float4 f = A.fimg[((size_t)view * cam.H + y) * cam.W + x];
            Cf0 = f.x;
            Cf1 = f.y;
            Cf2 = f.z;
            Tf = 1.0f - f.w;
            n = R.nsamp;
        }
    } else if (has_g) {
        int k = 0;
        while (k < R.nsamp) {
            float p[3];
            position_at(R, sample_t(R, k), p);
            Cell c;
            cell_of(a.vol, p, c);
            const int s = empty_level(a, a.lvl, c);
            if (s) {
                k = jump_block(R, a.vol, c, k, s);
                continue;
            }
            float4 e = eval_sample_x<ST, (SHADE ? kShade : 0) | (CUBIC ? kCubic : 0) | (TF2 ? kTF2 : 0), RM>(
                a.vol, a.p, s_tf, a.tf,
                                                                                          R.dir, c, a.p.rmode,
                                                               a.p.ratio);
            composite_add(e, Cf0, Cf1, Cf2, Tf);
            k++;
            if ((1.0f - Tf) >= a.p.term) break;
        }
        n = min(k, R.nsamp);
    }
    // pass 2: every sample again (an empty brick still has a gradient), the
    // prefix C_{<=k} rebuilt, one gradient contribution per sample; lanes that
    // hit the same table entries are summed first, then the group's leader
    // adds the sums to its warp's FP32 copy (or, for a large table, one 64-bit
    // fixed-point atomic per entry and channel)
    float C0 = 0.0f, C1 = 0.0f, C2 = 0.0f, T = 1.0f;
    for (int k = 0; __any_sync(0xffffffffu, k < n); k++) {
        const bool active = k < n;
        int i = -1;
        float v[NV];
#pragma unroll
        for (int c = 0; c < NV; c++) v[c] = 0.0f;
        if (active) {
            float p[3], gr[3], val;
            position_at(R, sample_t(R, k), p);
            Cell c;
            cell_of(a.vol, p, c);
            if constexpr (CUBIC && GRAD) val = bspline_grad<ST>(a.vol, c, gr);
            else if constexpr (CUBIC) val = bspline<ST>(a.vol, c);
            else if constexpr (GRAD) val = value_grad<ST>(a.vol, c, gr);
            else val = trilinear<ST>(a.vol, c);
            float w, wb = 0.0f;
            float4 e;
            if (TF2) {
                int j;
                e = classify2_at(a.tf, tf_coord<ST>(val, a.tf.ucoef), tf2_row_coord(a.tf, gr), i, j, w, wb,
                                 RC_DBG_ERR(a.vol));
                i += j * row_stride;                  // entry (i, j) of the M x K table
            } else {
                e = classify(s_tf, K, tf_coord<ST>(val, a.tf.ucoef), &i, &w, RC_DBG_ERR(a.vol));
            }
            float ap = correct_alpha<RM>(e.w, a.p.rmode, a.p.ratio);
            float r = e.x, gg = e.y, b = e.z;
            float d0 = 1.0f, d1 = 1.0f, d2 = 1.0f;
            if (SHADE) {
                float sf, spec;
                shade_factor(a.p, a.vol, gr, R.dir, sf, spec);
                float u0 = __fmaf_rn(r, sf, spec), u1 = __fmaf_rn(gg, sf, spec), u2 = __fmaf_rn(b, sf, spec);
                d0 = u0 < 1.0f ? sf : 0.0f;
                d1 = u1 < 1.0f ? sf : 0.0f;
                d2 = u2 < 1.0f ? sf : 0.0f;
                r = fminf(1.0f, u0);
                gg = fminf(1.0f, u1);
                b = fminf(1.0f, u2);
            }
            const float Tk = T;
            float ta = T * ap;
            C0 = __fmaf_rn(ta, r, C0);
            C1 = __fmaf_rn(ta, gg, C1);
            C2 = __fmaf_rn(ta, b, C2);
            T = T * (1.0f - ap);
            if (given && (1.0f - T) >= a.p.term) n = k + 1;        // the forward stopped after this sample
            const float om = 1.0f - ap;
            const float inv = om > 0.0f ? 1.0f / om : 0.0f;
            float dap = g.x * (Tk * r - (Cf0 - C0) * inv) + g.y * (Tk * gg - (Cf1 - C1) * inv) +
                        g.z * (Tk * b - (Cf2 - C2) * inv) + g.w * (Tk - (T - Tf) * inv);
            float ac = fminf(e.w, 1.0f - 1e-6f);
            const int m = RM >= 0 ? RM : a.p.rmode;
            const float dal = m == 0 ? dap : dap * dalpha_factor<RM>(1.0f - ac, a.p.ratio, m);
            float dr = g.x * ta * d0, dg = g.y * ta * d1, db = g.z * ta * d2;
            // bilinear weights of the cell's entries: (i, j), (i + 1, j), then
            // the next row (i, j + 1), (i + 1, j + 1) for a 2-D table
            const float w0 = 1.0f - w;
            const float wr[4] = {w0 * (1.0f - wb), w * (1.0f - wb), w0 * wb, w * wb};
#pragma unroll
            for (int q = 0; q < NV / 4; q++) {
                v[4 * q + 0] = wr[q] * dr;
                v[4 * q + 1] = wr[q] * dg;
                v[4 * q + 2] = wr[q] * db;
                v[4 * q + 3] = wr[q] * dal;
            }
        }
        const unsigned peers = __match_any_sync(0xffffffffu, active ? i : -1 - lane);
        group_sum<NV>(peers, v);
        scatter(i, v, active && (peers & ((1u << lane) - 1u)) == 0u);
    }
}

// 1-D tables: the table and the accumulators in shared memory, one CTA per
// 16 x 8 pixels.
template <int ST, bool SHADE, int RM, bool CUBIC>
__global__ void __launch_bounds__(32 * kAdjWarps) adjoint_kernel(const AdjointArgs A, const float *absmax) {
    const MarchArgs &a = A.m;
    const int K = a.tf.K;
    const bool wacc = warp_acc(K, CUBIC, A.fimg != nullptr);   // per-warp FP32 accumulators
    extern __shared__ float4 smem[];
    float4 *s_tf = smem;
    unsigned long long *s_acc = reinterpret_cast<unsigned long long *>(smem + K);
    float4 *s_wacc = smem + K;                        // [warp][entry], tables of <= kWarpAccK entries
    load_tf(a.tf, s_tf);
    if (wacc) {
        for (int e = threadIdx.x; e < kAdjWarps * K; e += blockDim.x) s_wacc[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    } else {
        for (int e = threadIdx.x; e < 4 * K; e += blockDim.x) s_acc[e] = 0ull;
    }
    __syncthreads();
    const float scale = fixed_scale(absmax);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const CamRec cam = a.cams ? a.cams[blockIdx.z] : a.cam;
    float4 *wa = s_wacc + warp * K;
    gradient_tile<ST, SHADE, RM, CUBIC, false>(
        A, s_tf, cam, blockIdx.z, blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7),
        blockIdx.y * 8 + (warp >> 1) * 4 + (lane >> 3), 1.0f, 0, [&](int i, const float (&v)[8], bool leader) {
            if (wacc) {
                // the leaders hold distinct entries i, but the i + 1 of one group
                // may be the i of another: entry i first, then (after the warp
                // barrier) entry i + 1, each a plain read-modify-write of a slot
                // no other leader touches in that phase. The barrier before the
                // first phase orders it after the previous sample's second phase.
                __syncwarp();
                if (leader) {
                    float4 q = wa[i];
                    q.x += v[0]; q.y += v[1]; q.z += v[2]; q.w += v[3];
                    wa[i] = q;
                }
                __syncwarp();
                if (leader) {
                    float4 q = wa[i + 1];
                    q.x += v[4]; q.y += v[5]; q.z += v[6]; q.w += v[7];
                    wa[i + 1] = q;
                }
            } else if (leader) {
#pragma unroll
                for (int c = 0; c < 8; c++) acc_add(s_acc, 4 * i + c, v[c], scale);
            }
        });
    __syncthreads();
    unsigned long long *g_acc = reinterpret_cast<unsigned long long *>(A.acc);
    if (wacc) {
        // the warps' copies summed in warp order, then one fixed-point add
        const float *w = reinterpret_cast<const float *>(s_wacc);
        for (int e = threadIdx.x; e < 4 * K; e += blockDim.x) {
            float sum = w[e];
#pragma unroll
            for (int wi = 1; wi < kAdjWarps; wi++) sum += w[wi * 4 * K + e];
            const long long q = __float2ll_rn(sum * scale);
            if (q != 0) atomicAdd(g_acc + e, (unsigned long long)q);
        }
    } else {
        for (int e = threadIdx.x; e < 4 * K; e += blockDim.x) {
            unsigned long long v = s_acc[e];
            if (v != 0ull) atomicAdd(g_acc + e, v);
        }
    }
}

// 2-D tables: persistent CTAs (one per SM) whose groups of warps take chunks of
// 16 x 16 pixels from a queue (A.next, zero at launch) until it is empty.
template <int ST, bool SHADE, bool CUBIC>
__global__ void __launch_bounds__(32 * kGroupWarps * group_count(CUBIC), 1)
adjoint2_kernel(const AdjointArgs A, const float *absmax, int slots, int tagged, int chunks_x, int chunks_y, int nchunks) {
    const MarchArgs &a = A.m;
    extern __shared__ float4 smem[];
    __shared__ int s_chunk[group_count(CUBIC)];
    const int K = a.tf.K;
    Acc2 acc;
    acc.words = reinterpret_cast<int *>(smem);
    acc.tagged = tagged;
    acc.K = K;
    acc.row = tagged ? K : K + kRowSkew;
    acc.g = reinterpret_cast<unsigned long long *>(A.acc);
    const float scale = fixed_scale(absmax);
    const int per_slot = tagged ? kTagWords : kSlotWords;
    for (int e = threadIdx.x; e < per_slot * slots; e += blockDim.x)
        acc.words[e] = tagged && e % kTagWords == 5 ? -1 : 0;
    __syncthreads();
    constexpr int kGroup = 32 * kGroupWarps;
    const int group = threadIdx.x / kGroup, t = threadIdx.x % kGroup, warp = t >> 5, lane = t & 31;
    for (;;) {
        if (t == 0) s_chunk[group] = (int)min(atomicAdd(A.next, 1u), (unsigned)nchunks);
        asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kGroup) : "memory");
        const int chunk = s_chunk[group];
        asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "n"(kGroup) : "memory");
        if (chunk >= nchunks) break;
        const int view = chunk / (chunks_x * chunks_y), in_view = chunk % (chunks_x * chunks_y);
        const CamRec cam = a.cams ? a.cams[view] : a.cam;
        gradient_tile<ST, SHADE, -1, CUBIC, true>(
            A, nullptr, cam, view, (in_view % chunks_x) * 16 + (warp & 1) * 8 + (lane & 7),
            (in_view / chunks_x) * 2 * kGroupWarps + (warp >> 1) * 4 + (lane >> 3), scale, acc.row,
            [&](int i, const float (&v)[16], bool leader) {
                if (!leader) return;
                acc2_add4(acc, i, v);
                acc2_add4(acc, i + 1, v + 4);
                acc2_add4(acc, i + acc.row, v + 8);
                acc2_add4(acc, i + acc.row + 1, v + 12);
            });
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 4 * slots; e += blockDim.x) {
        const int s = e >> 2, *slot = acc.words + per_slot * s;
        const int entry = tagged ? slot[5] : s % acc.row < K ? s : -1;
        const long long v = (long long)slot[e & 3] + ((e & 3) == 3 ? (long long)slot[4] << 32 : 0ll);
        if (entry >= 0 && v != 0) atomicAdd(acc.global(entry) + (e & 3), (unsigned long long)v);
    }
}

__global__ void finalize_kernel(const long long *acc, int n, const float *absmax, float *out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double scale = (double)fixed_scale(absmax);
    out[i] = (float)((double)acc[i] / scale);
}

template <bool CUBIC, typename Kern>
static cudaError_t launch_adj(Kern kern, const AdjointArgs &a, int nviews, const float *absmax, cudaStream_t s) {
    // the table and its accumulators in shared memory (per warp in FP32 where
    // warp_acc says so, else per CTA in 64-bit fixed point)
    const int K = a.m.tf.K;
    const size_t smem = warp_acc(K, CUBIC, a.fimg != nullptr) ? (size_t)K * (1 + kAdjWarps) * sizeof(float4)
                                                              : (size_t)K * (sizeof(float4) + 4 * sizeof(long long));
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((a.m.cam.W + 15) / 16, (a.m.cam.H + 7) / 8, nviews);
    kern<<<grid, 32 * kAdjWarps, smem, s>>>(a, absmax);
    return cudaGetLastError();
}

template <bool CUBIC, typename Kern>
static cudaError_t launch_adj2(Kern kern, const AdjointArgs &a, int nviews, const float *absmax, cudaStream_t s) {
    const long long direct = (long long)(a.m.tf.K + kRowSkew) * a.m.tf.M;
    const bool tagged = direct > kDirectSlots;
    const int slots = tagged ? kTagSlots : (int)direct;
    const size_t smem = (size_t)slots * (tagged ? kTagWords : kSlotWords) * sizeof(int);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(a.next, 0, sizeof(unsigned), s)) != cudaSuccess) return e;
    const int cx = (a.m.cam.W + 15) / 16, cy = (a.m.cam.H + 2 * kGroupWarps - 1) / (2 * kGroupWarps);
    const int nchunks = cx * cy * nviews;       // at most 2^31 pixels in all: fewer than 2^28
    const int grid = persistent_ctas(nchunks, sms);
    kern<<<grid, 32 * kGroupWarps * group_count(CUBIC), smem, s>>>(a, absmax, slots, tagged ? 1 : 0, cx, cy, nchunks);
    return cudaGetLastError();
}

// The instance for the volume's storage, shading, opacity-correction mode RM
// and reconstruction filter.
template <int RM, bool CUBIC>
static cudaError_t launch_adj_rm(const AdjointArgs &a, int nviews, const float *absmax, cudaStream_t s) {
    if (a.m.p.shade)
        return by_storage<!CUBIC>(a.m.vol, [&](auto st) {
            return launch_adj<CUBIC>(adjoint_kernel<decltype(st)::value, true, RM, CUBIC>, a, nviews, absmax, s);
        });
    return by_storage<false>(a.m.vol, [&](auto st) {
        return launch_adj<CUBIC>(adjoint_kernel<decltype(st)::value, false, RM, CUBIC>, a, nviews, absmax, s);
    });
}

template <bool CUBIC>
static cudaError_t launch_adj_tf2(const AdjointArgs &a, int nviews, const float *absmax, cudaStream_t s) {
    return by_storage<!CUBIC>(a.m.vol, [&](auto st) {
        constexpr int ST = decltype(st)::value;
        return a.m.p.shade ? launch_adj2<CUBIC>(adjoint2_kernel<ST, true, CUBIC>, a, nviews, absmax, s)
                           : launch_adj2<CUBIC>(adjoint2_kernel<ST, false, CUBIC>, a, nviews, absmax, s);
    });
}

// 1-D tables: one instance per opacity-correction mode; 2-D tables: the mode
// read at run time (the scatter dominates there).
template <bool CUBIC>
static cudaError_t launch_adj_filter(const AdjointArgs &a, int nviews, const float *absmax, cudaStream_t s) {
    if (a.m.tf.M >= 2) return launch_adj_tf2<CUBIC>(a, nviews, absmax, s);
    switch (a.m.p.rmode) {
        case 0: return launch_adj_rm<0, CUBIC>(a, nviews, absmax, s);
        case 1: return launch_adj_rm<1, CUBIC>(a, nviews, absmax, s);
        case 2: return launch_adj_rm<2, CUBIC>(a, nviews, absmax, s);
        default: return launch_adj_rm<3, CUBIC>(a, nviews, absmax, s);
    }
}

// acc must hold 4 K max(M, 1) long longs (one per table entry and channel)
// followed by one float (the |dL/dI| maximum) and one unsigned (the queue of a
// 2-D table's launch). With a.m.cams, nviews views
// (grid.z), dimg view-major; the gradient is the sum over the views.
cudaError_t launch_adjoint(AdjointArgs a, int nviews, float *dL_dtf, cudaStream_t s) {
    const int nent = a.m.tf.K * (a.m.tf.M >= 2 ? a.m.tf.M : 1);
    a.next = reinterpret_cast<unsigned *>(a.acc + 4 * (size_t)nent) + 1;
    float *absmax = reinterpret_cast<float *>(a.acc + 4 * (size_t)nent);
    cudaError_t e = launch_absmax(reinterpret_cast<const float *>(a.dimg),
                                  (long long)nviews * a.m.cam.W * a.m.cam.H * 4, absmax, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(a.acc, 0, sizeof(long long) * 4 * (size_t)nent, s);
    if (e != cudaSuccess) return e;
    e = a.m.p.filter == RC_FILTER_BSPLINE ? launch_adj_filter<true>(a, nviews, absmax, s)
                                          : launch_adj_filter<false>(a, nviews, absmax, s);
    if (e != cudaSuccess) return e;
    finalize_kernel<<<(4 * nent + 255) / 256, 256, 0, s>>>(a.acc, 4 * nent, absmax, dL_dtf);
    return cudaGetLastError();
}

}  // namespace rc
