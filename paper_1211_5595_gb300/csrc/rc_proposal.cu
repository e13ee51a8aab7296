// Learned sampling proposal: opacity profiles of the plain march (training
// targets), the per-ray feature encoder, a 112-64-64-64-40 BF16 network on the
// fifth-generation tensor cores (tcgen05 MMA, FP32 accumulators in tensor
// memory, one M = 128 tile of rays per CTA), its SIMT training kernels
// (deterministic gradient reduction, Adam), and the importance-sampled march
// with fallback to the plain march.
//
// The paper has no learned part: the proposal replaces the evenly spaced
// samples of Sec. 4.1 by 64 samples drawn where the network expects opacity,
// and keeps the compositing of Sec. 4.2 (Eq. 3-4) with each sample's opacity
// corrected to the length of the segment it stands for.
#include <cuda_bf16.h>

#include "rc_device.cuh"
#include "rc_tcgen05.cuh"

namespace rc {


__device__ __forceinline__ void tile_pixel(int &x, int &y) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    x = blockIdx.x * 16 + (warp & 1) * 8 + (lane & 7);
    y = blockIdx.y * 8 + (warp >> 1) * 4 + (lane >> 3);
}

// ---------------------------------------------------------------------------
// opacity profiles: 512 samples at the centres of 512 equal segments of the
// chord, no termination; weights T_k a'_k summed 16 per bin; T at the end
// ---------------------------------------------------------------------------
// Four lanes per ray: lane j evaluates samples 4i + j of a bin, then the group
// runs the bin's recurrence in sample order from shuffles (an empty sample has
// opacity exactly 0 and changes nothing, so the values are those of one lane
// marching alone). A ray's 512 samples are a serial chain and only the rays that
// meet the volume have one, so one lane per ray left the GPU waiting on latency
// (256x256x180, 256^2 view 240 us, 512^2 257, 1024^2 602; now 69, 133 and 399).
// When a whole bin is empty, the bins up to the exit of the last sample's block
// are too. Rows are staged in shared memory and written 132 contiguous bytes
// per ray.
constexpr int kProfLanes = 4, kProfTileX = 8, kProfTileY = 4;      // pixels per CTA of 4 warps (4 x 2 per warp)

__device__ __forceinline__ int jump_block_grid(const Ray &R, const VolDev &v, const Cell &c, int j, int s, float ta,
                                               float seg, int n);

template <int ST>
__global__ void __launch_bounds__(128) profiles_kernel(const MarchArgs a, float *out) {
    extern __shared__ float4 s_tf[];
    __shared__ float s_row[4][32 / kProfLanes][kOutUsed];
    load_tf(a.tf, s_tf);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, j = lane % kProfLanes, ray = lane / kProfLanes,
              first = lane - j;
    // more tile rows than the grid's y limit take further turns
    for (int tile_y = blockIdx.y; tile_y * kProfTileY < a.cam.H; tile_y += gridDim.y) {
        __syncwarp();
        const int x0 = blockIdx.x * kProfTileX + (warp & 1) * 4, y0 = tile_y * kProfTileY + (warp >> 1) * 2;
        const int x = x0 + (ray & 3), y = y0 + (ray >> 2);
        Ray R;
        const bool hit = x < a.cam.W && y < a.cam.H && setup_ray(a.cam, a.vol, a.p.step_vox, x, y, R);
        float *row = s_row[warp][ray];
        for (int b = j; b < kBins; b += kProfLanes) row[b] = 0.0f;
        __syncwarp();
        float T = 1.0f;
        if (__any_sync(0xffffffffu, hit)) {
            constexpr int kPerBin = kProfSamples / kBins, kPerLane = kPerBin / kProfLanes;
            const float delta = hit ? __fdiv_rn(__fsub_rn(R.tf, R.tn), (float)kProfSamples) : 0.0f;
            const float ratio = __fdiv_rn(delta, a.vol.smin);
            int b = hit ? 0 : kBins;
            while (__any_sync(0xffffffffu, b < kBins)) {
                const bool on = b < kBins;
                float al[kPerLane];
                Cell c;
                int s = 0;
                unsigned some = 0;
    #pragma unroll
                for (int i = 0; i < kPerLane; i++) {
                    al[i] = 0.0f;
                    if (on) {
                        float p[3];
                        position_at(R, __fmaf_rn((float)(b * kPerBin + i * kProfLanes + j) + 0.5f, delta, R.tn), p);
                        cell_of(a.vol, p, c);
                        s = a.p.skip ? empty_level(a, a.lvl, c) : 0;
                        if (!s) {
                            al[i] = eval_sample<ST, false>(a.vol, a.p, s_tf, a.tf.K, a.tf.ucoef, R.dir, c, 3, ratio).w;
                            some = 1;
                        }
                    }
                }
                float acc = 0.0f;
                if (__any_sync(0xffffffffu, some)) {
    #pragma unroll
                    for (int k = 0; k < kPerBin; k++) {
                        const float w = __shfl_sync(0xffffffffu, al[k / kProfLanes], first + k % kProfLanes);
                        acc = __fmaf_rn(T, w, acc);
                        T = T * (1.0f - w);
                    }
                }
                const unsigned in_group = (__ballot_sync(0xffffffffu, some) >> first) & ((1u << kProfLanes) - 1u);
                int next = b + 1;
                if (on && in_group == 0) {
                    // the sample after the block of each lane's last sample; the
                    // bins wholly before the last lane's stay zero
                    const int k = jump_block_grid(R, a.vol, c, b * kPerBin + kPerBin - kProfLanes + j, s, R.tn, delta, kProfSamples);
                    next = max(next, k / kPerBin);
                }
                next = __shfl_sync(0xffffffffu, next, first + kProfLanes - 1);
                if (on) {
                    if (j == 0 && in_group) row[b] = acc;
                    b = next;
                }
            }
        }
        if (j == 0) row[kBins] = T;
        __syncwarp();
        // two image rows of up to four rays, contiguous in the output
        const int rays = min(4, a.cam.W - x0);
        for (int r = 0; r < 2 && y0 + r < a.cam.H; r++) {
            float *o = out + ((size_t)(y0 + r) * a.cam.W + x0) * kOutUsed;
            const float *src = s_row[warp][4 * r];
            for (int e = lane; e < rays * kOutUsed; e += 32) o[e] = src[e];
        }
    }
}

// ---------------------------------------------------------------------------
// features: entry point (normalised to the box) and world direction, their
// sin/cos encodings at 6 octaves, 32 occupancy bits along the chord, 2 zeros
// ---------------------------------------------------------------------------
// A ray in units of cell-bricks (positions / 16), for occupancy lookups: scaling
// by a power of two is exact, so the truncated coordinate is the base cell's
// brick (min(i, n - 2) >> 4 = min(i >> 4, cb - 1)) without the shifts.
struct BrickRay {
    float o[3], d[3];
    __device__ __forceinline__ explicit BrickRay(const Ray &R) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            o[a] = R.o[a] * 0.0625f;
            d[a] = R.d[a] * 0.0625f;
        }
    }
    __device__ __forceinline__ bool occupied(const VolDev &v, const uint8_t *occ, float t) const {
        int b[3];
#pragma unroll
        for (int a = 0; a < 3; a++) b[a] = (int)min(__float2uint_rz(__fmaf_rn(t, d[a], o[a])), (unsigned)(v.cb[a] - 1));
        int at = (b[2] * v.cb[1] + b[1]) * v.cb[0] + b[0];
#ifdef RC_DEBUG
        at = dbg_index(at + v.dbg_poison, v.cb[0] * v.cb[1] * v.cb[2], v.dbg_err, kSiteBrick);
#endif
        return __ldg(occ + at) != 0;
    }
};

// Emits the 112 features in 14 chunks of 8 (emit(chunk, v) in chunk order) and
// returns the occupancy bits at the bin centres as a mask (bit b = bin b).
// Feature order: 0-5 entry point and direction; 6 + 12c + 2j and 7 + 12c + 2j
// sin and cos of pi 2^j x_c; 78 + b occupancy of bin b's centre; 110-111 zero.
template <typename Emit>
__device__ __forceinline__ uint32_t ray_features(const VolDev &v, const uint8_t *occ, const Ray &R, bool hit,
                                                 Emit emit) {
    float buf[8];
    int fill = 0, chunk = 0;
    auto put = [&](float x) {
        buf[fill++] = x;
        if (fill == 8) {
            emit(chunk++, buf);
            fill = 0;
        }
    };
    if (!hit) {
#pragma unroll
        for (int i = 0; i < kFeat; i++) put(0.0f);
        return 0u;
    }
    float xs[6];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        xs[c] = __fdiv_rn(__fmaf_rn(R.tn, R.d[c], R.o[c]), (float)(v.n[c] - 1));
        xs[3 + c] = R.dir[c];
    }
#pragma unroll
    for (int c = 0; c < 6; c++) put(xs[c]);
    // sin and cos of pi 2^j x for j = 0 and 3 directly; j = 1, 2 and 4, 5 by
    // angle doubling, sin 2a = 2 sin a cos a, cos 2a = (cos a - sin a)(cos a + sin a)
    // (two doublings keep the error below 1e-6)
#pragma unroll
    for (int c = 0; c < 6; c++) {
        float s, co;
#pragma unroll
        for (int j = 0; j < 6; j++) {
            if (j == 0 || j == 3) {
                sincospif(j == 0 ? xs[c] : 8.0f * xs[c], &s, &co);
            } else {
                const float s2 = 2.0f * s * co;
                co = (co - s) * (co + s);
                s = s2;
            }
            put(s);
            put(co);
        }
    }
    const float bw = __fdiv_rn(__fsub_rn(R.tf, R.tn), (float)kBins);
    const BrickRay B(R);
    uint32_t mask = 0;
#pragma unroll
    for (int b = 0; b < kBins; b++) {
        const bool o = B.occupied(v, occ, __fmaf_rn((float)b + 0.5f, bw, R.tn));
        mask |= (uint32_t)o << b;
        put(o ? 1.0f : 0.0f);
    }
    put(0.0f);
    put(0.0f);
    return mask;
}

// One thread per ray. A warp's 32 rows are staged in shared memory (rows padded
// to 116 floats: eight lanes' 16-byte stores then hit eight different bank
// groups) and written as four runs of contiguous rows. VEC: the output is
// 16-byte aligned. Bound by the stores: 262144 rays (117 MB) 151 us with each
// thread writing its own row by 4-byte stores, 40 by 16-byte stores, 25
// staged (17 at the copy rate); 1048576 rays 768, 303 and 79 (69).
constexpr int kFeatRow = kFeat + 4;
constexpr int kFeatSmem = 4 * 32 * kFeatRow * (int)sizeof(float);

template <bool VEC>
__global__ void __launch_bounds__(128) features_kernel(const MarchArgs a, float *out) {
    extern __shared__ float4 s_tf[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float *rows = reinterpret_cast<float *>(s_tf) + warp * 32 * kFeatRow;
    int x, y;
    tile_pixel(x, y);
    Ray R;
    const bool hit = x < a.cam.W && y < a.cam.H && setup_ray(a.cam, a.vol, a.p.step_vox, x, y, R);
    float4 *mine = reinterpret_cast<float4 *>(rows + lane * kFeatRow);
    ray_features(a.vol, a.occ, R, hit, [&](int chunk, const float (&v)[8]) {
        mine[2 * chunk] = make_float4(v[0], v[1], v[2], v[3]);
        mine[2 * chunk + 1] = make_float4(v[4], v[5], v[6], v[7]);
    });
    __syncwarp();
    const int x0 = x - (lane & 7), y0 = y - (lane >> 3);
    const int n = min(8, a.cam.W - x0);                       // rays of a run (none when the tile is outside)
    for (int r = 0; r < 4 && y0 + r < a.cam.H; r++) {
        float *o = out + ((size_t)(y0 + r) * a.cam.W + x0) * kFeat;
        const float *src = rows + 8 * r * kFeatRow;
        if (VEC) {
            for (int e = lane; e < n * (kFeat / 4); e += 32)
                reinterpret_cast<float4 *>(o)[e] =
                    *reinterpret_cast<const float4 *>(src + (e / (kFeat / 4)) * kFeatRow + 4 * (e % (kFeat / 4)));
        } else {
            for (int e = lane; e < n * kFeat; e += 32) o[e] = src[(e / kFeat) * kFeatRow + e % kFeat];
        }
    }
}

// ---------------------------------------------------------------------------
// the network on the tensor cores: one M = 128 tile of rays per MMA
// ---------------------------------------------------------------------------
// A network CTA runs G independent groups of 128 threads, each on its own
// tiles of 128 rays with its own A operand, MMA barrier and 64 TMEM columns
// (TMEM lane = ray); the weights and biases are shared. The A operand holds a
// tile's features (128 x 112 BF16) and then, layer by layer, its hidden
// activations (128 x 64): every layer's MMA has completed before its output
// overwrites the operand it read. The camera-ray kernel runs one CTA of
// kCamGroups groups per SM (one copy of the weights, 209 KB of shared memory,
// 80 registers per thread; measured per 1024^2 view: 2 x 2 groups 0.146 ms,
// one CTA of 4 groups 0.149, of 5 groups 0.129, of 6 groups 0.121); the
// feature-matrix kernel two CTAs of kFeatGroups groups (its wide TMEM loads
// need more registers).
constexpr int kCamGroups = 6;
constexpr int kFeatGroups = 2;
constexpr int kGroupThreads = 128;
// TMEM columns of a CTA: 64 per group, allocated as a power of two
constexpr int tmem_cols(int groups) { return groups * 64 <= 128 ? 128 : groups * 64 <= 256 ? 256 : 512; }

template <int G>
struct NetSmem {
    uint8_t w[kUmmaBytes];                 // B operands of the four layers
    uint8_t a[G][128 * kFeat * 2];         // A operands
    float bias[3 * kHid + kN4];
    unsigned long long bar_w, bar_mma[G];
    uint32_t tmem;
};

struct NetLayer {
    unsigned b_off;                        // B operand offset in NetSmem::w
    int K, N;
};
__device__ __forceinline__ NetLayer net_layer(int l) {
    switch (l) {
        case 0: return NetLayer{kUmmaL1, kFeat, kHid};
        case 1: return NetLayer{kUmmaL2, kHid, kHid};
        case 2: return NetLayer{kUmmaL3, kHid, kHid};
        default: return NetLayer{kUmmaL4, kHid, kN4};
    }
}

// Barrier of one group (named barrier 1 + g, 128 threads); returns the AND of
// every thread's `ok`.
__device__ __forceinline__ bool group_sync_and(int g, bool ok) {
    uint32_t r;
    asm volatile(
        "{\n.reg .pred p, q;\nsetp.ne.u32 p, %1, 0;\nbar.red.and.pred q, %2, %3, p;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(r)
        : "r"((uint32_t)ok), "r"(1 + g), "r"(kGroupThreads)
        : "memory");
    return r != 0;
}

__device__ __forceinline__ void group_sync(int g) {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(kGroupThreads) : "memory");
}

// One layer, issued by one thread: D[128 x N] = A[128 x K] * W^T, K / 16 MMAs,
// then a commit that arrives on the group's MMA barrier when they are done.
template <int G>
__device__ __forceinline__ void issue_layer(const NetSmem<G> &S, int g, int l, uint32_t tmem_d, uint32_t bar) {
    const NetLayer L = net_layer(l);
    const uint32_t a0 = tc::smem_addr(S.a[g]), b0 = tc::smem_addr(S.w) + L.b_off;
    const uint32_t lbo_a = (128 / 8) * 128, lbo_b = (uint32_t)(L.N / 8) * 128;
    const uint32_t idesc = tc::idesc_bf16_f32(128, L.N);
    for (int ks = 0; ks < L.K / 16; ks++)
        tc::mma_bf16(tmem_d, tc::smem_desc(a0 + ks * 2 * lbo_a, lbo_a, 128),
                     tc::smem_desc(b0 + ks * 2 * lbo_b, lbo_b, 128), idesc, ks > 0);
    tc::commit(bar);
}

// Bias, ReLU and BF16 rounding of this thread's 64 hidden values, written as
// row `row` of the next layer's A operand (K = 64). Pairs of values: FP32x2
// bias add, one rounding to a BF16 pair, ReLU on the pair (max with +0 after
// rounding gives the same values as rounding after the ReLU).
__device__ __forceinline__ uint32_t bias_relu_bf16x2(float lo, float hi, float2 b) {
    uint64_t x, y, z;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(lo), "f"(hi));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(z) : "l"(x), "l"(y));
    float zl, zh;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(zl), "=f"(zh) : "l"(z));
    uint32_t p, r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p) : "f"(zh), "f"(zl));
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(p), "r"(0u));
    return r;
}

// Bias, ReLU and BF16 rounding of 16 hidden values (columns c .. c + 15),
// stored as two 16-byte chunks of row `row` of the next A operand.
__device__ __forceinline__ void store_hidden16(uint8_t *A, const float *v, const float2 *b2, int c, int row) {
#pragma unroll
    for (int j = 0; j < 16; j += 8) {
        uint4 q;
        uint32_t *w = reinterpret_cast<uint32_t *>(&q);
#pragma unroll
        for (int h = 0; h < 4; h++) w[h] = bias_relu_bf16x2(v[j + 2 * h], v[j + 2 * h + 1], b2[(c + j) / 2 + h]);
        *reinterpret_cast<uint4 *>(A + tc::core_offset(row, c + j, 128)) = q;
    }
}

// WIDE: the whole row in one TMEM load and wait (faster where the 64 live
// registers fit: the feature-matrix network and the training kernel); else
// four 16-column loads, each consumed before the next (the camera-ray
// network, at its register limit).
template <bool WIDE>
__device__ __forceinline__ void store_hidden(uint8_t *A, uint32_t taddr, const float *bias, int row) {
    const float2 *b2 = reinterpret_cast<const float2 *>(bias);
    if (WIDE) {
        float v[kHid];
        tc::tmem_ld64(taddr, v);
#pragma unroll
        for (int c = 0; c < kHid; c += 16) store_hidden16(A, v + c, b2, c, row);
    } else {
#pragma unroll
        for (int c = 0; c < kHid; c += 16) {
            float v[16];
            tc::tmem_ld16(taddr + c, v);
            store_hidden16(A, v, b2, c, row);
        }
    }
}

// Eight values as BF16 at (row, 8 * chunk .. 8 * chunk + 7) of an A operand:
// one 16-byte store (a warp's 32 rows fill 512 contiguous bytes).
__device__ __forceinline__ void store_chunk(uint8_t *A, int row, int chunk, const float (&v)[8]) {
    uint4 q;
    uint32_t *w = reinterpret_cast<uint32_t *>(&q);
#pragma unroll
    for (int h = 0; h < 4; h++) {
        __nv_bfloat162 b2 = __floats2bfloat162_rn(v[2 * h], v[2 * h + 1]);
        w[h] = *reinterpret_cast<uint32_t *>(&b2);
    }
    *reinterpret_cast<uint4 *>(A + tc::core_offset(row, 8 * chunk, 128)) = q;
}

// Network head: 32 logits -> PDF (softmax), logit 32 -> T^ (sigmoid).
template <bool WIDE>
__device__ __forceinline__ void net_head(uint32_t taddr, const float *bias, float (&pdf)[kBins], float &that) {
    // the head uses 33 of its 48 accumulator columns
    float z[kN4];
    if (WIDE) {
        float v[kHid];
        tc::tmem_ld64(taddr, v);
#pragma unroll
        for (int j = 0; j < kN4; j++) z[j] = v[j] + bias[j];
    } else {
#pragma unroll
        for (int c = 0; c < kN4; c += 16) {
            float v[16];
            tc::tmem_ld16(taddr + c, v);
#pragma unroll
            for (int j = 0; j < 16; j++) z[c + j] = v[j] + bias[c + j];
        }
    }
    float mx = z[0];
#pragma unroll
    for (int b = 1; b < kBins; b++) mx = fmaxf(mx, z[b]);
    // exponentials on the special-function unit (relative error ~2^-21,
    // far below the network's BF16 rounding)
    float sum = 0.0f;
#pragma unroll
    for (int b = 0; b < kBins; b++) {
        pdf[b] = __expf(z[b] - mx);
        sum += pdf[b];
    }
    const float inv = 1.0f / sum;
#pragma unroll
    for (int b = 0; b < kBins; b++) pdf[b] *= inv;
    that = 1.0f / (1.0f + __expf(-z[kBins]));
}

// Runs the four layers of group g on its A operand (the group's 128 threads
// call; thread t of the group is TMEM lane t). Returns false when a wait gave
// up; the caller then stops.
template <bool WIDE, int G>
__device__ __forceinline__ bool run_network(const TcNetArgs &A, NetSmem<G> &S, int g, uint32_t tmem, uint32_t bar,
                                            uint32_t &phase, float (&pdf)[kBins], float &that) {
    const int t = threadIdx.x - g * kGroupThreads;
    const uint32_t tmem_d = tmem + 64u * (uint32_t)g;
    const uint32_t taddr = tmem_d + ((uint32_t)(t & ~31) << 16);    // this warp's 32 lanes
#pragma unroll 1
    for (int l = 0; l < 4; l++) {
        tc::fence_async_smem();           // A written by ordinary stores -> visible to the MMA
        tc::fence_before();
        group_sync(g);
        tc::fence_after();
        if (t == 0 && A.issue_mma) issue_layer(S, g, l, tmem_d, bar);
        const bool ok = group_sync_and(g, tc::bar_wait(bar, phase, A.budget));
        if (!ok) return false;
        phase ^= 1u;
        tc::fence_after();
        if (l < 3) store_hidden<WIDE>(S.a[g], taddr, S.bias + l * kHid, t);
        else net_head<WIDE>(taddr, S.bias + 3 * kHid, pdf, that);
    }
    return true;
}

__device__ __forceinline__ void range_of(const MarchArgs &a, const Ray &R, const float (&pdf)[kBins], uint32_t centre,
                                         bool have_centre, int &b0, int &b1);

// FEAT: rays are rows of a feature matrix (outputs: the 33 network outputs);
// otherwise rays are the pixels of the cameras' views (outputs: the range
// record of each ray for the importance march).
template <bool FEAT, int G>
__global__ void __launch_bounds__(G * kGroupThreads) tc_net_kernel(const TcNetArgs A) {
    constexpr int kTmemCols = tmem_cols(G);
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    NetSmem<G> &S = *reinterpret_cast<NetSmem<G> *>(smem_raw);
    const int tid = threadIdx.x, g = tid / kGroupThreads, t = tid % kGroupThreads;
    const int warp = t >> 5, lane = t & 31;
    const uint32_t bar_w = tc::smem_addr(&S.bar_w), bar_m = tc::smem_addr(&S.bar_mma[g]);
    if (tid < 32) tc::tmem_alloc<kTmemCols>(tc::smem_addr(&S.tmem));
    if (tid == 0) {
        tc::bar_init(bar_w, 1);
        for (int i = 0; i < G; i++) tc::bar_init(tc::smem_addr(&S.bar_mma[i]), 1);
    }
    for (int i = tid; i < 3 * kHid + kN4; i += blockDim.x) {
        const int l = i / kHid, j = i % kHid;
        float b = 0.0f;
        if (l < 3) b = A.net.params[(l == 0 ? kOffB1 : l == 1 ? kOffB2 : kOffB3) + j];
        else if (j < kOut) b = A.net.params[kOffB4 + j];
        S.bias[i] = b;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = S.tmem;
    if (tid == 0) tc::bulk_g2s(tc::smem_addr(S.w), A.net.umma, kUmmaBytes, bar_w);
    bool ok = __syncthreads_and(tc::bar_wait(bar_w, 0, A.budget));
    if (!ok) tc::bar_wait(bar_w, 0, A.budget);      // the weight copy may still be in flight
    uint32_t phase = 0;
    bool mma_waited_out = false;
    uint8_t *Ag = S.a[g];
    const long long stride = (long long)gridDim.x * G;
#pragma unroll 1
    for (long long tile = (long long)blockIdx.x * G + g; ok && tile < A.ntiles; tile += stride) {
        Ray R;
        bool hit = false;
        long long out_idx = -1;
        uint32_t centre = 0;
        if (FEAT) {
            // the tile's rows are one contiguous block of 128 x 112 floats:
            // coalesced float4 loads, each 4 features of one row -> 8 bytes
            // of BF16 in the A operand
            const long long r0 = tile * 128;
            const long long valid = min((long long)128, A.n - r0);
            const float4 *src = reinterpret_cast<const float4 *>(A.feat + r0 * kFeat);
#pragma unroll 7
            for (int i = 0; i < 128 * kFeat / 4 / kGroupThreads; i++) {
                const int e = i * kGroupThreads + t;          // float4 index within the tile
                const int row = e / (kFeat / 4), k = (e % (kFeat / 4)) * 4;
                float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (row < valid) v = __ldg(src + e);
                __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
                uint2 q;
                q.x = *reinterpret_cast<uint32_t *>(&lo);
                q.y = *reinterpret_cast<uint32_t *>(&hi);
                *reinterpret_cast<uint2 *>(Ag + tc::core_offset(row, k, 128)) = q;
            }
        } else {
            const int per_view = A.tiles_x * A.tiles_y;
            const int view = (int)(tile / per_view), tl = (int)(tile % per_view);
            const CamRec &cam = A.m.cams[view];
            const int x = (tl % A.tiles_x) * 16 + (warp & 1) * 8 + (lane & 7);
            const int y = (tl / A.tiles_x) * 8 + (warp >> 1) * 4 + (lane >> 3);
            if (x < cam.W && y < cam.H) {
                hit = setup_ray(cam, A.m.vol, A.m.p.step_vox, x, y, R);
                out_idx = ((long long)view * cam.H + y) * cam.W + x;
            }
            // a tile none of whose rays meets the volume needs no network: the
            // importance march reads the records of rays that hit only (the
            // background around the volume: 61% of the tiles on a 1024^2 orbit
            // of the 256x256x180 phantom)
            if (group_sync_and(g, !hit)) continue;
            centre = ray_features(A.m.vol, A.m.occ, R, hit,
                                  [&](int chunk, const float (&v)[8]) { store_chunk(Ag, t, chunk, v); });
        }
        float pdf[kBins], that;
        ok = run_network<FEAT>(A, S, g, tmem, bar_m, phase, pdf, that);
        if (!ok) {
            mma_waited_out = true;
            break;
        }
        if (FEAT) {
            // stage the tile's 128 x 33 outputs in the A operand (its last
            // reader, the head layer's MMA, has completed), then store the
            // contiguous block with coalesced writes
            float *stage = reinterpret_cast<float *>(Ag);
#pragma unroll
            for (int b = 0; b < kBins; b++) stage[t * kOutUsed + b] = pdf[b];
            stage[t * kOutUsed + kBins] = that;
            group_sync(g);
            const long long r0 = tile * 128;
            const int valid = (int)min((long long)128, A.n - r0);
            float *o = A.net_out + r0 * kOutUsed;
            for (int e = t; e < valid * kOutUsed; e += kGroupThreads) o[e] = stage[e];
            group_sync(g);                  // before the next tile's features overwrite the stage
        } else if (out_idx >= 0) {
            if (A.pdf_out) {
                // the ray's PDF and T^ for the inverse-CDF march (32 + 1 floats)
                float4 *o = reinterpret_cast<float4 *>(A.pdf_out + out_idx * kBins);
#pragma unroll
                for (int b = 0; b < kBins; b += 4) o[b / 4] = make_float4(pdf[b], pdf[b + 1], pdf[b + 2], pdf[b + 3]);
                A.that_out[out_idx] = that;
            } else {
                int b0 = 0, b1 = kBins - 1;
                if (hit) range_of(A.m, R, pdf, centre, true, b0, b1);
                A.range[out_idx] = make_uint2((unsigned)b0 | ((unsigned)b1 << 8), __float_as_uint(that));
            }
        }
    }
    if (!ok) {
        if (t == 0) atomicOr(A.err, 1);
        if (mma_waited_out && A.issue_mma) tc::bar_wait(bar_m, phase, A.budget);   // MMAs may still be in flight
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid < 32) tc::tmem_free<kTmemCols>(tmem);
}

// ---------------------------------------------------------------------------
// importance-sampled march, with the plain march as fallback
// ---------------------------------------------------------------------------
// The plain march of one ray (the same arithmetic as composite_kernel).
template <int ST, bool SHADE>
__device__ __forceinline__ void plain_ray(const MarchArgs &a, const float4 *s_tf, const Ray &R, float &C0, float &C1,
                                          float &C2, float &T, unsigned &evald) {
    C0 = C1 = C2 = 0.0f;
    T = 1.0f;
    int k = 0;
    while (k < R.nsamp) {
        float p[3];
        position_at(R, sample_t(R, k), p);
        Cell c;
        cell_of(a.vol, p, c);
        if (a.p.skip) {
            const int s = empty_level(a, a.lvl, c);
            if (s) {
                k = jump_block(R, a.vol, c, k, s);
                continue;
            }
        }
        float4 e = eval_sample<ST, SHADE>(a.vol, a.p, s_tf, a.tf.K, a.tf.ucoef, R.dir, c, a.p.rmode, a.p.ratio);
        composite_add(e, C0, C1, C2, T);
        evald++;
        k++;
        if ((1.0f - T) >= a.p.term) break;
    }
}

// The PDF marks where the ray's contribution ends: b_end is one bin past the
// first bin >= b_start where its running sum reaches 1 - 1/64 (a margin for
// early predictions; at most 31, and 31 if never); b_start is the
// first bin whose start, centre or end lies in an occupied cell-brick (the
// whole chord when none does). FP32 operations as written.
__device__ __forceinline__ void range_of(const MarchArgs &a, const Ray &R, const float (&pdf)[kBins], uint32_t centre,
                                         bool have_centre, int &b0, int &b1) {
    const float bw = __fdiv_rn(__fsub_rn(R.tf, R.tn), (float)kBins);
    // bin b's start is boundary b, its end boundary b + 1 (both at
    // fma(k, bw, t_near)); its centre bit comes from the features when known
    b0 = -1;
    b1 = kBins - 1;
    const BrickRay B(R);
    bool start = B.occupied(a.vol, a.occ, R.tn);
    for (int b = 0; b < kBins && b0 < 0; b++) {
        const bool mid = have_centre ? ((centre >> b) & 1u) != 0
                                     : B.occupied(a.vol, a.occ, __fmaf_rn((float)b + 0.5f, bw, R.tn));
        if (start || mid) {
            b0 = b;
            break;
        }
        const bool end = B.occupied(a.vol, a.occ, __fmaf_rn((float)(b + 1), bw, R.tn));
        if (end) b0 = b;
        start = end;
    }
    if (b0 < 0) {
        b0 = 0;
        return;
    }
    float P = 0.0f;
    bool found = false;
#pragma unroll
    for (int b = 0; b < kBins; b++) {
        P = __fadd_rn(P, pdf[b]);
        if (!found && b >= b0 && P >= 1.0f - 1.0f / 64.0f) {
            b1 = min(b + 1, kBins - 1);
            found = true;
        }
    }
}

// nimp samples at the centres of nimp equal segments of [t_a, t_b] (start of
// bin b0 to end of bin b1), each with its opacity corrected to the segment.
// jump_block on the evenly spaced grid t_j = ta + (j + 0.5) seg, j < n, of a
// range march: the first sample index that may lie outside the empty block
// of 2^s cells around cell c (sample j is in it). The sample m just before
// the computed exit is verified to be in the same block, with its position
// computed exactly as the march computes it; positions are monotone in j
// along each axis, so every sample between j and m is in the block too.
// Falls back to j + 1 when the check fails.
__device__ __forceinline__ int jump_block_grid(const Ray &R, const VolDev &v, const Cell &c, int j, int s, float ta,
                                               float seg, int n) {
    float texit;
    if (!block_exit(R, v, c, s, texit)) return n;
    const float fm = floorf(__fsub_rn(__fdividef(texit - ta, seg), 0.5f));
    int m = fm >= (float)n ? n - 1 : (int)fm;
    if (m <= j) return j + 1;
#pragma unroll 1
    for (int tries = 0; tries < 2 && m > j; tries++, m--) {
        float p[3];
        position_at(R, __fmaf_rn((float)m + 0.5f, seg, ta), p);
        Cell cm;
        cell_of(v, p, cm);
        if (((cm.i[0] ^ c.i[0]) >> s) == 0 && ((cm.i[1] ^ c.i[1]) >> s) == 0 && ((cm.i[2] ^ c.i[2]) >> s) == 0)
            return m + 1;
    }
    return j + 1;
}

// JUMP: past an empty block in one step (jump_block_grid) instead of sample by
// sample; pays where a block spans several samples (measured on the bench
// orbit, ms per frame: 64 samples per ray 0.1735 -> 0.169, 128 samples
// 0.254 -> 0.228; 16 and 32 samples 3-4% slower, so chosen from 48 samples up)
template <int ST, bool SHADE, bool JUMP>
__device__ __forceinline__ void march_range(const ImportanceArgs &A, const float4 *s_tf, const Ray &R, int b0, int b1,
                                            float &C0, float &C1, float &C2, float &T, unsigned &evald) {
    const MarchArgs &a = A.m;
    const float bw = __fdiv_rn(__fsub_rn(R.tf, R.tn), (float)kBins);
    const float ta = b0 == 0 ? R.tn : __fmaf_rn((float)b0, bw, R.tn);
    const float tb = b1 == kBins - 1 ? R.tf : __fmaf_rn((float)(b1 + 1), bw, R.tn);
    const float seg = __fdiv_rn(__fsub_rn(tb, ta), (float)A.nimp);
    const float ratio = __fdiv_rn(seg, a.vol.smin);
    C0 = C1 = C2 = 0.0f;
    T = 1.0f;
    for (int j = 0; j < A.nimp;) {
        float p[3];
        position_at(R, __fmaf_rn((float)j + 0.5f, seg, ta), p);
        Cell c;
        cell_of(a.vol, p, c);
        if (a.p.skip) {          // opacity exactly 0: past the largest empty block around the sample
            const int s = empty_level(a, a.lvl, c);
            if (s) {
                j = JUMP ? jump_block_grid(R, a.vol, c, j, s, ta, seg, A.nimp) : j + 1;
                continue;
            }
        }
        float4 e = eval_sample<ST, SHADE>(a.vol, a.p, s_tf, a.tf.K, a.tf.ucoef, R.dir, c, 3, ratio);
        composite_add(e, C0, C1, C2, T);
        evald++;
        j++;
        if ((1.0f - T) >= a.p.term) break;
    }
}

// Stratified inverse-CDF samples of the mixture q_b = (1 - lambda) pdf_b +
// lambda / 32 over the bins of the chord: sample j where the mixture's CDF
// reaches (j + 0.5) / nimp of its total, standing for the stretch between the
// midpoints to its neighbours (t_near and t_far at the ends), with its
// opacity corrected to that length. FP32 operations as written (the bin
// search continues from the previous sample's bin: the targets increase).
// pdf: the ray's 32 bins, or null for the uniform density (lambda = 1).
template <int ST, bool SHADE>
__device__ __forceinline__ void march_invcdf(const ImportanceArgs &A, const float4 *s_tf, const Ray &R,
                                             const float *pdf, float &C0, float &C1, float &C2, float &T,
                                             unsigned &evald) {
    const MarchArgs &a = A.m;
    const float bw = __fdiv_rn(__fsub_rn(R.tf, R.tn), (float)kBins);
    const float wp = __fsub_rn(1.0f, A.lambda), wu = __fdiv_rn(A.lambda, (float)kBins);
    auto qb = [&](int b) { return __fmaf_rn(wp, pdf ? __ldg(pdf + b) : 0.0f, wu); };
    float total = 0.0f;
#pragma unroll 8
    for (int b = 0; b < kBins; b++) total = __fadd_rn(total, qb(b));
    int b = 0;
    float Qb = 0.0f, q = qb(0);
    float Qn = __fadd_rn(Qb, q);
    auto position = [&](int j) {
        const float y = __fmul_rn(__fdiv_rn((float)j + 0.5f, (float)A.nimp), total);
        while (b < kBins - 1 && !(Qn > y)) {
            b++;
            Qb = Qn;
            q = qb(b);
            Qn = __fadd_rn(Qb, q);
        }
        float f = 0.0f;
        if (q > 0.0f) f = fminf(fmaxf(__fdiv_rn(__fsub_rn(y, Qb), q), 0.0f), 1.0f);
        return __fmaf_rn(__fadd_rn((float)b, f), bw, R.tn);
    };
    C0 = C1 = C2 = 0.0f;
    T = 1.0f;
    float tj = position(0), m = R.tn;
    for (int j = 0; j < A.nimp; j++) {
        const bool last = j + 1 == A.nimp;
        const float tn1 = last ? R.tf : position(j + 1);
        const float mn = last ? R.tf : __fmul_rn(__fadd_rn(tj, tn1), 0.5f);
        const float len = __fsub_rn(mn, m);
        float p[3];
        position_at(R, tj, p);
        Cell c;
        cell_of(a.vol, p, c);
        if (!(a.p.skip && empty_level(a, a.lvl, c))) {                    // empty: opacity exactly 0
            const float ratio = __fdiv_rn(len, a.vol.smin);
            float4 e = eval_sample<ST, SHADE>(a.vol, a.p, s_tf, a.tf.K, a.tf.ucoef, R.dir, c, 3, ratio);
            composite_add(e, C0, C1, C2, T);
            evald++;
            if ((1.0f - T) >= a.p.term) break;
        }
        m = mn;
        tj = tn1;
    }
}

__device__ __forceinline__ void importance_stats(const MarchArgs &a, unsigned evald, unsigned fb, bool hit,
                                                 bool inimg) {
    unsigned e = __reduce_add_sync(0xffffffffu, evald), f = __reduce_add_sync(0xffffffffu, fb);
    unsigned h = __reduce_add_sync(0xffffffffu, hit ? 1u : 0u), n = __reduce_add_sync(0xffffffffu, inimg ? 1u : 0u);
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(a.stats + 0, (unsigned long long)f);     // fallback rays in the dense slot
        atomicAdd(a.stats + 1, (unsigned long long)e);
        atomicAdd(a.stats + 2, (unsigned long long)h);
        atomicAdd(a.stats + 3, (unsigned long long)n);
    }
}

// SRC = kSrcRecords: the sample range and T^ of each ray come from the
// network kernel's range records; kSrcRange: the range from the given per-ray
// PDF; kSrcInvCdf: inverse-CDF samples of the given PDF (or of the uniform
// density when A.pdf is null). Several views, grid.z = view, inputs
// view-major. Rays with |T_nimp - T^| > eps are re-marched by the plain march
// (never without a T^).
enum { kSrcRecords = 0, kSrcRange = 1, kSrcInvCdf = 2 };

template <int ST, bool SHADE, int SRC, bool JUMP = false>
__global__ void __launch_bounds__(128) importance_kernel(const ImportanceArgs A) {
    const MarchArgs &a = A.m;
    extern __shared__ float4 s_tf[];
    load_tf(a.tf, s_tf);
    __syncthreads();
    const CamRec cam = a.cams ? a.cams[blockIdx.z] : a.cam;
    const size_t view_off = (size_t)blockIdx.z * cam.W * cam.H;
    int x, y;
    tile_pixel(x, y);
    const bool inimg = x < cam.W && y < cam.H;
    Ray R;
    const bool hit = inimg && setup_ray(cam, a.vol, a.p.step_vox, x, y, R);
    const size_t pix = view_off + (size_t)y * cam.W + x;
    float C0 = 0.0f, C1 = 0.0f, C2 = 0.0f, T = 1.0f;
    unsigned evald = 0, fb = 0;
    if (hit) {
        float that;
        bool check = true;
        if (SRC == kSrcInvCdf) {
            march_invcdf<ST, SHADE>(A, s_tf, R, A.pdf ? A.pdf + pix * kBins : nullptr, C0, C1, C2, T, evald);
            check = A.that != nullptr;
            that = check ? A.that[pix] : 0.0f;
        } else {
            int b0, b1;
            if (SRC == kSrcRecords) {
                const uint2 rec = A.range[pix];
                b0 = min((int)(rec.x & 255u), kBins - 1);
                b1 = min(max((int)((rec.x >> 8) & 255u), b0), kBins - 1);
                that = __uint_as_float(rec.y);
            } else {
                float pdf[kBins];
#pragma unroll
                for (int b = 0; b < kBins; b++) pdf[b] = A.pdf[pix * kBins + b];
                that = A.that[pix];
                range_of(a, R, pdf, 0u, false, b0, b1);
            }
            march_range<ST, SHADE, JUMP>(A, s_tf, R, b0, b1, C0, C1, C2, T, evald);
        }
        if (check && fabsf(T - that) > A.eps) {
            fb = 1;
            plain_ray<ST, SHADE>(a, s_tf, R, C0, C1, C2, T, evald);
        }
    }
    if (inimg) {
        a.out[pix] = make_float4(C0, C1, C2, 1.0f - T);
        if (A.fallback) A.fallback[pix] = (uint8_t)fb;
    }
    if (a.stats) importance_stats(a, evald, fb, hit, inimg);
}

// ---------------------------------------------------------------------------
// training on the tensor cores: forward as the inference, then per layer the
// weight gradient (rays as K, accumulated in TMEM over the CTA's tiles) and
// the input gradient (rays as M)
// ---------------------------------------------------------------------------
// A CTA runs two groups of 128 threads (thread = ray = TMEM lane), each on its
// own tiles of 128 rays, and one thread that issues every MMA of both: while one
// group's MMAs run, the other group's threads work on their accumulators. The
// issuing order is fixed (step by step, group 0 then group 1, tiles in ascending
// order), so the groups share the weight-gradient accumulators and the sums do
// not depend on timing.
//
// Weight gradient of layer l: dW_l = H_{l-1}^T dZ_l over the tile's 128 rays, an
// M = 128, K = 128 MMA that reads both operands MN-major straight from the
// forward's K-major ones: A starts at H_{l-1} (or at the ones chunk before it)
// and covers 16 chunks of 8 columns; the row of the ones column is the bias
// gradient, and rows that fall on whatever lies beyond H_{l-1} are never read
// back. Input gradient: dH_{l-1} = dZ_l W_l^T, whose B operand is the forward's
// weight operand read MN-major. dZ_l overwrites H_l in place (its readers, the
// MMAs of step l + 1, have completed). Shared memory per group, in chunks of
// 8 columns x 128 rays (2 KB): X 14 | ones | H1 8 | H2 8 | ones | H3 8 | dZ4 6.
// All operands BF16 (dZ rounded once), FP32 accumulation.
//
// Bound: the chain of eight dependent MMA steps per tile with the threads' work
// between them (the loss is the longest stretch). 1048576 rays 746 us with one
// group of 128 threads per SM that issued for itself and kept 128-column
// operands, 421 with two groups, 388 with the input gradient committed before
// the weight gradient and the targets fetched under the forward (features and
// targets: 90 us at the copy rate). Fetching the next tile's features under the
// backward as well: 384, and 1.5 us more for a batch of 8192.
constexpr int kChX = 0, kChOne0 = 14, kChH1 = 15, kChH2 = 23, kChOne1 = 31, kChH3 = 32, kChDz4 = 40, kChunks = 46;
constexpr int kChunkBytes = 2048;
constexpr int kTrainThreads = 2 * kGroupThreads + 32;      // two groups and the issuing warp
struct TrainSmem {
    uint8_t op[2][kChunks * kChunkBytes];  // operands of the groups (the last A operand reads one chunk into what follows)
    uint8_t w[kUmmaBytes];                 // the four layers' weight operands
    float bias[3 * kHid + kN4];
    float wloss[8];
    unsigned long long bar_w, ready[2], done[2], done_w[2];
    uint32_t tmem;
};
constexpr int kTrainCols = 512;
constexpr uint32_t kColD = 0, kColW = 128;                 // D of group g at 64 g; dW of layer l at 128 + 64 l

// First chunk of the layer input H_l (l = 0: the features), of the weight
// gradient's A operand of layer l, and its accumulator row of input 0 and of
// the bias.
__device__ __forceinline__ int input_chunk(int l) { return l == 0 ? kChX : l == 1 ? kChH1 : l == 2 ? kChH2 : kChH3; }
__device__ __forceinline__ int grad_chunk(int l) { return l == 0 ? kChX : l == 1 ? kChOne0 : l == 2 ? kChH2 : kChOne1; }
__device__ __forceinline__ int grad_row0(int l) { return l == 1 || l == 3 ? 8 : 0; }
__device__ __forceinline__ int bias_row(int l) { return l == 0 ? kFeat : l == 2 ? kHid : 0; }

// One layer of the forward: D = A W^T.
__device__ __forceinline__ void issue_forward(uint32_t op, uint32_t w, int l, uint32_t tmem_d) {
    const NetLayer L = net_layer(l);
    const uint32_t a0 = op + input_chunk(l) * kChunkBytes, b0 = w + L.b_off, lbo_b = (uint32_t)(L.N / 8) * 128;
    const uint32_t idesc = tc::idesc_bf16_f32(128, L.N);
    for (int ks = 0; ks < L.K / 16; ks++)
        tc::mma_bf16(tmem_d, tc::smem_desc(a0 + ks * 2 * kChunkBytes, kChunkBytes, 128),
                     tc::smem_desc(b0 + ks * 2 * lbo_b, lbo_b, 128), idesc, ks > 0);
}

// Backward of layer l: the input gradient first (the group works on it while
// the weight gradient runs), each with its own commit.
__device__ __forceinline__ void issue_backward(uint32_t op, uint32_t w, int l, uint32_t tmem_w, uint32_t tmem_d,
                                               bool accumulate, uint32_t done, uint32_t done_w) {
    const NetLayer L = net_layer(l);
    const uint32_t dz = op + (l == 3 ? kChDz4 : input_chunk(l + 1)) * kChunkBytes;
    const uint32_t a0 = op + grad_chunk(l) * kChunkBytes;
    if (l > 0) {
        const uint32_t id_d = tc::idesc_bf16_f32(128, kHid) | tc::kIdescMnMajorB;
        for (int ks = 0; ks < L.N / 16; ks++)  // 16 outputs each
            tc::mma_bf16(tmem_d, tc::smem_desc(dz + ks * 2 * kChunkBytes, kChunkBytes, 128),
                         tc::smem_desc(w + L.b_off + ks * 256, 128, (uint32_t)(L.N / 8) * 128), id_d, ks > 0);
        tc::commit(done);
    }
    const uint32_t id_w = tc::idesc_bf16_f32(128, L.N) | tc::kIdescMnMajorA | tc::kIdescMnMajorB;
    for (int ks = 0; ks < 8; ks++)             // 16 rays each
        tc::mma_bf16(tmem_w, tc::smem_desc(a0 + ks * 256, 128, kChunkBytes), tc::smem_desc(dz + ks * 256, 128, kChunkBytes),
                     id_w, accumulate || ks > 0);
    tc::commit(done_w);
}

// dZ of this thread's ray (N values, zeros up to a multiple of 8) as row t of a
// K-major operand, 8 values per 16-byte store.
template <int N>
__device__ __forceinline__ void put_dz(uint8_t *A, const float (&dz)[N], int t) {
#pragma unroll
    for (int j0 = 0; j0 < N; j0 += 8) {
        uint4 q;
        uint32_t *w = reinterpret_cast<uint32_t *>(&q);
#pragma unroll
        for (int h = 0; h < 4; h++) {
            __nv_bfloat162 b2 = __floats2bfloat162_rn(dz[j0 + 2 * h], dz[j0 + 2 * h + 1]);
            w[h] = *reinterpret_cast<uint32_t *>(&b2);
        }
        *reinterpret_cast<uint4 *>(A + tc::core_offset(t, j0, 128)) = q;
    }
}

__global__ void __launch_bounds__(kTrainThreads, 1) tc_train_kernel(const TrainArgs A) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    TrainSmem &S = *reinterpret_cast<TrainSmem *>(smem_raw);
    const int tid = threadIdx.x, g = tid / kGroupThreads, t = tid % kGroupThreads;     // g = 2: the issuing warp
    const int warp = t >> 5, lane = t & 31;
    if (tid < 32) tc::tmem_alloc<kTrainCols>(tc::smem_addr(&S.tmem));
    if (tid == 0) {
        tc::bar_init(tc::smem_addr(&S.bar_w), 1);
        for (int i = 0; i < 2; i++) {
            tc::bar_init(tc::smem_addr(&S.ready[i]), kGroupThreads);
            tc::bar_init(tc::smem_addr(&S.done[i]), 1);
            tc::bar_init(tc::smem_addr(&S.done_w[i]), 1);
        }
    }
    for (int i = tid; i < 3 * kHid + kN4; i += blockDim.x) {
        const int l = i / kHid, j = i % kHid;
        float b = 0.0f;
        if (l < 3) b = A.params[(l == 0 ? kOffB1 : l == 1 ? kOffB2 : kOffB3) + j];
        else if (j < kOut) b = A.params[kOffB4 + j];
        S.bias[i] = b;
    }
    if (g < 2) {
        const uint4 one = make_uint4(0x3F80u, 0u, 0u, 0u);          // BF16 1, then seven zeros
        *reinterpret_cast<uint4 *>(S.op[g] + kChOne0 * kChunkBytes + t * 16) = one;
        *reinterpret_cast<uint4 *>(S.op[g] + kChOne1 * kChunkBytes + t * 16) = one;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = S.tmem;
    if (tid == 0) tc::bulk_g2s(tc::smem_addr(S.w), A.umma, kUmmaBytes, tc::smem_addr(&S.bar_w));
    bool ok = __syncthreads_and(tc::bar_wait(tc::smem_addr(&S.bar_w), 0, A.budget));
    if (!ok) tc::bar_wait(tc::smem_addr(&S.bar_w), 0, A.budget);     // the copy may still be in flight
    const long long ntiles = (A.n + 127) / 128;
    float loss_sum = 0.0f;
    if (ok && tid == 2 * kGroupThreads) {
        // the issuing thread: steps 0-3 the forward layers, 4-7 the backward
        // ones, for the tiles i = 2 pair + group of this CTA
        const uint32_t w = tc::smem_addr(S.w);
        uint32_t phase[2] = {0u, 0u};
        int issued[2] = {-1, -1};                    // last step issued
        uint32_t tiles_done[2] = {0u, 0u};
        for (long long pair = 0; ok && blockIdx.x + 2 * pair * gridDim.x < ntiles; pair++) {
#pragma unroll 1
            for (int step = 0; step < 8 && ok; step++) {
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    if (blockIdx.x + (2 * pair + q) * gridDim.x >= ntiles || !ok) continue;
                    ok = tc::bar_wait(tc::smem_addr(&S.ready[q]), phase[q], A.budget);
                    if (!ok) continue;
                    phase[q] ^= 1u;
                    tc::fence_after();
                    if (!A.issue_mma) continue;
                    if (step == 0 && issued[q] == 7) tiles_done[q]++;
                    const uint32_t op = tc::smem_addr(S.op[q]), d = tmem + kColD + 64u * q;
                    const uint32_t done = tc::smem_addr(&S.done[q]);
                    if (step < 4) {
                        issue_forward(op, w, step, d);
                        tc::commit(done);
                    } else {
                        issue_backward(op, w, 7 - step, tmem + kColW + 64u * (7 - step), d, pair > 0 || q > 0, done,
                                       tc::smem_addr(&S.done_w[q]));
                    }
                    issued[q] = step;
                }
            }
        }
        // every commit but the last step's was waited for by the group before it
        // made the next step ready; wait (bounded) for those still in flight.
        // Steps 0-6 of a tile commit to `done` (7 per tile), 4-7 to `done_w` (4).
        for (int q = 0; q < 2; q++) {
            const uint32_t n = tiles_done[q] * 7u + (uint32_t)min(issued[q] + 1, 7);
            const uint32_t nw = tiles_done[q] * 4u + (uint32_t)max(issued[q] - 3, 0);
            if (n) tc::bar_wait(tc::smem_addr(&S.done[q]), (n - 1u) & 1u, A.budget);
            if (nw) tc::bar_wait(tc::smem_addr(&S.done_w[q]), (nw - 1u) & 1u, A.budget);
        }
        if (!ok) atomicOr(A.err, 1);
    } else if (ok && g < 2) {
        const uint32_t ready = tc::smem_addr(&S.ready[g]), done = tc::smem_addr(&S.done[g]), done_w = tc::smem_addr(&S.done_w[g]);
        uint8_t *op = S.op[g];
        const uint32_t taddr = tmem + kColD + 64u * g + ((uint32_t)(warp * 32) << 16);     // this warp's lanes of D
        uint32_t phase = 0, phase_w = 0;
        // makes the operands just written (and D, if read) available to the
        // issuing thread
        auto hand_over = [&]() {
            tc::fence_async_smem();
            tc::fence_before();
            tc::bar_arrive(ready);
        };
        // the group's MMAs of the step are complete; the same answer in every
        // thread of the group, and a barrier of it
        auto wait_done = [&]() {
            ok = group_sync_and(g, tc::bar_wait(done, phase, A.budget));
            phase ^= 1u;
            tc::fence_after();
            return ok;
        };
        auto wait_done_w = [&]() {
            ok = group_sync_and(g, tc::bar_wait(done_w, phase_w, A.budget));
            phase_w ^= 1u;
            return ok;
        };
#pragma unroll 1
        for (long long tile = blockIdx.x + (long long)g * gridDim.x; ok && tile < ntiles; tile += 2ll * gridDim.x) {
            const long long r0 = tile * 128;
            const int nvalid = (int)min((long long)128, A.n - r0);
            const bool valid = t < nvalid;
            // the group's next tile (features and targets) into L2
            const long long nt = tile + 2ll * gridDim.x;
            if (t == 0 && nt < ntiles) {
                const long long nrows = min((long long)128, A.n - nt * 128);
                tc::prefetch_l2(A.feat + nt * 128 * kFeat, (uint32_t)(nrows * kFeat * sizeof(float)));
                tc::prefetch_l2(A.target + nt * 128 * kOutUsed, (uint32_t)((nrows * kOutUsed * sizeof(float)) & ~15ull));
            }
            // features: coalesced float4 loads of the contiguous tile, all in
            // flight at once -> BF16
            {
                const float4 *src = reinterpret_cast<const float4 *>(A.feat + r0 * kFeat);
                constexpr int kLoads = 128 * kFeat / 4 / 128;
                float4 v[kLoads];
#pragma unroll
                for (int i = 0; i < kLoads; i++) {
                    const int e = i * 128 + t;
                    v[i] = e / (kFeat / 4) < nvalid ? __ldg(src + e) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                }
#pragma unroll
                for (int i = 0; i < kLoads; i++) {
                    const int e = i * 128 + t, row = e / (kFeat / 4), k = (e % (kFeat / 4)) * 4;
                    __nv_bfloat162 lo = __floats2bfloat162_rn(v[i].x, v[i].y), hi = __floats2bfloat162_rn(v[i].z, v[i].w);
                    uint2 q;
                    q.x = *reinterpret_cast<uint32_t *>(&lo);
                    q.y = *reinterpret_cast<uint32_t *>(&hi);
                    *reinterpret_cast<uint2 *>(op + kChX * kChunkBytes + tc::core_offset(row, k, 128)) = q;
                }
            }
            hand_over();
            // this warp's targets, 17 and 16 columns of its 32 rows, in flight
            // under the forward
            float yc[kOutUsed];
            {
                const float *src = A.target + (r0 + warp * 32) * kOutUsed;
                const int rows = max(0, min(32, nvalid - warp * 32));
#pragma unroll
                for (int i = 0; i < kOutUsed; i++) {
                    const int nc = i < 17 ? 17 : 16, e = (i < 17 ? i : i - 17) * 32 + lane, row = e / nc;
                    yc[i] = row < rows ? __ldg(src + row * kOutUsed + (i < 17 ? 0 : 17) + e % nc) : 0.0f;
                }
            }
            // forward: layers 1-3 into H1..H3
#pragma unroll 1
            for (int l = 0; l < 3; l++) {
                if (!wait_done()) break;
                store_hidden<true>(op + input_chunk(l + 1) * kChunkBytes, taddr, S.bias + l * kHid, t);
                hand_over();
            }
            if (!ok) break;
            // while layer 4 runs: the targets turned from the coalesced order to
            // one ray per lane, through the dZ4 operand's memory (2 KB per warp,
            // free until dZ4 is written after the group's next barrier), 17
            // columns at a time
            float y[kOutUsed + 1];
            {
                float *stage = reinterpret_cast<float *>(op + kChDz4 * kChunkBytes) + warp * (32 * 17);
#pragma unroll
                for (int half = 0; half < 2; half++) {
                    const int nc = half ? 16 : 17;
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < nc; i++) {
                        const int e = i * 32 + lane;
                        stage[(e / nc) * 17 + e % nc] = yc[17 * half + i];
                    }
                    __syncwarp();
#pragma unroll
                    for (int c = 0; c < 17; c++) y[17 * half + c] = c < nc ? stage[lane * 17 + c] : 0.0f;
                }
            }
            if (!wait_done()) break;
            // loss per ray: w KL(q || p) + (T^ - T)^2, q = bins / w, w = sum(bins):
            // w q (log q - log p) = y (log y - log w - log p); dZ4 = dL/dz / n with
            // w (p - q) = w p - y
            {
                float dz[kN4];
                float v[64];
                tc::tmem_ld64(taddr, v);               // the 48 used of the 64 D columns, one round trip
#pragma unroll
                for (int j = 0; j < kN4; j++) dz[j] = v[j] + S.bias[3 * kHid + j];
                float kl = 0.0f, mx = dz[0], W = 0.0f, se = 0.0f;
#pragma unroll
                for (int b = 0; b < kBins; b++) {
                    mx = fmaxf(mx, dz[b]);
                    W += y[b];
                }
#pragma unroll
                for (int b = 0; b < kBins; b++) {
                    v[b] = expf(dz[b] - mx);
                    se += v[b];
                }
                const float lse = mx + logf(se), wp = W / se, lw = W > 0.0f ? logf(W) : 0.0f;
#pragma unroll
                for (int b = 0; b < kBins; b++) {
                    kl += fmaxf(y[b], 0.0f) * ((logf(fmaxf(y[b], 1e-37f)) - lw) - (dz[b] - lse));     // 0 where y is 0
                    dz[b] = W > 0.0f && valid ? (wp * v[b] - y[b]) * A.inv_n : 0.0f;
                }
                const float th = 1.0f / (1.0f + expf(-dz[kBins]));
                const float dt = th - y[kBins];
                const float loss = (W > 0.0f ? kl : 0.0f) + dt * dt;
                dz[kBins] = valid ? 2.0f * dt * th * (1.0f - th) * A.inv_n : 0.0f;
#pragma unroll
                for (int j = kOutUsed; j < kN4; j++) dz[j] = 0.0f;
                if (valid) loss_sum += loss;
                put_dz(op + kChDz4 * kChunkBytes, dz, t);
            }
            hand_over();
            // backward: dZ_l = dH_l * [H_l > 0] over H_l, layers 3..1
#pragma unroll 1
            for (int l = 3; l > 0; l--) {
                if (!wait_done()) break;
                uint8_t *H = op + input_chunk(l) * kChunkBytes;
                float v[kHid];
                tc::tmem_ld64(taddr, v);
#pragma unroll
                for (int j0 = 0; j0 < kHid; j0 += 8) {
                    const uint4 q = *reinterpret_cast<const uint4 *>(H + tc::core_offset(t, j0, 128));
                    const uint32_t h[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                    for (int i = 0; i < 4; i++) {          // a ReLU output is positive unless its bits are zero
                        if ((h[i] & 0x7FFFu) == 0u) v[j0 + 2 * i] = 0.0f;
                        if ((h[i] & 0x7FFF0000u) == 0u) v[j0 + 2 * i + 1] = 0.0f;
                    }
                }
                // the weight gradient of layer l + 1 reads H_l
                if (!wait_done_w()) break;
                put_dz(H, v, t);
                hand_over();
            }
            // the last step reads X and dZ1, which the next tile overwrites
            if (!ok || !wait_done_w()) break;
        }
        if (!ok && t == 0) atomicOr(A.err, 1);
    }
    // the CTA's gradient: accumulator row = input (or the bias), column = output;
    // group 0 reads layers 1 and 2, group 1 layers 3 and 4
    tc::fence_before();
    ok = __syncthreads_and(ok);
    tc::fence_after();
    if (g < 2) {
        float *part = A.partial + (size_t)blockIdx.x * kParams;
        const int acc_row = warp * 32 + lane;
#pragma unroll 1
        for (int l = 2 * g; l < 2 * g + 2; l++) {
            const int n_in = l == 0 ? kFeat : kHid, n_out = l == 3 ? kOut : kHid;
            const int offW = l == 0 ? kOffW1 : l == 1 ? kOffW2 : l == 2 ? kOffW3 : kOffW4;
            const int offB = l == 0 ? kOffB1 : l == 1 ? kOffB2 : l == 2 ? kOffB3 : kOffB4;
            const int row = acc_row - grad_row0(l);
            float *dst = acc_row == bias_row(l) ? part + offB : row >= 0 && row < n_in ? part + offW + row * n_out : nullptr;
            float v[kHid];
            tc::tmem_ld64(tmem + kColW + 64u * l + ((uint32_t)(warp * 32) << 16), v);
            if (!dst) continue;
#pragma unroll
            for (int c = 0; c < kHid; c += 4)
                if (c < n_out)
                    *reinterpret_cast<float4 *>(dst + c) =
                        ok ? make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        // loss: per-warp sums in a fixed order, then the CTA's
        for (int o = 16; o > 0; o >>= 1) loss_sum += __shfl_xor_sync(0xffffffffu, loss_sum, o);
        if (lane == 0) S.wloss[4 * g + warp] = loss_sum;
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid == 0) {
        float sum = S.wloss[0];
        for (int i = 1; i < 8; i++) sum += S.wloss[i];
        A.loss_partial[blockIdx.x] = sum;
    }
    if (tid < 32) tc::tmem_free<kTrainCols>(tmem);
}

// Byte of parameter i's BF16 copy in the packed B operands (element (n, k) of
// layer l is W_l[k][n], core-matrix layout), or -1 for a bias.
__device__ __forceinline__ int operand_offset(int i) {
    int off, nw, N;
    unsigned base;
    if (i < kOffB1) { off = i; nw = N = kHid; base = kUmmaL1; }
    else if (i < kOffW2) return -1;
    else if (i < kOffB2) { off = i - kOffW2; nw = N = kHid; base = kUmmaL2; }
    else if (i < kOffW3) return -1;
    else if (i < kOffB3) { off = i - kOffW3; nw = N = kHid; base = kUmmaL3; }
    else if (i < kOffW4) return -1;
    else if (i < kOffB4) { off = i - kOffW4; nw = kOut; N = kN4; base = kUmmaL4; }
    else return -1;
    return (int)(base + tc::core_offset(off % nw, off / nw, N));
}

// Sums the CTAs' partials: 32 parameters per block, eight threads on each
// (every eighth partial, then a fixed order), so that the loads are whole lines
// and eight chains of them run side by side (one thread per parameter took
// 12.5 us for 152 partials). STEP: the Adam update (beta1 0.9, beta2 0.999, eps
// 1e-8) of the FP32 parameters and their BF16 operands follows in the same
// thread (a training step of 8192 rays 60 -> 25 us with the gradient kernel).
template <bool STEP>
__global__ void __launch_bounds__(256) reduce_grad_kernel(const float *partial, const float *loss_partial, int nblocks,
                                                          float inv_n, float *grad, float *loss, AdamArgs P) {
    __shared__ float s_sum[8][32];
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5, i = blockIdx.x * 32 + lane;
    float s = 0.0f;
    if (i < kParams)
        for (int b = seg; b < nblocks; b += 8) s += partial[(size_t)b * kParams + i];
    s_sum[seg][lane] = s;
    __syncthreads();
    if (seg == 0 && i < kParams) {
        float gi = s_sum[0][lane];
#pragma unroll
        for (int q = 1; q < 8; q++) gi += s_sum[q][lane];
        grad[i] = gi;
        if (STEP) {
            const float mi = 0.9f * P.m[i] + 0.1f * gi;
            const float vi = 0.999f * P.v[i] + 0.001f * gi * gi;
            P.m[i] = mi;
            P.v[i] = vi;
            const float pi = P.params[i] - P.lr * (mi / P.c1) / (sqrtf(vi / P.c2) + 1e-8f);
            P.params[i] = pi;
            const int o = operand_offset(i);
            if (o >= 0) *reinterpret_cast<__nv_bfloat16 *>(P.umma + o) = __float2bfloat16_rn(pi);
        }
    }
    if (loss && blockIdx.x == 0 && seg == 1) {
        float q = 0.0f;
        for (int b = lane; b < nblocks; b += 32) q += loss_partial[b];
        for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        if (lane == 0) *loss = q * inv_n;
    }
}

int train_grid(long long n) {
    int dev = 0, sms = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long tiles = (n + 127) / 128;
    return (int)max(1ll, min((long long)sms, tiles));
}

cudaError_t launch_train_grad(const TrainArgs &a, int grid, float *grad, float *loss, const AdamArgs *step, cudaStream_t s) {
    const int smem = (int)sizeof(TrainSmem);
    cudaError_t e = cudaFuncSetAttribute(tc_train_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    tc_train_kernel<<<grid, kTrainThreads, smem, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const int blocks = (kParams + 31) / 32;
    if (step) reduce_grad_kernel<true><<<blocks, 256, 0, s>>>(a.partial, a.loss_partial, grid, a.inv_n, grad, loss, *step);
    else reduce_grad_kernel<false><<<blocks, 256, 0, s>>>(a.partial, a.loss_partial, grid, a.inv_n, grad, loss, AdamArgs{});
    return cudaGetLastError();
}

// B operands of the four layers in the core-matrix layout: element (n, k) of
// layer l is bf16(W_l[k][n]) (0 for the padding rows n >= 40 of layer 4).
__global__ void pack_umma_kernel(const float *params, uint8_t *umma) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    constexpr int n1 = kHid * kFeat, n2 = kHid * kHid, n4 = kN4 * kHid;
    if (idx >= n1 + 2 * n2 + n4) return;
    int r, K, N, nw, woff;
    unsigned boff;
    if (idx < n1) { r = idx; K = kFeat; N = kHid; nw = kHid; woff = kOffW1; boff = kUmmaL1; }
    else if (idx < n1 + n2) { r = idx - n1; K = kHid; N = kHid; nw = kHid; woff = kOffW2; boff = kUmmaL2; }
    else if (idx < n1 + 2 * n2) { r = idx - n1 - n2; K = kHid; N = kHid; nw = kHid; woff = kOffW3; boff = kUmmaL3; }
    else { r = idx - n1 - 2 * n2; K = kHid; N = kN4; nw = kOut; woff = kOffW4; boff = kUmmaL4; }
    const int n = r / K, k = r % K;
    const float w = n < nw ? params[woff + k * nw + n] : 0.0f;
    *reinterpret_cast<__nv_bfloat16 *>(umma + boff + tc::core_offset(n, k, N)) = __float2bfloat16_rn(w);
}

cudaError_t launch_pack(const float *params, uint8_t *umma, cudaStream_t s) {
    constexpr int total = kHid * kFeat + 2 * kHid * kHid + kN4 * kHid;
    pack_umma_kernel<<<(total + 255) / 256, 256, 0, s>>>(params, umma);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static dim3 image_grid(const CamRec &c) { return dim3((c.W + 15) / 16, (c.H + 7) / 8); }

cudaError_t launch_profiles(const MarchArgs &a, float *out, cudaStream_t s) {
    const size_t smem = (size_t)a.tf.K * sizeof(float4);
    auto go = [&](auto kern) -> cudaError_t {
        if (smem > 40 * 1024) {       // the staged rows take 4.2 KB of the 48 KB beside it
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        const dim3 grid((a.cam.W + kProfTileX - 1) / kProfTileX, min(65535, (a.cam.H + kProfTileY - 1) / kProfTileY));
        kern<<<grid, 128, smem, s>>>(a, out);
        return cudaGetLastError();
    };
    return by_storage<false>(a.vol, [&](auto st) { return go(profiles_kernel<decltype(st)::value>); });
}

cudaError_t launch_features(const MarchArgs &a, float *out, cudaStream_t s) {
    auto kern = (reinterpret_cast<uintptr_t>(out) & 15u) == 0 ? features_kernel<true> : features_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kFeatSmem);
    if (e != cudaSuccess) return e;
    kern<<<image_grid(a.cam), 128, kFeatSmem, s>>>(a, out);
    return cudaGetLastError();
}

// Persistent network CTAs: as many as fit on the device at once (shared
// memory, registers and the SM's 512 TMEM columns), at most one per G tiles.
template <bool FEAT, int G>
static cudaError_t launch_tc(const TcNetArgs &a, cudaStream_t s) {
    constexpr int kTmemCols = tmem_cols(G);
    auto kern = tc_net_kernel<FEAT, G>;
    const int smem = (int)sizeof(NetSmem<G>);
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100)) != cudaSuccess) return e;
    // CTAs per SM from the SM's shared memory and registers (the occupancy
    // query does not see the carveout preference and answers 1), at most as
    // many as the 512 TMEM columns hold
    int dev = 0, sms = 0, smem_sm = 0, smem_rsv = 0, regs_sm = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&smem_rsv, cudaDevAttrReservedSharedMemoryPerBlock, dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev)) != cudaSuccess) return e;
    cudaFuncAttributes fa;
    if ((e = cudaFuncGetAttributes(&fa, kern)) != cudaSuccess) return e;
    const int threads = G * kGroupThreads;
    const int by_smem = smem_sm / (smem + smem_rsv);
    const int by_regs = regs_sm / max(1, fa.numRegs * threads);
    const int per_sm = max(1, min(min(by_smem, by_regs), 512 / kTmemCols));
    const long long grid = min((long long)sms * per_sm, (a.ntiles + G - 1) / G);
    if (grid < 1) return cudaSuccess;
    kern<<<(unsigned)grid, threads, smem, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_tc_net(const TcNetArgs &a, cudaStream_t s) {
    return a.feat ? launch_tc<true, kFeatGroups>(a, s) : launch_tc<false, kCamGroups>(a, s);
}

template <int ST, bool SHADE>
static cudaError_t launch_imp_st(const ImportanceArgs &a, int nviews, cudaStream_t s) {
    const size_t smem = (size_t)a.m.tf.K * sizeof(float4);
    auto go = [&](auto kern) -> cudaError_t {
        if (smem > 48 * 1024) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        dim3 grid = image_grid(a.m.cam);
        grid.z = nviews;
        kern<<<grid, 128, smem, s>>>(a);
        return cudaGetLastError();
    };
    // the range marches jump empty blocks from 48 samples per ray up
    const bool jump = a.nimp >= 48;
    if (a.range)
        return jump ? go(importance_kernel<ST, SHADE, kSrcRecords, true>) : go(importance_kernel<ST, SHADE, kSrcRecords>);
    if (a.sampling == RC_SAMPLING_INVCDF) return go(importance_kernel<ST, SHADE, kSrcInvCdf>);
    return jump ? go(importance_kernel<ST, SHADE, kSrcRange, true>) : go(importance_kernel<ST, SHADE, kSrcRange>);
}

cudaError_t launch_importance(const ImportanceArgs &a, int nviews, cudaStream_t s) {
    if (a.m.p.shade)
        return by_storage<true>(a.m.vol, [&](auto st) { return launch_imp_st<decltype(st)::value, true>(a, nviews, s); });
    return by_storage<false>(a.m.vol, [&](auto st) { return launch_imp_st<decltype(st)::value, false>(a, nviews, s); });
}

}  // namespace rc
