// Host-side rules that choose the form of a launch from its sizes. Plain C++
// without CUDA types, so that they can be compiled and tested by themselves.
#pragma once

#include <math.h>

namespace rc {

// CTAs of a persistent launch that takes `chunks` pieces of work from a queue,
// one CTA per SM: as many as there are SMs or chunks. A CTA of the 2-D table's
// gradient runs two or three groups, each with its own chunk, but an SM for
// each chunk comes first (128x128x96, 32 x 256 table, one 128^2 view of 64
// chunks: 748 us packed three to a CTA, 674 spread; 2 x 2 table 735 and 615).
inline int persistent_ctas(int chunks, int sms) { return chunks < sms ? chunks : sms; }

// The camera record's fields that say where the volume's box lies in an image.
struct ViewGeom {
    double o[3], f[3], r[3], u[3];     // eye (index space), view basis (world)
    double tx, ty;                     // tangents of the half angles
    int W, H;
};

struct BoxGeom {
    int n[3];                          // voxels
    double s[3];                       // spacing
};

// About how many rays of a view meet the volume, and what part of the box's
// diagonal they cross: the box's corners bound the part of the image whose rays
// can, and its silhouette fills about two thirds of that rectangle. From inside
// the box every ray meets it, and leaves it after about a third of the diagonal.
inline void view_rays(const ViewGeom &c, const BoxGeom &b, double &hits, double &chord) {
    const double pixels = (double)c.W * c.H;
    bool inside = true;
    for (int i = 0; i < 3; i++) inside = inside && c.o[i] >= 0.0 && c.o[i] <= b.n[i] - 1;
    chord = inside ? 0.35 : 1.0;
    hits = inside ? pixels : 0.65 * pixels;
    if (inside) return;
    double lo[2] = {1.0, 1.0}, hi[2] = {-1.0, -1.0};
    for (int q = 0; q < 8; q++) {
        double z = 0.0, e[2] = {0.0, 0.0};
        for (int i = 0; i < 3; i++) {
            const double d = (((q >> i) & 1 ? b.n[i] - 1 : 0) - c.o[i]) * b.s[i];
            z += d * c.f[i];
            e[0] += d * c.r[i];
            e[1] += d * c.u[i];
        }
        if (!(z > 0.0)) return;                            // a corner behind the eye: the whole image
        e[0] /= z * c.tx;
        e[1] /= z * c.ty;
        for (int i = 0; i < 2; i++) {
            lo[i] = e[i] < lo[i] ? e[i] : lo[i];
            hi[i] = e[i] > hi[i] ? e[i] : hi[i];
        }
    }
    for (int i = 0; i < 2; i++) {
        const double l = lo[i] > -1.0 ? lo[i] : -1.0, h = hi[i] < 1.0 ? hi[i] : 1.0;
        hits *= h > l ? (h - l) * 0.5 : 0.0;
    }
}

// The size of a march launch over all its views: rays that meet the volume,
// samples along the diagonal (from inside the box, along their shorter chords),
// and the rays of one view per voxel of the box's cross-section (the two-thirds
// power of its voxels). The views are summed (up to kSizedViews of them, evenly
// spread): the first one alone says nothing about the others. Eight 1024^2 views
// of 256x256x180, unshaded, took 3.37 ms instead of 1.14 when the first of them
// looked past the volume, and 2.07 when it was far away.
struct LaunchSize {
    double hits = 0.0, steps = 0.0, density = 0.0;
};
constexpr int kSizedViews = 32;
inline int sized_stride(int views) { return (views + kSizedViews - 1) / kSizedViews; }

class LaunchSizer {
  public:
    LaunchSizer(const BoxGeom &b, double step) : box(b) {      // step: sample distance (world)
        double diag2 = 0.0;
        for (int i = 0; i < 3; i++) diag2 += (b.n[i] - 1) * b.s[i] * (b.n[i] - 1) * b.s[i];
        across = sqrt(diag2) / step;
    }
    void add(const ViewGeom &c) {
        double h, part;
        view_rays(c, box, h, part);
        hits += h;
        chords += h * part;
        added++;
    }
    // for `views` views of which the added ones are a sample
    LaunchSize size(double views) const {
        LaunchSize z;
        z.hits = added ? hits * views / added : 0.0;
        z.steps = hits > 0.0 ? across * (chords / hits) : across;
        z.density = z.hits / views / pow((double)box.n[0] * box.n[1] * box.n[2], 2.0 / 3.0);
        return z;
    }

  private:
    BoxGeom box;
    double across, hits = 0.0, chords = 0.0;
    int added = 0;
};

// Lanes per ray of a compositing launch. A ray's samples are a serial chain (a
// few hundred of them, 0.3 us each), so a launch with few rays takes the time of
// its longest ray however few there are; more lanes shorten the chain until the
// shuffles and the samples past termination fill the GPU. The lines lie where
// the measured times cross, in rays that meet the volume (`hits`, 0.27 of the
// pixels there) and per sample along the diagonal (`steps`); us per view with
// 1, 2, 4 and 8 lanes, FP32 shaded / FP32 plain:
//   64x64x32, 256^2:    79 58 46 42 / 68 44 35 40
//   128x128x96, 384^2: 118 107 74 88 / 102 65 66 73
//   256x256x180, 256^2: 147 102 72 61 / 162 84 58 56
//   256x256x180, 512^2: 172 142 135 161 / 135 105 99 131
//   256x256x180, 724^2: 223 201 214 293 / 150 143 162 235
//   256x256x180, 1024^2: 292 307 386 572 / 193 229 287 456
// From inside the box the chains are short and every pixel has one, so the
// lines come sooner: 256x256x180, 128^2 74 61 45 44 / 52 45 35 35, 181^2 76 70 68
// 79 / 51 51 48 60, 256^2 94 103 116 136 / 57 67 78 102.
// `heavy`: forms whose samples take longer (shading without 8-byte
// value+gradient entries, which the FP32 shaded figures above are for;
// B-spline; 2-D table) gain further up than the others.
inline int lanes_per_ray(const LaunchSize &z, bool heavy) {
    if (z.hits <= (heavy ? 22e3 : 7e3) && z.hits <= 70.0 * z.steps) return 8;
    if (z.hits <= 76e3 && z.hits <= 190.0 * z.steps) return 4;
    if (z.hits <= 155e3 && z.hits <= (heavy ? 390.0 : 190.0) * z.steps) return 2;
    return 1;
}

// Rays of a view per voxel of the cross-section, as far as it matters.
inline double pixel_density(const LaunchSize &z) { return z.density < 16.0 ? z.density : 16.0; }

// Samples finer than voxels and voxels not much coarser than pixels: two lanes
// of a ray share their footprints, and pay however many rays there are.
inline bool shared_footprints(const LaunchSize &z) { return z.density <= 10.0 && z.steps >= 400.0; }

// Lanes per ray of the sums: every ray marches its whole chord, so no sample is
// in vain, and what more lanes cost is the ray setup and the shuffles, which
// short chains do not repay, and the coherence of neighbouring rays, which is
// worth more the denser the pixels lie on the voxels (`density`). us with 1, 2
// and 4 lanes, FP32 trilinear / B-spline:
//   128x128x96, 512^2, 408 samples along the diagonal: 92 70 61 / 326 244 215
//   the same with 20 samples:                          15 14 18 / 35 33 37
//   128x128x96, 1024^2 (27 rays per voxel):           148 159 180 / 564 539 611
//   64x64x32, 1024^2 (128 rays per voxel):             66 74 97 / 209 210 246
//   256x256x180, 1024^2 (7 rays per voxel):           371 296 315 / 1797 1286 1380
//   51x302x86, four 870^2 views:                      288 244 273 / 1292 921 891
//   256x256x180, four 1024^2 views:                  1064 1051 1224 / 5685 4863 5112
//   the same, eight views:                                          / 11779 9970
// Fixed lines in rays (4 lanes up to 200e3, B-spline 600e3) took 2.3 times as
// long as one lane at a few samples per ray. Over 578 sizes these lines are
// within 1.3% of the best choice on average, 9% slower than one lane at worst.
inline int lanes_per_sum(const LaunchSize &z, bool cubic) {
    const double d = pixel_density(z);
    if (cubic) {
        if (!shared_footprints(z) && z.hits > 40e3 + 1600.0 * z.steps) return 1;
        return z.hits * pow(d, 0.7) <= 80e3 + 1600.0 * z.steps ? 4 : 2;
    }
    if (z.hits * pow(d, 0.4) > 80e3 + 1700.0 * z.steps) return 1;
    return z.hits * sqrt(d) <= 60e3 + 600.0 * z.steps ? 4 : 2;
}

// Lanes per ray of a maximum: as for the sums, with no shuffle per sample. us
// with 1, 2 and 4 lanes, FP32 trilinear / B-spline:
//   256x256x180, 256^2:              278 145 78 / 1172 644 347
//   128x128x96, 512^2:                92 65 50 / 331 242 208
//   128x128x96, four 1024^2 views:    475 499 571 / 2057 2089 2398
//   256x256x180, eight 1024^2 views: 2188 1984 2035
//   51x302x86, four 870^2 views:      287 230 245 / 1277 917 868
// Within 1% of the best choice on average over 510 sizes, 16% slower than one
// lane at worst.
inline int lanes_per_max(const LaunchSize &z, bool cubic) {
    const double d = pixel_density(z), x = z.hits * pow(d, cubic ? 0.25 : 0.7);
    if (!shared_footprints(z) && x > (cubic ? 60e3 + 4000.0 * z.steps : 40e3 + 6000.0 * z.steps)) return 1;
    return (cubic ? z.hits * sqrt(d) <= 120e3 + 1000.0 * z.steps : x <= 120e3 + 1600.0 * z.steps) ? 4 : 2;
}

}  // namespace rc
