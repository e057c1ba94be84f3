// k_rays.cu -- hierarchical, mesh-adaptive HEALPix ray sets (Section 2.1.3,
// Eq. 4, Fig. 1).
//
// Fixed level: every point gets all antipodal pairs of that level.
// Adaptive (one CTA per point): the directions from the point to the global
// sample of points are counted per pixel of the finest level (vec2pix in
// double precision, explicitly rounded operations); coarser counts come from
// nested downgrading (children 4p..4p+3 of pixel p).  Starting from all pairs
// of l_min, each level ranks the candidate pairs by the count of both members
// (ties to the smaller pixel index), keeps the bottom half as rays of that
// level and refines the top half into their four child pairs; at l_max every
// candidate is a ray.  The pairs are written sorted ascending.
#include "mgx_internal.cuh"

namespace mgx {

namespace {

constexpr double kTwoOverPi = 0.636619772367581343075535053490057448;

__device__ __forceinline__ int64_t spread2_64(int64_t v) {
    int64_t out = 0;
#pragma unroll
    for (int b = 0; b < 16; ++b) out |= ((v >> b) & 1) << (2 * b);
    return out;
}

// nested pixel of level l containing direction (dx, dy, dz); HEALPix zones of
// Gorski et al. (2005): equatorial |z| <= 2/3, polar caps otherwise
__device__ int32_t vec2pix_nest(int l, double dx, double dy, double dz) {
    const int64_t ns = int64_t(1) << l;
    const double len = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
    const double z = __ddiv_rn(dz, len);
    const double za = fabs(z);
    double t = __dmul_rn(atan2(dy, dx), kTwoOverPi);
    if (t < 0.0) t = __dadd_rn(t, 4.0);
    if (t >= 4.0) t = __dsub_rn(t, 4.0);
    int64_t face, x, y;
    if (za <= 2.0 / 3.0) {
        const double c1 = __dmul_rn(double(ns), __dadd_rn(0.5, t));
        const double c2 = __dmul_rn(double(ns), __dmul_rn(0.75, z));
        const int64_t asc = int64_t(__dsub_rn(c1, c2));
        const int64_t dsc = int64_t(__dadd_rn(c1, c2));
        const int64_t fa = asc >> l, fd = dsc >> l;
        face = (fa == fd) ? (fa | 4) : (fa < fd ? fa : fd + 8);
        x = dsc & (ns - 1);
        y = ns - 1 - (asc & (ns - 1));
    } else {
        int64_t q = int64_t(t);
        if (q > 3) q = 3;
        const double tp = __dsub_rn(t, double(q));
        const double w = __dmul_rn(double(ns), __dsqrt_rn(__dmul_rn(3.0, __dsub_rn(1.0, za))));
        int64_t a = int64_t(__dmul_rn(tp, w));
        int64_t b = int64_t(__dmul_rn(__dsub_rn(1.0, tp), w));
        if (a > ns - 1) a = ns - 1;
        if (b > ns - 1) b = ns - 1;
        if (z >= 0.0) {
            face = q;
            x = ns - 1 - b;
            y = ns - 1 - a;
        } else {
            face = q + 8;
            x = a;
            y = b;
        }
    }
    return int32_t((face << (2 * l)) + spread2_64(x) + 2 * spread2_64(y));
}

// The same pixel in single precision, certified: returns false when a
// rounding could move any of the decisions (the zone test, the face and the
// in-face indices, all truncations of non-negative arguments) away from those
// of vec2pix_nest above, which the caller then takes.  The translation unit is
// compiled without contraction, so each operation rounds once (u = 2^-24).
// The direction's components come as sums of two single-precision differences
// (split_direction): each within 2.01u of itself plus 0.05u of the largest one,
// of which the horizontal part is at least 1/16:
//   z = c / |v| within 10u |z| + 0.1u of the double z (inputs, sum of squares,
//     sqrt, division);
//   phi = atan2f(b, a) within kAtanErr + 3.3u of the double angle (3 ulp
//     documented; the rest from the inputs);
//   t = phi 2/pi (+4) within et = 0.64 kAtanErr + 15u (and not within et of 0,
//     where the wrap into [0, 4) jumps);
//   equatorial arguments ns (0.5 + t) -+ ns 0.75 z within ns (et + 0.75 ez + 11u);
//   polar w = ns sqrt(3 (1 - |z|)) within w ((ez + 2u) / (2 (1 - |z|)) + 2u), and
//   a, b = trunc(tp w), trunc((1 - tp) w) within et w + ew + 2u w.
// The double path's own rounding (about 1e-15) is inside these margins.
constexpr float kAtanErr = 9.5367431640625e-7f;  // 2^-20 rad

// Bits of v < 2^16 spread to the even places.
__device__ __forceinline__ int32_t spread2(uint32_t v) {
    v = (v | v << 8) & 0x00ff00ffu;
    v = (v | v << 4) & 0x0f0f0f0fu;
    v = (v | v << 2) & 0x33333333u;
    return int32_t((v | v << 1) & 0x55555555u);
}

__device__ __forceinline__ bool trunc_certain(float v, float e, int32_t &k) {
    // trunc of the double value equals trunc(v) when v is farther than e from
    // every integer other than 0 (trunc maps (-1, 1) to 0)
    if (!(v > -1.0f + e)) return false;
    if (v < 1.0f - e) {
        k = 0;
        return true;
    }
    const float f = floorf(v);
    if (v - f < e || f + 1.0f - v < e) return false;
    k = int32_t(f);
    return true;
}

__device__ bool vec2pix_nest_f(int l, float a, float b, float c, int32_t &pix) {
    constexpr float kU = 5.9604644775390625e-8f;  // 2^-24
    const int32_t ns = 1 << l;
    const float fns = float(ns);
    const float len = sqrtf(a * a + b * b + c * c);
    const float z = c / len;
    const float za = fabsf(z);
    const float ez = 10.0f * kU * za + 0.1f * kU;
    float t = atan2f(b, a) * 0.636619772367581343f;
    const float et = 0.64f * kAtanErr + 15.0f * kU;
    // the wrap into [0, 4) is discontinuous at t = 0: both precisions must be on the same side
    if (fabsf(t) < et) return false;
    if (t < 0.0f) t = t + 4.0f;
    if (t >= 4.0f) t = t - 4.0f;
    constexpr float kTwoThirds = 0.666666666666666667f;
    int32_t face, x, y;
    if (za <= kTwoThirds - ez - 2.0f * kU) {
        const float c1 = fns * (0.5f + t), c2 = fns * (0.75f * z);
        const float eA = fns * (et + 0.75f * ez + 11.0f * kU);
        int32_t asc, dsc;
        if (!trunc_certain(c1 - c2, eA, asc) || !trunc_certain(c1 + c2, eA, dsc)) return false;
        const int32_t fa = asc >> l, fd = dsc >> l;
        face = (fa == fd) ? (fa | 4) : (fa < fd ? fa : fd + 8);
        x = dsc & (ns - 1);
        y = ns - 1 - (asc & (ns - 1));
    } else if (za > kTwoThirds + ez + 2.0f * kU) {
        int32_t q;
        if (t > 3.0f + et) q = 3;
        else if (!trunc_certain(t, et, q)) return false;
        const float tp = t - float(q);
        const float om = 1.0f - za;
        const float w = fns * sqrtf(3.0f * om);
        const float ew = w * ((ez + 2.0f * kU) / (2.0f * om) + 2.0f * kU);
        if (!(ew < 0.25f)) return false;  // next to the pole
        int32_t ia, ib;
        if (!trunc_certain(tp * w, et * w + ew + 2.0f * kU * w, ia)) return false;
        if (!trunc_certain((1.0f - tp) * w, et * w + ew + 2.0f * kU * w, ib)) return false;
        if (ia > ns - 1) ia = ns - 1;
        if (ib > ns - 1) ib = ns - 1;
        if (z >= 0.0f) {
            face = q;
            x = ns - 1 - ib;
            y = ns - 1 - ia;
        } else {
            face = q + 8;
            x = ia;
            y = ib;
        }
    } else {
        return false;  // at the zone boundary
    }
    pix = (face << (2 * l)) + spread2(uint32_t(x)) + 2 * spread2(uint32_t(y));
    return true;
}

// A position's coordinate, scaled, as two floats.
__device__ __forceinline__ void split_coordinate(double x, double scale, float &hi, float &lo) {
    x = __dmul_rn(x, scale);
    hi = __double2float_rn(x);
    lo = __double2float_rn(__dsub_rn(x, double(hi)));
}

// The direction between two points from their scaled positions split into two
// floats each (hi = fl(x), lo = fl(x - hi)): a double subtraction takes the FP64
// pipe 77 cycles a warp.  Each component carries the roundings of the two
// differences and their sum, 2.01u of itself, and 2^-45.5 X from the split and the
// cancellation; false (scaled_direction takes it) unless the largest component is
// at least 2^-17 X, so that the latter is below 0.05u of it, and the horizontal
// part at least 1/16 of it.
__device__ __forceinline__ bool split_direction(const float4 &h, const float4 &l, const float4 &oh, const float4 &ol,
                                                float X, float &a, float &b, float &c) {
    a = (h.x - oh.x) + (l.x - ol.x);
    b = (h.y - oh.y) + (l.y - ol.y);
    c = (h.z - oh.z) + (l.z - ol.z);
    const float hor = fmaxf(fabsf(a), fabsf(b)), M = fmaxf(hor, fabsf(c));
    return M >= 7.62939453125e-6f * X && hor >= 0.0625f * M;
}

// The direction in single precision from the double differences, scaled by the
// power of two of the largest: each component within u of itself (2^-99 of the
// largest where it is left out).  False when all are 0 or next to the end of the range.
__device__ __forceinline__ bool scaled_direction(double dx, double dy, double dz, float &a, float &b, float &c) {
    auto field = [](double d) { return (__double2hiint(d) >> 20) & 0x7ff; };
    const int top = max(field(dx), max(field(dy), field(dz)));
    if (top <= 100) return false;
    auto part = [&](double d) {
        if (field(d) + 100 < top) return 0.0f;
        return __double2float_rn(__hiloint2double(__double2hiint(d) + (1023 - top) * (1 << 20), __double2loint(d)));
    };
    a = part(dx);
    b = part(dy);
    c = part(dz);
    return true;
}

// The sample's positions scaled and split (x, y, z of sp[2s] and sp[2s + 1]), the
// point's index in sp[2s].w (-1: out of range).
__global__ void k_split_sample(DevMesh m, int64_t n_sample, const int32_t *__restrict__ sample,
                               float4 *__restrict__ sp) {
    const int64_t s = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (s >= n_sample) return;
    const int32_t j = sample[s];
    const bool ok = j >= 0 && j < m.n;
    float4 h = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(ok ? j : -1)), l = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (ok) {
        split_coordinate(m.x[j], m.scale, h.x, l.x);
        split_coordinate(m.y[j], m.scale, h.y, l.y);
        split_coordinate(m.z[j], m.scale, h.z, l.z);
    }
    sp[2 * s] = h;
    sp[2 * s + 1] = l;
}

// atan2f as the single-precision ray-set screen evaluates it (for the tests of kAtanErr).
__global__ void k_eval_atan2(const float *__restrict__ x, int64_t n, float *__restrict__ y) {
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        y[i] = atan2f(x[n + i], x[i]);
}

__global__ void k_rays_fixed(int32_t n, int32_t level, int32_t npairs, const uint32_t *__restrict__ pairs,
                             uint32_t *__restrict__ rays) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= int64_t(n) * npairs) return;
    rays[i] = (uint32_t(level) << 28) | pairs[i % npairs];
}

__global__ void __launch_bounds__(256)
k_rays_adaptive(DevMesh m, int32_t lmin, int32_t lmax, int32_t npairs, int64_t n_sample,
                const float4 *__restrict__ sp, const int32_t *__restrict__ anti,
                const uint32_t *__restrict__ pairs_lmin, int32_t n_pairs_lmin,
                uint32_t *__restrict__ rays, int *status) {
    extern __shared__ uint32_t sm[];
    const int32_t o = blockIdx.x;
    const int tid = threadIdx.x, nt = blockDim.x;
    // shared layout: histograms of levels lmin..lmax, then candidate buffers
    uint32_t *hist[MGX_MAX_ADAPT_LEVEL + 1];
    int64_t off = 0;
    for (int l = lmax; l >= lmin; --l) {
        hist[l] = sm + off;
        off += int64_t(12) << (2 * l);
    }
    const int32_t cmax = int32_t((int64_t(12) << (2 * lmax)) / 2);
    uint32_t *cand = sm + off;
    uint32_t *next = cand + cmax;
    uint32_t *score = next + cmax;
    uint32_t *out = score + cmax;
    __shared__ int32_t nout;

    const int32_t nfine = int32_t(int64_t(12) << (2 * lmax));
    for (int32_t i = tid; i < nfine; i += nt) hist[lmax][i] = 0;
    if (tid == 0) nout = 0;
    __syncthreads();
    const double xo = m.x[o], yo = m.y[o], zo = m.z[o];
    // Single precision where the screen certifies the pixel, from the split positions or,
    // where they do not carry the direction (a distance below 2^-17 of the mesh's farthest
    // point from the coordinate origin; next to the z axis), from the double differences.
    // The directions that need either (`far`) or that the screen leaves open (`open`, below
    // a per cent) wait in lists of the warp and are taken 32 at a time: taken at once, by one
    // lane, they cost the whole warp the double path's 100-odd FP64 instructions (77 cycles
    // each) in a third of its steps.  30 000 points with 10 000 directions each: 19.4 ms so,
    // 9.7 with the list, 5.2 with the split positions and 32-bit indices in place of FP64
    // differences and 64-bit ones, 3.7 with the second list; 3.7 in any unit of length, 5.4 and
    // 4.9 when the mesh (of 100) is moved by 1e6 and 1e9 (with one list 57 in units of 1e16 or
    // when moved by 1e9, 31 when moved by 1e6).
    constexpr int kList = 64;
    __shared__ int32_t lists[256 / 32][2][kList];
    const int lane = tid & 31;
    int32_t *far = lists[tid >> 5][0], *open = lists[tid >> 5][1];
    int n_far = 0, n_open = 0;
    auto push = [&](int32_t *list, int &n, bool on, int32_t j) {  // returns whether 32 are waiting
        const unsigned mask = __ballot_sync(0xffffffffu, on);
        if (on) list[n + __popc(mask & ((1u << lane) - 1u))] = j;
        n += __popc(mask);
        __syncwarp();
        return n >= 32;
    };
    auto exact = [&](int32_t j) {
        const double dx = __dsub_rn(m.x[j], xo), dy = __dsub_rn(m.y[j], yo), dz = __dsub_rn(m.z[j], zo);
        if (dx == 0.0 && dy == 0.0 && dz == 0.0) return;  // a coincident point has no direction
        atomicAdd(&hist[lmax][vec2pix_nest(lmax, dx, dy, dz)], 1u);
    };
    auto take_open = [&]() {
        n_open -= 32;
        exact(open[n_open + lane]);
        __syncwarp();
    };
    auto take_far = [&](bool on, int32_t j) {
        float a, b, c;
        int32_t pix;
        bool left = false;
        if (on) {
            left = !scaled_direction(__dsub_rn(m.x[j], xo), __dsub_rn(m.y[j], yo), __dsub_rn(m.z[j], zo), a, b, c) ||
                   !vec2pix_nest_f(lmax, a, b, c, pix);
            if (!left) atomicAdd(&hist[lmax][pix], 1u);
        }
        if (push(open, n_open, left, j)) take_open();
    };
    const float X = m.g0 * 8796093022208.0f;  // bounds |x|_1, scaled: g0 >= 2^-43 of its largest
    float4 oh, ol;
    split_coordinate(xo, m.scale, oh.x, ol.x);
    split_coordinate(yo, m.scale, oh.y, ol.y);
    split_coordinate(zo, m.scale, oh.z, ol.z);
    for (int64_t s0 = tid - lane; s0 < n_sample; s0 += nt) {
        int32_t j = -1;
        bool is_far = false, is_open = false;
        if (s0 + lane < n_sample) {
            const float4 h = __ldg(sp + 2 * (s0 + lane)), l = __ldg(sp + 2 * (s0 + lane) + 1);
            j = __float_as_int(h.w);
            if (j >= 0 && j != o) {
                float a, b, c;
                int32_t pix;
                is_far = !split_direction(h, l, oh, ol, X, a, b, c);
                if (!is_far) {
                    is_open = !vec2pix_nest_f(lmax, a, b, c, pix);
                    if (!is_open) atomicAdd(&hist[lmax][pix], 1u);
                }
            }
        }
        if (push(open, n_open, is_open, j)) take_open();
        if (push(far, n_far, is_far, j)) {
            n_far -= 32;
            const int32_t q = far[n_far + lane];
            __syncwarp();
            take_far(true, q);
        }
    }
    take_far(lane < n_far, lane < n_far ? far[lane] : 0);
    if (lane < n_open) exact(open[lane]);
    __syncthreads();
    for (int l = lmax - 1; l >= lmin; --l) {
        const int32_t np = int32_t(int64_t(12) << (2 * l));
        for (int32_t q = tid; q < np; q += nt)
            hist[l][q] = hist[l + 1][4 * q] + hist[l + 1][4 * q + 1] + hist[l + 1][4 * q + 2] +
                         hist[l + 1][4 * q + 3];
        __syncthreads();
    }
    int32_t ncand = n_pairs_lmin;
    for (int32_t c = tid; c < ncand; c += nt) cand[c] = pairs_lmin[c];
    __syncthreads();
    for (int l = lmin; l < lmax; ++l) {
        const int32_t *al = anti + level_offset(l);
        const int32_t *an = anti + level_offset(l + 1);
        for (int32_t c = tid; c < ncand; c += nt) score[c] = hist[l][cand[c]] + hist[l][al[cand[c]]];
        __syncthreads();
        const int32_t half = ncand / 2;
        for (int32_t c = tid; c < ncand; c += nt) {
            const uint32_t sc = score[c], pc = cand[c];
            int32_t rank = 0;
            for (int32_t c2 = 0; c2 < ncand; ++c2)
                rank += (score[c2] > sc) || (score[c2] == sc && cand[c2] < pc);
            if (rank >= half) {
                const int32_t slot = atomicAdd(&nout, 1);
                if (slot < cmax) out[slot] = (uint32_t(l) << 28) | pc;
            } else {
                for (int ch = 0; ch < 4; ++ch) {
                    const uint32_t cp = 4 * pc + ch, ap = uint32_t(an[cp]);
                    next[4 * rank + ch] = cp < ap ? cp : ap;
                }
            }
        }
        __syncthreads();
        ncand = 4 * half;
        for (int32_t c = tid; c < ncand; c += nt) cand[c] = next[c];
        __syncthreads();
    }
    for (int32_t c = tid; c < ncand; c += nt) {
        const int32_t slot = atomicAdd(&nout, 1);
        if (slot < cmax) out[slot] = (uint32_t(lmax) << 28) | cand[c];
    }
    __syncthreads();
    if (nout != npairs) {
        if (tid == 0) dev_fail(status, kDevBadInput);
        return;
    }
    for (int32_t i = tid; i < npairs; i += nt) {
        const uint32_t v = out[i];
        int32_t rank = 0;
        for (int32_t j = 0; j < npairs; ++j) rank += out[j] < v;
        rays[int64_t(o) * npairs + rank] = v;
    }
}

}  // namespace

void launch_eval_atan2(const float *x, int64_t n, float *y, cudaStream_t st) {
    if (n <= 0) return;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_eval_atan2<<<unsigned(blocks), 256, 0, st>>>(x, n, y);
}

float atan2_bound() { return kAtanErr; }

void launch_rays_fixed(int32_t n, int32_t level, int32_t npairs, const uint32_t *pairs, uint32_t *rays,
                       cudaStream_t st) {
    const int64_t tot = int64_t(n) * npairs;
    const int tb = 256;
    k_rays_fixed<<<unsigned((tot + tb - 1) / tb), tb, 0, st>>>(n, level, npairs, pairs, rays);
}

void launch_rays_adaptive(const DevMesh &m, int32_t lmin, int32_t lmax, int32_t npairs, int64_t n_sample,
                          const int32_t *sample, float4 *split, const int32_t *anti, const uint32_t *pairs_lmin,
                          int32_t n_pairs_lmin, uint32_t *rays, int *status, cudaStream_t st) {
    int64_t words = 0;
    for (int l = lmin; l <= lmax; ++l) words += int64_t(12) << (2 * l);
    const int64_t cmax = (int64_t(12) << (2 * lmax)) / 2;
    words += 4 * cmax;
    const size_t smem = size_t(words) * sizeof(uint32_t);
    cudaFuncSetAttribute(k_rays_adaptive, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (n_sample > 0) k_split_sample<<<unsigned((n_sample + 127) / 128), 128, 0, st>>>(m, n_sample, sample, split);
    k_rays_adaptive<<<unsigned(m.n), 256, smem, st>>>(m, lmin, lmax, npairs, n_sample, split, anti,
                                                      pairs_lmin, n_pairs_lmin, rays, status);
}

}  // namespace mgx
