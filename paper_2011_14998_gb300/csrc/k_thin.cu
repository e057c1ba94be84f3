// k_thin.cu -- thinning with keep-probabilities weighted by a score (the
// learned reduction's prediction), in the spirit of the random thinning that
// replaces re-meshing (Section 2.2.2): point i is kept when
//   u_i < min(1, c w_i),   w_i = 10^(alpha y_i),
// y_i the predicted log10 J error if i is dropped, u_i the SplitMix64 uniform
// of (seed, i), and c the scale at which the expected kept count
// sum_i min(1, c w_i) equals the target.  Unlike keeping the top-ranked points,
// every region keeps some points.
#include "mgx_internal.cuh"

namespace mgx {

namespace {

__global__ void k_thin_weights(const float *__restrict__ y, int64_t n, float alpha, float *__restrict__ w) {
    const int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    if (i >= n) return;
    float e = alpha * y[i] * 3.3219280948873622f;  // log2(10)
    e = fminf(fmaxf(e, -100.0f), 100.0f);
    w[i] = exp2f(e);
}

// One Newton step towards the scale c at which S(c) = sum_i min(1, c w_i)
// equals the target.  S is piecewise linear, increasing and concave, so from
// c = target / sum w, which is not above the root, the steps
//   c' = (target - #{c w_i >= 1}) / sum_{c w_i < 1} w_i
// rise to it and end there exactly, once the saturated set stays the same
// (typically 5 to 15 steps).  The last block to finish takes the step, so the
// host neither waits between steps nor chooses their number; a finished solve
// lets further launches return at once.  (Bisection from the host, 80 passes
// with a copy back each, took 2.1 ms for 200 000 points.)
__global__ void k_thin_newton(const float *__restrict__ w, int64_t n, double target, ThinSolve *__restrict__ s) {
    if (s->done) return;
    const double c = s->c;
    double acc = 0.0;
    unsigned long long sat = 0;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const double x = double(w[i]);
        if (c * x < 1.0) acc += x;
        else ++sat;
    }
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) {
        acc += __shfl_down_sync(0xffffffffu, acc, sh);
        sat += __shfl_down_sync(0xffffffffu, sat, sh);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&s->sum, acc);
        if (sat) atomicAdd(&s->sat, sat);
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x != 0 || atomicAdd(&s->blocks, 1u) != gridDim.x - 1) return;
    __threadfence();
    const double sum = *(volatile double *)&s->sum;
    const unsigned long long k = *(volatile unsigned long long *)&s->sat;
    const double next = (target - double(k)) / sum;
    if (!(sum > 0.0) || !(next > c)) {
        s->done = 1;  // at the root (or, by rounding, an ulp beside it)
    } else {
        s->c = next;
        if (s->steps > 0 && k == s->last) s->done = 1;  // the same saturated points: next is the root
    }
    s->last = k;
    s->steps += 1;
    s->sum = 0.0;
    s->sat = 0;
    s->blocks = 0;
    __threadfence();
}

__global__ void k_thin_mark(const float *__restrict__ w, int64_t n, double c, uint64_t seed,
                            uint8_t *__restrict__ keep, unsigned long long *__restrict__ kept) {
    unsigned long long cnt = 0;
    for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const double p = __dmul_rn(c, double(w[i]));
        const uint8_t k = splitmix_uniform(seed, i) < (p < 1.0 ? p : 1.0) ? 1 : 0;
        keep[i] = k;
        cnt += k;
    }
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) cnt += __shfl_down_sync(0xffffffffu, cnt, sh);
    if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(kept, cnt);
}

unsigned thin_grid(int64_t n) {
    int64_t g = (n + 255) / 256;
    if (g > 152 * 8) g = 152 * 8;
    return unsigned(g < 1 ? 1 : g);
}

}  // namespace

void launch_thin_weights(const float *y, int64_t n, float alpha, float *w, cudaStream_t st) {
    if (n > 0) k_thin_weights<<<unsigned((n + 255) / 256), 256, 0, st>>>(y, n, alpha, w);
}

void launch_thin_newton(const float *w, int64_t n, double target, ThinSolve *s, cudaStream_t st) {
    if (n > 0) k_thin_newton<<<thin_grid(n), 256, 0, st>>>(w, n, target, s);
}

void launch_thin_mark(const float *w, int64_t n, double c, uint64_t seed, uint8_t *keep, unsigned long long *kept,
                      cudaStream_t st) {
    cudaMemsetAsync(kept, 0, sizeof(unsigned long long), st);
    if (n > 0) k_thin_mark<<<thin_grid(n), 256, 0, st>>>(w, n, c, seed, keep, kept);
}

}  // namespace mgx
