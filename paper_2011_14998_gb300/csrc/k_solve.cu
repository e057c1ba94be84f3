// k_solve.cu -- the second-order instantiation of the formal solution
// (k_solve_impl.cuh) and the dispatch on the scheme's order; the Hermitian
// instantiation is compiled separately (k_solve_herm.cu).
#include "k_solve_impl.cuh"

namespace mgx {

// Bins per lane: 2 when there are more bins than lanes (the frequency-independent
// work is then shared by two bins; the double-precision Hermitian form has one),
// 4 in the single-precision second-order form of one line when that takes no
// more bin slots than 2, else 1.
int solve_bins_per_lane(int precision, int order, int32_t n_lines, int32_t n_bins) {
    if (precision == MGX_FP64 && order == 4) return 1;
    if (precision == MGX_FP32 && order != 4 && n_lines == 1 && (n_bins + 127) / 128 * 2 == (n_bins + 63) / 64) return 4;
    return n_bins > 32 ? 2 : 1;
}

// Warps per origin and tile.  A warp takes all pairs of an item one after the
// other, which leaves the chip idle when there are few items, and its last wave
// nearly empty when there are a few waves: with fewer items than about four
// waves of warps (a line on their number, 152 SMs with 28 warps in single
// precision and 16 in the forms with double; the forms hold 12 to 36)
// the pairs of an item are dealt to several warps, which store u, and J is
// summed from u in the same order (400 points, 33 pairs: 1.95 -> 0.34 ms;
// 12 000 points, 96 pairs, Hermitian: 50.8 -> 48.2 ms; 4001 points in double
// precision 194 -> 165 ms).  Not when u would take more than a GiB.
int32_t solve_parts(int precision, int64_t n_items, int32_t npairs, size_t u_bytes) {
    const int64_t want = int64_t(4) * 152 * (precision == MGX_FP32 ? 28 : 16);
    if (n_items <= 0 || n_items >= want || u_bytes > (size_t(1) << 30)) return 1;
    const int64_t parts = (want + n_items - 1) / n_items;
    return int32_t(parts < npairs ? parts : npairs);
}

namespace {

// J = sum of 2 w u over the pairs in ascending order, Neumaier's compensated sum.
__global__ void k_sum_pairs(const __grid_constant__ DevRays R, const __grid_constant__ SolveArgs a, int32_t n_bins) {
    const int64_t t = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
    const int64_t oc = t / n_bins;
    if (oc >= a.o_end - a.o_begin) return;
    const int32_t b = int32_t(t - oc * n_bins);
    const uint32_t *rays = R.rays + (a.o_begin + oc) * R.npairs;
    const double *u = a.u_out + oc * R.npairs * n_bins + b;
    double sum = 0.0, comp = 0.0;
    for (int32_t p = 0; p < R.npairs; ++p) {
        const double x = a.w2[rays[p] >> 28] * u[int64_t(p) * n_bins];
        const double t2 = sum + x;
        comp += fabs(sum) >= fabs(x) ? (sum - t2) + x : (x - t2) + sum;
        sum = t2;
    }
    a.J[(a.o_begin + oc) * n_bins + b] = sum + comp;
}

}  // namespace

void launch_sum_pairs(const DevRays &R, const SolveArgs &a, int32_t n_bins, cudaStream_t st) {
    const int64_t n = int64_t(a.o_end - a.o_begin) * n_bins;
    if (n > 0) k_sum_pairs<<<unsigned((n + 127) / 128), 128, 0, st>>>(R, a, n_bins);
}

template void launch_solve_ord<2>(const DevMesh &, const DevLines &, const DevRays &, const SolveArgs &, int,
                                  cudaStream_t);
template void launch_solve_queue_ord<2>(int, int, int, const BatchSlot *, const uint2 *, int64_t,
                                        unsigned long long *, cudaStream_t);
extern template void launch_solve_ord<4>(const DevMesh &, const DevLines &, const DevRays &, const SolveArgs &, int,
                                         cudaStream_t);
extern template void launch_solve_queue_ord<4>(int, int, int, const BatchSlot *, const uint2 *, int64_t,
                                               unsigned long long *, cudaStream_t);

void launch_solve(const DevMesh &m, const DevLines &Ln, const DevRays &R, const SolveArgs &a, int precision,
                  int order, cudaStream_t st) {
    if (order == 4) launch_solve_ord<4>(m, Ln, R, a, precision, st);
    else launch_solve_ord<2>(m, Ln, R, a, precision, st);
}

void launch_solve_queue(int precision, int order, int bins_per_lane, int max_lines, const BatchSlot *slots,
                        const uint2 *work, int64_t n_work, unsigned long long *next, cudaStream_t st) {
    if (order == 4) launch_solve_queue_ord<4>(precision, bins_per_lane, max_lines, slots, work, n_work, next, st);
    else launch_solve_queue_ord<2>(precision, bins_per_lane, max_lines, slots, work, n_work, next, st);
}

}  // namespace mgx
