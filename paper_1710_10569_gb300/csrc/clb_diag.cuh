// clb_diag.cuh -- the FP64 diagnostics of one lattice and of batched lattices: the Nusselt number of
// Eq. 29 and the steady-state residual, as fixed-order sums of per-node terms, and the residual's
// snapshot. Kept apart from the step kernels (clb_kernels.cuh), which they only read.
#pragma once

#include "clb_kernels.cuh"

namespace clb {

constexpr int kReduceThreads = 256;

// A float as a double, exactly, by its bits: a conversion instruction takes the FP64 pipe as long as
// an addition does (64 clocks per warp and SM quarter), the integer instructions here a third of that.
__device__ __forceinline__ double widen(double v) { return v; }
__device__ __forceinline__ double widen(float v)
{
    const int b = __float_as_int(v);
    const int e = b & 0x7f800000, sign = b & (int)0x80000000;
    if (e == 0) return v == 0.0f ? __hiloint2double(sign, 0) : double(v);  // (subnormal numbers: rare)
    const int hi = ((b & 0x7fffffff) >> 3) + (e == 0x7f800000 ? 0x7ff00000 - (0x7f800000 >> 3) : 0x38000000);
    return __hiloint2double(sign | hi, b << 29);
}

// Fixed-order block sum of RS_N doubles (the same order for every launch shape of the step): out[k]
// (shared or global memory) is written by thread k, and not visible to the others. Within a warp the
// sums of lanes 16, 8, 4, 2, 1 apart are shared out: at each level a lane keeps some of its values,
// adds its partner's to them and hands over the others, so that a warp makes 8 FP64 additions instead
// of 30 for the same pairs. The warps' sums are then added in order, one value per thread.
__device__ __forceinline__ void block_sum(double v[RS_N], double* out)
{
    static_assert(RS_N == 6, "the exchange below is laid out for six values");
    __shared__ double sh[kReduceThreads / 32][RS_N];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned all = 0xffffffffu;
    const bool h = lane & 16, q = lane & 8, p = lane & 4;
    // lower half: values 0-2, upper half: 3-5
    double s[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) s[k] = (h ? v[k + 3] : v[k]) + __shfl_xor_sync(all, h ? v[k] : v[k + 3], 16);
    // of these three, the lanes without bit 8 keep the first two, the others the third
    const double t0 = (q ? s[2] : s[0]) + __shfl_xor_sync(all, q ? s[0] : s[2], 8);
    const double t1 = s[1] + __shfl_xor_sync(all, s[1], 8);
    // of two, the lanes without bit 4 keep the first, the others the second; a third stays in both
    const bool second = !q && p;
    double r = (second ? t1 : t0) + __shfl_xor_sync(all, q || p ? t0 : t1, 4);
    r += __shfl_xor_sync(all, r, 2);
    r += __shfl_xor_sync(all, r, 1);
    if ((lane & 3) == 0 && !(q && p)) sh[warp][(h ? 3 : 0) + (q ? 2 : p ? 1 : 0)] = r;
    __syncthreads();
    if (threadIdx.x < RS_N) {
        double t = 0.0;
        for (int w = 0; w < kReduceThreads / 32; ++w) t += sh[w][threadIdx.x];
        out[threadIdx.x] = t;
    }
}

// The Nusselt term u_axis (T - T0) of one node (Eq. 29), in the arithmetic precision A; T is
// returned through T_out.
template <typename A, typename S>
__device__ __forceinline__ A nu_term(const LatParams<S>& P, const Macro<A>& m, int axis, A& T_out)
{
    T_out = m.T;
    return (axis == 0 ? m.ux : m.uy) * (m.T - A(P.T0));
}

// One node's terms of the diagnostics sums, added to v: the fields come from the pulled populations,
// the terms are formed in the arithmetic precision A (FP64 for FP64 storage, FP32 for the FP32 and
// FP16 forms, whose fields are FP32 values) and accumulated in FP64. The residual's snapshot is kept
// in A as well: it holds those same values exactly, and GB300 issues FP64 instructions (the
// conversions included) slowly enough that they bound this pass. With update != 0 the node's
// snapshot entries are replaced by the current fields. The Nusselt term is weighted by wet_weight
// (wet-wall rows and columns count half: the trapezoid rule over [0, H]; 1, 1/2 and 1/4 scale
// exactly in A). Non-finite nodes are counted in nbad.
template <typename E, typename A>
__device__ __forceinline__ void node_diag(const E* __restrict__ src, const LatParams<A>& P, int x, int y,
                                          int axis, A* __restrict__ snap, int update, double v[RS_N], int& nbad)
{
    const long long N = (long long)P.nx * P.ny;
    A f[9], g[5];
    gather(src, P, x, y, f, g);
    const Macro<A> m = macroscopic(P, f, g, row_base(P, y));
    A T;
    const A q = nu_term(P, m, axis, T);
    const long long n = (long long)y * P.nx + x;
    const A dux = m.ux - snap[n], duy = m.uy - snap[N + n], dT = T - snap[2 * N + n];
    v[RS_UT] += widen(q * A(wet_weight(P, x, y)));
    v[RS_DU] += widen(dux * dux + duy * duy);
    v[RS_U] += widen(m.ux * m.ux + m.uy * m.uy);
    v[RS_DT] += widen(dT * dT);
    v[RS_T] += widen(T * T);
    nbad += (isfinite(m.ux) && isfinite(m.uy) && isfinite(T) && isfinite(m.rho)) ? 0 : 1;
    if (update) {
        snap[n] = m.ux;
        snap[N + n] = m.uy;
        snap[2 * N + n] = T;
    }
}

// The residual's snapshot of the current fields (u_x, u_y, T as A [3][ny][nx]), as node_diag keeps it.
template <int ST>
__global__ void k_snap(const typename Storage<ST>::T* __restrict__ src, const LatParams<typename Storage<ST>::A> P,
                       typename Storage<ST>::A* __restrict__ snap)
{
    using A = typename Storage<ST>::A;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    A f[9], g[5];
    gather(src, P, x, y, f, g);
    const Macro<A> m = macroscopic(P, f, g, row_base(P, y));
    const long long n = (long long)y * P.nx + x, N = (long long)P.nx * P.ny;
    snap[n] = m.ux;
    snap[N + n] = m.uy;
    snap[2 * N + n] = m.T;
}

// Per-row FP64 partial sums for the diagnostics: sum u_axis (T - T0), sum |u - u_snap|^2,
// sum |u|^2, sum (T - T_snap)^2, sum T^2 and the count of non-finite nodes. One block of
// kReduceThreads per row y; threads stride over x in a fixed order, so the sums do not depend on
// how the step kernel is launched. With update != 0 the snapshot (u_x, u_y, T as double
// [3][ny][nx]) is replaced by the current fields. (The batched lattices use this form; a single
// lattice uses the row-segment form below.)
template <typename E, typename A>
__device__ __forceinline__ void reduce_row(const E* __restrict__ src, const LatParams<A>& P, int y,
                                           int axis, A* __restrict__ snap, int update,
                                           double* __restrict__ partial_row)
{
    double v[RS_N] = {0, 0, 0, 0, 0, 0};
    int nbad = 0;
    for (int x = threadIdx.x; x < P.nx; x += kReduceThreads) node_diag(src, P, x, y, axis, snap, update, v, nbad);
    v[RS_BAD] = double(nbad);
    block_sum(v, partial_row);
}

// The same sums over row segments of kDiagNodes = kReduceThreads * 8 nodes: block b covers segment
// seg of row y (b = y * nseg + seg), each thread sums its 8 nodes x = seg * kDiagNodes + t + 256 k in
// order, then the shuffle tree within each warp and the warps in order give partial[b]. The per-node
// sums are FP64 and GB300 issues FP64 slowly, so each thread takes 8 nodes (the warp tree's
// FP64 adds per thread are shared by 8 nodes); the register cap keeps 4 blocks per SM so that
// enough gathers are in flight. For nx <= kDiagNodes the order is that of reduce_row. The FP64 pipe
// bounded it: per node 5 additions for the FP32 and FP16 forms (10 instructions while the terms were
// converted by it) and 1 per node for the tree (4 before the exchange in block_sum). It is 50% busy
// now, DRAM 46%, and the wait for the gathers is what is left. A whole check takes 72.6 us on
// 2048 x 1024 FP32 nodes (103.0 before both, 78.9 with the final sum as it was), 204 on 4096 x 2048 FP16
// (304, 213). With 5 blocks per SM: 77.4 and 205.
constexpr int kDiagNodes = kReduceThreads * 8;

template <int ST>
__global__ void __launch_bounds__(kReduceThreads, 4) k_reduce_nodes(
    const typename Storage<ST>::T* __restrict__ src, const LatParams<typename Storage<ST>::A> P,
    int axis, typename Storage<ST>::A* __restrict__ snap, int update, double* __restrict__ partial, int nseg)
{
    step_prologue();
    const int seg = blockIdx.x % nseg, y = blockIdx.x / nseg;
    const int x0 = seg * kDiagNodes, x1 = min(P.nx, x0 + kDiagNodes);
    double v[RS_N] = {0, 0, 0, 0, 0, 0};
    int nbad = 0;
    for (int x = x0 + threadIdx.x; x < x1; x += kReduceThreads) node_diag(src, P, x, y, axis, snap, update, v, nbad);
    v[RS_BAD] = double(nbad);
    block_sum(v, partial + (long long)blockIdx.x * RS_N);
}

// Sum the per-row partials in row order and finish the diagnostics in FP64: out[0..RS_N-1] = the
// sums, out[RS_N] = Nu (Eq. 29), out[RS_N+1] = E_R. One block, all latency: FP64 divisions and square
// roots are long chains of slow instructions, so the two parts of E_R are formed by two lanes of one
// warp and Nu by another warp. out may be pinned host memory, which spares the host a copy after the
// kernel: it is written once, by neighbouring threads. A whole check, with the kernels also chained to the one
// before: 513 x 385 FP32 31.5 -> 26.0 us, 256 x 256 FP64 38.1 -> 28.4, 60 x 31 FP64 28.0 -> 21.7.
__device__ __forceinline__ void reduce_final(const double* __restrict__ partial, int rows,
                                             double nodes, double cells, double H, double dT,
                                             double sign, double kappa, double u_ref, double dT_ref,
                                             double* __restrict__ out)
{
    double v[RS_N] = {0, 0, 0, 0, 0, 0};
    for (int r = threadIdx.x; r < rows; r += kReduceThreads)
        for (int k = 0; k < RS_N; ++k) v[k] += partial[(long long)r * RS_N + k];
    __shared__ double tot[RS_N + 2];
    block_sum(v, tot);
    __syncthreads();
    const int t = threadIdx.x;
    if (t < 2) {
        const double r = residual_of(tot[t == 0 ? RS_DU : RS_DT], tot[t == 0 ? RS_U : RS_T], nodes, t == 0 ? u_ref : dT_ref);
        const double rt = __shfl_down_sync(0x3u, r, 1);
        if (t == 0) tot[RS_N + 1] = r > rt ? r : rt;
    } else if (t == 32) {
        tot[RS_N] = nusselt_of(tot[RS_UT], cells, H, dT, sign, kappa);
    }
    __syncthreads();
    if (t < RS_N + 2) out[t] = tot[t];
}

static __global__ void __launch_bounds__(kReduceThreads) k_reduce_final(const double* __restrict__ partial,
                                                                 int rows, double nodes, double cells,
                                                                 double H, double dT, double sign,
                                                                 double kappa, double u_ref,
                                                                 double dT_ref, double* __restrict__ out)
{
    step_prologue();
    reduce_final(partial, rows, nodes, cells, H, dT, sign, kappa, u_ref, dT_ref, out);
}

}  // namespace clb
