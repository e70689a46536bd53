// clb_thermal.cu -- the D2Q5 central-moment equation alone with a prescribed velocity field
// (include/clb.h: clb_thermal_*). Sec. 3.1 of the paper solves only the D2Q5 equation for a given
// velocity; this is that mode, for convection-diffusion of a passive scalar. Per node and step:
// pull the 5 temperature populations (Eq. 22, the same wall rules as the coupled step), read the
// node's velocity, collide (Eqs. 16-21), store. The collision is the same device function as the
// coupled step's D2Q5 part.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "clb_march.cuh"

using namespace clb;

namespace {

constexpr int NT = 5;  // planes per buffer

// Two consecutive elements loaded or stored as one aligned access.
template <typename E>
struct alignas(2 * sizeof(E)) Pair {
    E e[2];
};

// Velocity storage of the thermal handle: the arithmetic type of the storage.
template <int ST>
using VelT = typename Storage<ST>::A;

template <typename A>
__device__ __forceinline__ void thermal_slots(const LatParams<A>& P, int x, int y, long long idx[NT], int& mask)
{
    const bool inL = P.per_x || x > 0;
    const bool inR = P.per_x || x < P.nx - 1;
    const bool inB = P.per_y || y > 0;
    const bool inT = P.per_y || y < P.ny - 1;
    const int xm = x > 0 ? x - 1 : P.nx - 1;
    const int xp = x < P.nx - 1 ? x + 1 : 0;
    const long long r0 = (long long)y * P.pitch;
    const long long rm = (long long)(y > 0 ? y - 1 : P.ny - 1) * P.pitch;
    const long long rp = (long long)(y < P.ny - 1 ? y + 1 : 0) * P.pitch;
    const long long here = r0 + x;
    const long long pl = P.plane;
    idx[0] = here;
    idx[1] = inL ? 1 * pl + r0 + xm : 3 * pl + here;
    idx[2] = inB ? 2 * pl + rm + x : 4 * pl + here;
    idx[3] = inR ? 3 * pl + r0 + xp : 1 * pl + here;
    idx[4] = inT ? 4 * pl + rp + x : 2 * pl + here;
    mask = (inL ? 0 : 1) | (inR ? 0 : 2) | (inB ? 0 : 4) | (inT ? 0 : 8);
}

template <typename E, typename A>
__device__ __forceinline__ void thermal_gather(const E* __restrict__ src, const LatParams<A>& P, int x, int y, A g[NT])
{
    long long idx[NT];
    int mask;
    thermal_slots(P, x, y, idx, mask);
#pragma unroll
    for (int i = 0; i < NT; ++i) g[i] = to_a(src[idx[i]]);
    // g2 (g4) pulled from the row below (above) is re-based to this row; bounced values are not
    g[2] = (mask & 4) ? g[2] : g[2] - P.T_dyw;
    g[4] = (mask & 8) ? g[4] : g[4] + P.T_dyw;
    if (mask) {
        if ((mask & 1) && P.kind[0] == WALL_DIRICHLET) g[1] = P.Tw_c2[0] - g[1];
        if ((mask & 2) && P.kind[1] == WALL_DIRICHLET) g[3] = P.Tw_c2[1] - g[3];
        if ((mask & 4) && P.kind[2] == WALL_DIRICHLET) g[2] = P.Tw_c2[2] - g[2];
        if ((mask & 8) && P.kind[3] == WALL_DIRICHLET) g[4] = P.Tw_c2[3] - g[4];
    }
}

// D2Q5 equilibrium g^eq(T, u) in stored form (minus w^T T_b(y) for deviation storage; dT = T - T_b(y)).
template <bool DEV, typename A>
__device__ __forceinline__ void thermal_eq(const LatParams<A>& P, A T, A dT, A u, A v, A g[NT])
{
    if constexpr (DEV) eq_dev_d2q5(T, dT, u, v, P.cs2T, g);
    else back_d2q5(T, A(0), A(0), T * P.cs2T, T * P.cs2T, u, v, g);
}

// Pulled populations of node (x, y) with the wall rules, including wet walls: a node on a wet
// wall takes g_i = g^eq_i(T_w, u) + [g_i(q) - g^eq_i(T(q), u(q))] from the fluid node q next to it
// (along the normal; the diagonal neighbour at a corner, where T_w is the mean of the two walls'
// temperatures), u being the prescribed velocity of each node (the paper's non-equilibrium
// extrapolation, Sec. 3).
template <bool DEV, typename E, typename A, typename VT>
__device__ __forceinline__ void thermal_gather_node(const E* __restrict__ src, const LatParams<A>& P,
                                                    const VT* __restrict__ ux, const VT* __restrict__ uy,
                                                    int x, int y, A g[NT])
{
    const bool onx = P.wet_x && (x == 0 || x == P.nx - 1);
    const bool ony = P.wet_y && (y == 0 || y == P.ny - 1);
    if (!onx && !ony) {
        thermal_gather(src, P, x, y, g);
        return;
    }
    const int qx = onx ? (x == 0 ? 1 : x - 1) : x, qy = ony ? (y == 0 ? 1 : y - 1) : y;
    const int side_x = x == 0 ? 0 : 1, side_y = y == 0 ? 2 : 3;
    const A Tw = (onx && ony) ? A(0.5) * (P.Twall[side_x] + P.Twall[side_y]) : P.Twall[ony ? side_y : side_x];
    const A dTw = (onx && ony) ? Tw - P.T_b : P.dTw[ony ? side_y : side_x];
    A gq[NT], eq_q[NT], eq_b[NT];
    thermal_gather(src, P, qx, qy, gq);
    const A dTq = (gq[0] + gq[1]) + (gq[2] + gq[3]) + gq[4];
    const long long nq = (long long)qy * P.nx + qx, nb = (long long)y * P.nx + x;
    thermal_eq<DEV>(P, row_base(P, qy) + dTq, dTq, A(ux[nq]), A(uy[nq]), eq_q);
    thermal_eq<DEV>(P, Tw, dTw, A(ux[nb]), A(uy[nb]), eq_b);
#pragma unroll
    for (int i = 0; i < NT; ++i) g[i] = eq_b[i] + (gq[i] - eq_q[i]);
}

// One node's collision (Eqs. 16-21) with its prescribed velocity.
template <int ST>
__device__ __forceinline__ void thermal_collide(const LatParams<typename Storage<ST>::A>& P,
                                                typename Storage<ST>::A u, typename Storage<ST>::A v,
                                                typename Storage<ST>::A g[NT], typename Storage<ST>::A Tb)
{
    using A = typename Storage<ST>::A;
    if constexpr (Storage<ST>::DEV) {
        const A dT = (g[0] + g[1]) + (g[2] + g[3]) + g[4];
        collide_d2q5_dev(P, Tb + dT, dT, u, v, g);
    } else {
        const double s1 = g[1] + g[3], d1 = g[1] - g[3], s2 = g[2] + g[4], d2 = g[2] - g[4];
        collide_d2q5(P, g[0] + (s1 + s2), u, v, s1, d1, s2, d2, g);
    }
}

// One time step, two neighbouring nodes x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x) and x0 + 1
// of row y = blockIdx.y per thread. A pair whose pulls all stay inside the lattice without wrapping
// reads the planes pulled along y (and the rest plane) as aligned pairs and stores every plane as
// an aligned pair; other pairs (next to a wall or a periodic seam, or the single node at the end of
// an odd row) gather node by node with the wall rules. The values are those of the node-by-node
// path.
template <int ST>
__global__ void __launch_bounds__(128, ST == ST_F64 ? 8 : 12) k_thermal_step(const typename Storage<ST>::T* __restrict__ src,
                                                      typename Storage<ST>::T* __restrict__ dst,
                                                      const VelT<ST>* __restrict__ ux,
                                                      const VelT<ST>* __restrict__ uy,
                                                      const LatParams<typename Storage<ST>::A> P)
{
    using A = typename Storage<ST>::A;
    using E = typename Storage<ST>::T;
    step_prologue();
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int y = blockIdx.y;
    if (x0 >= P.nx) return;
    const bool two = x0 + 1 < P.nx;
    const long long pl = P.plane;
    const long long here = (long long)y * P.pitch + x0;
    const long long n = (long long)y * P.nx + x0;
    A ga[NT], gb[NT];
    if (two && x0 > 0 && x0 + 2 < P.nx && y > 0 && y + 1 < P.ny) {
        const Pair<E> c0 = *reinterpret_cast<const Pair<E>*>(src + here);
        const Pair<E> c2 = *reinterpret_cast<const Pair<E>*>(src + 2 * pl + here - P.pitch);
        const Pair<E> c4 = *reinterpret_cast<const Pair<E>*>(src + 4 * pl + here + P.pitch);
        ga[0] = to_a(c0.e[0]);
        gb[0] = to_a(c0.e[1]);
        ga[1] = to_a(src[pl + here - 1]);
        gb[1] = to_a(src[pl + here]);
        ga[2] = to_a(c2.e[0]);
        gb[2] = to_a(c2.e[1]);
        ga[3] = to_a(src[3 * pl + here + 1]);
        gb[3] = to_a(src[3 * pl + here + 2]);
        ga[4] = to_a(c4.e[0]);
        gb[4] = to_a(c4.e[1]);
        // re-based to this row (see thermal_gather)
        ga[2] = ga[2] - P.T_dyw;
        gb[2] = gb[2] - P.T_dyw;
        ga[4] = ga[4] + P.T_dyw;
        gb[4] = gb[4] + P.T_dyw;
    } else {
        thermal_gather_node<Storage<ST>::DEV>(src, P, ux, uy, x0, y, ga);
        if (two) thermal_gather_node<Storage<ST>::DEV>(src, P, ux, uy, x0 + 1, y, gb);
    }
    const A Tb = row_base(P, y);
    thermal_collide<ST>(P, A(ux[n]), A(uy[n]), ga, Tb);
    if (two) {
        thermal_collide<ST>(P, A(ux[n + 1]), A(uy[n + 1]), gb, Tb);
        // here is even (x0 and the row pitch are): one aligned pair per plane
#pragma unroll
        for (int i = 0; i < NT; ++i) {
            Pair<E> o;
            o.e[0] = from_a(ga[i], (E*)nullptr);
            o.e[1] = from_a(gb[i], (E*)nullptr);
            *reinterpret_cast<Pair<E>*>(dst + i * pl + here) = o;
        }
    } else {
#pragma unroll
        for (int i = 0; i < NT; ++i) dst[i * pl + here] = from_a(ga[i], (E*)nullptr);
    }
}

// ---------------------------------------------------------------------------------------------
// kSteps time steps per launch (FP32 and FP16 forms, large lattices). One step moves 48 bytes a node
// (FP32: 5 populations in and out, the velocity in) for some 45 operations and runs at the copy
// bandwidth; what can give is the bytes per step. As in the coupled lattice's two-step kernel
// (clb_march.cuh) a warp takes a window of 64 columns, two nodes per lane, and marches along y: level
// k of the pipeline computes step k + 1 of row r - k from the rows that level k - 1 has just left. Here
// a level hands on five populations only, so the rows between levels stay in registers (the
// velocities, read once, in shared-memory slots private to the thread). Each step loses the outermost
// column of the window (of 64 columns the inner 56 are stored) and a row at either end of the segment.
// The arithmetic of a node is that of k_thermal_step, with the intermediate states rounded to the
// storage type: bitwise the same. Measured on 4096 x 4096 (us per step, one step per launch -> four):
// FP32 117.2 -> 45.9 (365 GLUPS), FP16 90.0 -> 47.8. It is then bound by the latency of a turn, whose
// levels follow one another (some 110 instructions per pair of nodes and level, 45 of them packed
// arithmetic, at 24 warps per SM). Tried: turns unrolled by two and four, which saves the moves of the
// handed-on rows but takes 120 registers (51.8 at 16 warps per SM); the next row loaded a turn
// ahead (54.2); velocities in registers (54.4).
constexpr int kSteps = 4;                       // a power of two
constexpr int kMarchOutT = 64 - 4 * ((kSteps + 1) / 2);
constexpr int kLanesLost = (kSteps + 1) / 2;    // lanes at either end of a window that store nothing
constexpr int kResidentT = 24;                  // warps per SM that the register bound of k_thermal_steps leaves

__device__ __forceinline__ F2 load_pair(const float* p)
{
    F2 r;
    r.u = *reinterpret_cast<const unsigned long long*>(p);
    return r;
}
__device__ __forceinline__ F2 load_pair(const __half* p)
{
    const __half2 h = *reinterpret_cast<const __half2*>(p);
    return F2(__low2float(h), __high2float(h));
}
__device__ __forceinline__ void store_pair(float* p, F2 v) { *reinterpret_cast<unsigned long long*>(p) = v.u; }
__device__ __forceinline__ void store_pair(__half* p, F2 v)
{
    float a, b;
    v.split(a, b);
    *reinterpret_cast<__half2*>(p) = __floats2half2_rn(a, b);
}
// The values as the storage type holds them.
__device__ __forceinline__ F2 as_stored(F2 v, const float*) { return v; }
__device__ __forceinline__ F2 as_stored(F2 v, const __half*)
{
    float a, b;
    v.split(a, b);
    const __half2 h = __floats2half2_rn(a, b);
    return F2(__low2float(h), __high2float(h));
}

// Pull and collide one row of a window: before the shift along x, g[i] holds population i of this
// lane's nodes on the row it is pulled from (bounced at a y wall: the opposite one of the own row).
template <bool HI1, bool WALLS>
__device__ __forceinline__ void thermal_row(const LatParams<float>& P, F2 g[NT], const MarchWalls& w, F2 u, F2 v, float Tb)
{
    const F2 g1 = g[1], g3 = g[3];
    g[1] = pull_shr(g1);
    g[3] = pull_shl(g3);
    if (WALLS && (w.bottom || w.top || w.any_x)) {
        float a[NT], b[NT], oa, ob;
#pragma unroll
        for (int i = 0; i < NT; ++i) g[i].split(a[i], b[i]);
        g3.split(oa, ob);
        if (w.m0 & 1) a[1] = oa;
        g1.split(oa, ob);
        if (w.m0 & 2) a[3] = oa;
        if (w.m1 & 2) b[3] = ob;
        const auto rules = [&](float* q, int m) {
            q[2] = w.bottom ? q[2] : q[2] - P.T_dyw;
            q[4] = w.top ? q[4] : q[4] + P.T_dyw;
            if ((m & 1) && P.kind[0] == WALL_DIRICHLET) q[1] = P.Tw_c2[0] - q[1];
            if ((m & 2) && P.kind[1] == WALL_DIRICHLET) q[3] = P.Tw_c2[1] - q[3];
            if (w.bottom && P.kind[2] == WALL_DIRICHLET) q[2] = P.Tw_c2[2] - q[2];
            if (w.top && P.kind[3] == WALL_DIRICHLET) q[4] = P.Tw_c2[3] - q[4];
        };
        rules(a, w.m0);
        rules(b, w.m1);
#pragma unroll
        for (int i = 0; i < NT; ++i) g[i] = F2(a[i], b[i]);
    } else {
        // re-based to this row (see thermal_gather)
        g[2] = g[2] - F2(P.T_dyw);
        g[4] = g[4] + F2(P.T_dyw);
    }
    const F2 dT = (g[0] + g[1]) + (g[2] + g[3]) + g[4];
    collide_d2q5_dev<HI1>(P, F2(Tb) + dT, dT, u, v, g);
}

// What level k of the pipeline has left for level k + 1: g0, g1, g3 of its last row, g2 of its last two
// (and g4 of its last, for a bounce at the bottom wall).
struct ThermalPipe {
    F2 c0[kSteps - 1], c1[kSteps - 1], c3[kSteps - 1], up[kSteps - 1], upp[kSteps - 1], dn[kSteps - 1];
};

// kSteps steps of rows [ya, yb), columns [xo, xe) by one warp (xo even, xe - xo <= kMarchOutT, xe even or
// nx). WALLS = false: no row (ya - kSteps + 1 to yb + kSteps - 2) or column next to a wall, all columns load
// as aligned pairs.
template <int ST, bool HI1, bool WALLS>
__device__ __forceinline__ void thermal_march(const typename Storage<ST>::T* __restrict__ src,
                                              typename Storage<ST>::T* __restrict__ dst, const float* __restrict__ ux,
                                              const float* __restrict__ uy, const LatParams<float>& P, const MarchCols& M,
                                              int xo, int xe, int ya, int yb, int lane, F2* __restrict__ slots)
{
    using E = typename Storage<ST>::T;
    constexpr int L = kSteps - 1;  // rows that a segment needs beyond its own at either end, for the first step
    const int x0 = xo - 2 * kLanesLost + 2 * lane;
    const bool pairs = !WALLS || M.pairs;
    const bool vpairs = pairs && P.nx % 2 == 0;  // velocity rows are dense
    MarchWalls w = M.w;
    const bool store = lane >= kLanesLost && lane < 32 - kLanesLost && x0 < xe;
    const bool store2 = !WALLS || x0 + 1 < P.nx;
    const long long pl = P.plane;
    const auto wrap = [&](int r) { return r < 0 ? r + P.ny : r >= P.ny ? r - P.ny : r; };
    ThermalPipe S;
#pragma unroll
    for (int k = 0; k < L; ++k) S.c0[k] = S.c1[k] = S.c3[k] = S.up[k] = S.upp[k] = S.dn[k] = F2(0.0f, 0.0f);
    const auto vel = [&](int row, int c) -> F2& { return slots[((row & (kSteps - 1)) * 2 + c) * 32]; };

    // the populations that row r pulls and its velocity
    const auto load_row = [&](int r, F2 g[NT], F2& u, F2& v) {
        const int y = wrap(r);
        const bool bottom = WALLS && !P.per_y && y == 0, top = WALLS && !P.per_y && y == P.ny - 1;
        const E* sc = src + (long long)y * P.pitch;
        // across a y wall the node's own opposite plane
        const E* su = bottom ? sc + 2 * pl : src + (long long)(y > 0 ? y - 1 : P.ny - 1) * P.pitch;
        const E* sd = top ? sc - 2 * pl : src + (long long)(y < P.ny - 1 ? y + 1 : 0) * P.pitch;
        const auto load = [&](const E* p) { return pairs ? load_pair(p + M.xa) : F2(to_a(p[M.xa]), to_a(p[M.xb])); };
        g[0] = load(sc);
        g[1] = load(sc + pl);
        g[3] = load(sc + 3 * pl);
        g[2] = load(su + 2 * pl);
        g[4] = load(sd + 4 * pl);
        const long long n = (long long)y * P.nx;
        u = vpairs ? load_pair(ux + n + M.xa) : F2(ux[n + M.xa], ux[n + M.xb]);
        v = vpairs ? load_pair(uy + n + M.xa) : F2(uy[n + M.xa], uy[n + M.xb]);
    };
    // One turn of the pipeline: row r enters with its pulled populations in g, row r - L leaves. ALL:
    // every level has its rows (not so in the first turns, nor beyond the top wall).
    const auto turn = [&](auto all, int r, F2 g[NT], F2 u, F2 v) {
        constexpr bool ALL = decltype(all)::value;
        if (ALL || !WALLS || P.per_y || r < P.ny) {
            w.bottom = WALLS && !P.per_y && r == 0;
            w.top = WALLS && !P.per_y && r == P.ny - 1;
            vel(r, 0) = u;
            vel(r, 1) = v;
            thermal_row<HI1, WALLS>(P, g, w, u, v, row_base(P, wrap(r)));
        }
        bool left = true;  // level k - 1 has just left row q + 1 in g
#pragma unroll
        for (int k = 1; k < kSteps; ++k) {
            const int q = r - k;  // level k: step k + 1 of row q
            w.bottom = WALLS && !P.per_y && q == 0;
            w.top = WALLS && !P.per_y && q == P.ny - 1;
            const F2 above = as_stored(g[4], src);
            F2 h[NT];
            h[0] = S.c0[k - 1];
            h[1] = S.c1[k - 1];
            h[3] = S.c3[k - 1];
            h[2] = w.bottom ? S.dn[k - 1] : S.upp[k - 1];
            h[4] = w.top ? S.up[k - 1] : above;
            if (ALL || left) {
                S.upp[k - 1] = S.up[k - 1];
                S.up[k - 1] = as_stored(g[2], src);
                S.c0[k - 1] = as_stored(g[0], src);
                S.c1[k - 1] = as_stored(g[1], src);
                S.c3[k - 1] = as_stored(g[3], src);
                if (WALLS) S.dn[k - 1] = above;
            }
            left = left && q >= (WALLS && !P.per_y ? max(0, ya - L + k) : ya - L + k);
            if (ALL || (left && (!WALLS || P.per_y || q < P.ny)))
                thermal_row<HI1, WALLS>(P, h, w, vel(q, 0), vel(q, 1), row_base(P, wrap(q)));
#pragma unroll
            for (int i = 0; i < NT; ++i) g[i] = h[i];
        }
        if (ALL || left) {
            if (store) {
                E* dc = dst + (long long)(r - L) * P.pitch + x0;
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    if (store2) {
                        store_pair(dc + i * pl, g[i]);
                    } else {
                        float a, b;
                        g[i].split(a, b);
                        dc[i * pl] = from_a(a, (E*)nullptr);
                    }
                }
            }
        }
    };
    const int last = yb - 1 + L;
    int r = WALLS && !P.per_y ? max(0, ya - L) : ya - L;
    // the first turns fill the pipeline; with walls every turn is of this kind
    const int full = WALLS ? last + 1 : r + 2 * L;
    F2 g[NT], u, v;
    for (; r < full; ++r) {
        if (!WALLS || P.per_y || r < P.ny) load_row(r, g, u, v);
        turn(std::false_type(), r, g, u, v);
    }
    if constexpr (!WALLS) {
        for (; r <= last; ++r) {
            load_row(r, g, u, v);
            turn(std::true_type(), r, g, u, v);
        }
    }
}

// kSteps steps over a lattice: block (one warp) b takes strip b % strips of segment b / strips.
template <int ST, bool HI1>
__global__ void __launch_bounds__(32, kResidentT)
    k_thermal_steps(const typename Storage<ST>::T* __restrict__ src, typename Storage<ST>::T* __restrict__ dst,
                    const float* __restrict__ ux, const float* __restrict__ uy, const LatParams<float> P, const MarchGeom G)
{
    step_prologue();
    __shared__ F2 slots[2 * kSteps * 32];
    const int strip = blockIdx.x % G.strips, seg = blockIdx.x / G.strips;
    const int xo = strip * G.width, xe = min(P.nx, xo + G.width), ya = seg * G.rows, yb = min(P.ny, ya + G.rows);
    const MarchCols M = march_cols(P, xo - 2 * kLanesLost, threadIdx.x);
    if (M.pairs && !M.w.any_x && (P.per_y || (ya >= kSteps && yb <= P.ny - kSteps)))
        thermal_march<ST, HI1, false>(src, dst, ux, uy, P, M, xo, xe, ya, yb, threadIdx.x, slots + threadIdx.x);
    else
        thermal_march<ST, HI1, true>(src, dst, ux, uy, P, M, xo, xe, ya, yb, threadIdx.x, slots + threadIdx.x);
}

// g^eq(T, u) written to the slots the next pull reads (as k_init does for the coupled step), and
// the velocity stored in the handle's precision.
template <int ST>
__global__ void k_thermal_init(typename Storage<ST>::T* __restrict__ dst, VelT<ST>* __restrict__ uxs,
                               VelT<ST>* __restrict__ uys, const LatParams<typename Storage<ST>::A> P,
                               const double* __restrict__ T, const double* __restrict__ ux,
                               const double* __restrict__ uy)
{
    using A = typename Storage<ST>::A;
    using E = typename Storage<ST>::T;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long n = (long long)y * P.nx + x;
    const A u = ux ? A(ux[n]) : A(0), v = uy ? A(uy[n]) : A(0);
    const A t = T ? A(T[n]) : P.T0;
    uxs[n] = u;
    uys[n] = v;
    A g[NT];
    if constexpr (Storage<ST>::DEV) {
        eq_dev_d2q5(t, t - row_base(P, y), u, v, P.cs2T, g);
    } else {
        back_d2q5(t, A(0), A(0), t * P.cs2T, t * P.cs2T, u, v, g);
    }
    const int EX[NT] = {0, 1, 0, -1, 0};
    const int EY[NT] = {0, 0, 1, 0, -1};
    const int OPP[NT] = {0, 3, 4, 1, 2};
#pragma unroll
    for (int i = 0; i < NT; ++i) {
        int sx = x - EX[i], sy = y - EY[i];
        int side = -1;
        if (sx < 0) { if (P.per_x) sx += P.nx; else side = 0; }
        if (sx >= P.nx) { if (P.per_x) sx -= P.nx; else side = 1; }
        if (sy < 0) { if (P.per_y) sy += P.ny; else side = 2; }
        if (sy >= P.ny) { if (P.per_y) sy -= P.ny; else side = 3; }
        A val = g[i];
        long long slot;
        int plane;
        if (side < 0) {
            plane = i;
            slot = (long long)sy * P.pitch + sx;
        } else {
            plane = OPP[i];
            slot = (long long)y * P.pitch + x;
            if (P.kind[side] == WALL_DIRICHLET) val = P.Tw_c2[side] - val;
        }
        // a value the pull reads from the row below (above) is stored against that row's base
        if (side < 0 && EY[i] == 1) val = val + P.T_dyw;
        if (side < 0 && EY[i] == -1) val = val - P.T_dyw;
        dst[plane * P.plane + slot] = from_a(val, (E*)nullptr);
    }
}

template <int ST>
__global__ void k_thermal_out(const typename Storage<ST>::T* __restrict__ src,
                              const LatParams<typename Storage<ST>::A> P, const VelT<ST>* __restrict__ ux,
                              const VelT<ST>* __restrict__ uy, double* __restrict__ T, double* __restrict__ pops)
{
    using A = typename Storage<ST>::A;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    A g[NT];
    thermal_gather_node<Storage<ST>::DEV>(src, P, ux, uy, x, y, g);
    const long long n = (long long)y * P.nx + x, N = (long long)P.nx * P.ny;
    const double base = fma(double(y), double(P.T_dy), double(P.T_b));
    if (T) T[n] = base + double((g[0] + g[1]) + (g[2] + g[3]) + g[4]);
    if (pops)
#pragma unroll
        for (int i = 0; i < NT; ++i) pops[i * N + n] = double(g[i]) + double(w5<A>(i, P.cs2T)) * base;
}

constexpr int kChunkT = 32;

}  // namespace

struct clb_thermal {
    int nx = 0, ny = 0;
    clb_params p{};
    int device = 0;
    cudaStream_t stream = nullptr, cap = nullptr;
    char* mem = nullptr;
    void* buf[2] = {nullptr, nullptr};
    void* vel[2] = {nullptr, nullptr};
    double* stage = nullptr;
    int cur = 0;
    long steps = 0;
    int march = 0;  // > 0: kSteps steps per launch (k_thermal_steps), in segments of this many rows
    cudaGraphExec_t graph[2] = {nullptr, nullptr};
    LatParams<double> Pd{};
    LatParams<float> Pf{};
};

namespace {

size_t thermal_buffer_bytes(int nx, int ny, int storage)
{
    return align256((size_t)NT * (size_t)plane_elems(nx, ny, storage) * elem_size(storage));
}

size_t thermal_footprint(int nx, int ny, int storage)
{
    const size_t N = (size_t)nx * ny;
    const size_t vb = align256(N * (storage == CLB_F64 ? 8 : 4));
    return 2 * thermal_buffer_bytes(nx, ny, storage) + 2 * vb + align256(5 * N * sizeof(double));
}

clb_status thermal_launch(clb_thermal* h, int from, cudaStream_t s)
{
    const dim3 block(128, 1), grid((h->nx + 255) / 256, h->ny);  // two nodes per thread
    const void* a = h->buf[from];
    void* b = h->buf[from ^ 1];
    switch (h->p.storage) {
    case CLB_F64:
        CLB_CUDA(launch_chained(k_thermal_step<ST_F64>, grid, block, 0, s, (const double*)a, (double*)b, (const double*)h->vel[0], (const double*)h->vel[1], h->Pd));
        break;
    case CLB_F32:
        CLB_CUDA(launch_chained(k_thermal_step<ST_F32>, grid, block, 0, s, (const float*)a, (float*)b, (const float*)h->vel[0], (const float*)h->vel[1], h->Pf));
        break;
    default:
        CLB_CUDA(launch_chained(k_thermal_step<ST_F16DEV>, grid, block, 0, s, (const __half*)a, (__half*)b, (const float*)h->vel[0], (const float*)h->vel[1], h->Pf));
        break;
    }
    return CLB_OK;
}

MarchGeom thermal_geom(int nx, int ny, int rows)
{
    MarchGeom G;
    G.strips = (nx + kMarchOutT - 1) / kMarchOutT;
    G.width = ((nx + G.strips - 1) / G.strips + 1) & ~1;
    G.strips = (nx + G.width - 1) / G.width;
    G.rows = rows;
    G.segs = (ny + rows - 1) / rows;
    return G;
}

// Rows per segment of the kSteps-step kernel, 0 where one step per launch is the faster form (small
// lattices: 512 x 512 2.8 us against 2.9, 700 x 700 4.1 against 3.3; few rows; rows that fill their
// windows badly; wet walls, whose nodes pull through their neighbours; FP64, bound by its arithmetic).
// A segment of R rows takes R + 2 (kSteps - 1) turns; the R of the least turns over the rounds of
// resident warps is taken, counting two rounds at least: warps that all start together load and
// compute in step, and one round runs at half the rate (2048 x 2048: one of 22 rows 17.2 us per step,
// two of 12 to 14 rows 14.7 - 15.2; 4096 x 4096: two of 44 rows 45.9, three of 28 46.8).
// One step per launch is kept where the two estimates say so (both fitted to 330 shapes of 0.4 to 4 million
// nodes, to 5 and 10%, in us per step): one step takes 0.37 ns per warp of 64 nodes and 0.44 per block of
// 256, less the more nodes share the launch, and the FP32 bytes at the copy bandwidth where those leave L2; a
// turn of the pipeline takes a + b w at w warps per SM, more between x walls, whose windows take the wall rules
// every turn and end last, more on rows of three or four windows between them, more for lambda2 other than 1 and in the
// FP16 form, and 1.2 to 1.5 times as long on odd rows, whose velocities load one by one. One step per launch / four: FP32 cavities 640 x 640 3.6 / 4.1, 1024 x 1024 6.2 /
// 6.5, 802 x 829 5.5 / 4.9, 1500 x 1000 8.4 / 7.2; FP16 with lambda2 = 1.3 cavities 1800 x 1200 11.0 / 11.9,
// 162 x 5968 9.0 / 7.9, 2048 x 2048 24.6 / 18.6; layers 2971 x 220 4.6 / 5.4, 727 x 1495 6.8 / 7.5, 1024 x 1024
// 6.2 / 5.6. The choice costs 0.2% on average against the better one (four always: 2.5%).
constexpr long long kMarchNodesT = 400000;
struct TurnCost {
    double a, b;
};
// [FP32, FP16][no x walls, x walls][lambda2 = 1, other]
constexpr TurnCost kTurn[2][2][2] = {{{{0.55, 0.046}, {0.60, 0.053}}, {{0.75, 0.064}, {0.80, 0.072}}},
                                     {{{0.55, 0.053}, {0.55, 0.062}}, {{0.75, 0.065}, {0.80, 0.077}}}};
constexpr double kOddRowsOne = 1.03, kOddRowsTurn[2] = {1.4, 1.5}, kOddRowsTurnWalls = 1.2, kFewWindowsWalls = 1.2;
bool several_steps_pay(int nx, int ny, const clb_params& p, int rows, int sms)
{
    const double n = double(nx) * ny;
    double one = 1.96 + 0.367e-3 * ((nx + 63) / 64) * ny + 0.438e-3 * ((nx + 255) / 256) * ny - 3.38e-6 * std::min(n, 2.5e6);
    const bool odd = nx % 2 != 0;
    if (odd) one *= kOddRowsOne;
    if (p.storage == CLB_F32 && n >= 1.8e6) one = std::max(one, n * 48.0 / 7.0e6);
    const bool x_walls = p.wall[0] != CLB_PERIODIC;
    const TurnCost c = kTurn[p.storage == CLB_F16DEV][x_walls][p.lambda2 != 1.0];
    const double turns = double(rows + 2 * (kSteps - 1)) / kSteps;
    const MarchGeom G = thermal_geom(nx, ny, rows);
    double four = turns * (c.a + c.b * G.warps() / sms);
    if (odd) four *= x_walls ? kOddRowsTurnWalls : kOddRowsTurn[p.lambda2 != 1.0];
    if (x_walls && G.strips > 2 && G.strips <= 4) four *= kFewWindowsWalls;
    return four < one;
}
int thermal_rows_rule(int nx, int ny, const clb_params& p, int sms)
{
    const bool wet = p.wall[0] == CLB_WALL_WET || p.wall[2] == CLB_WALL_WET;
    if (p.storage == CLB_F64 || wet || (long long)nx * ny < kMarchNodesT || ny < 24) return 0;
    if ((double)nx < 0.7 * kMarchOutT * thermal_geom(nx, ny, 6).strips) return 0;
    int best = 6;
    long long least = 1LL << 60;
    for (int rows = 6; rows <= 64; ++rows) {
        const long long warps = thermal_geom(nx, ny, rows).warps(), round = (long long)sms * kResidentT;
        const long long turns = (rows + 2 * (kSteps - 1)) * std::max(2LL, (warps + round - 1) / round);
        if (turns < least) {
            least = turns;
            best = rows;
        }
    }
    return several_steps_pay(nx, ny, p, best, sms) ? best : 0;
}

// kSteps steps from buffer `from` into the other one.
clb_status thermal_launch_steps(clb_thermal* h, int from, cudaStream_t s)
{
    const MarchGeom G = thermal_geom(h->nx, h->ny, h->march);
    const void* a = h->buf[from];
    void* b = h->buf[from ^ 1];
    const float *u = (const float*)h->vel[0], *v = (const float*)h->vel[1];
    const bool hi1 = h->p.lambda2 == 1.0;
    if (h->p.storage == CLB_F32)
        CLB_CUDA(launch_chained(hi1 ? k_thermal_steps<ST_F32, true> : k_thermal_steps<ST_F32, false>, G.warps(), 32, 0, s,
                                (const float*)a, (float*)b, u, v, h->Pf, G));
    else
        CLB_CUDA(launch_chained(hi1 ? k_thermal_steps<ST_F16DEV, true> : k_thermal_steps<ST_F16DEV, false>, G.warps(), 32, 0,
                                s, (const __half*)a, (__half*)b, u, v, h->Pf, G));
    return CLB_OK;
}

clb_status thermal_out(clb_thermal* h, double* T, double* pops)
{
    const dim3 block(128, 1), grid((h->nx + 127) / 128, h->ny);  // one node per thread
    const void* a = h->buf[h->cur];
    switch (h->p.storage) {
    case CLB_F64:
        k_thermal_out<ST_F64><<<grid, block, 0, h->stream>>>((const double*)a, h->Pd, (const double*)h->vel[0],
                                                             (const double*)h->vel[1], T, pops);
        break;
    case CLB_F32:
        k_thermal_out<ST_F32><<<grid, block, 0, h->stream>>>((const float*)a, h->Pf, (const float*)h->vel[0],
                                                             (const float*)h->vel[1], T, pops);
        break;
    default:
        k_thermal_out<ST_F16DEV><<<grid, block, 0, h->stream>>>((const __half*)a, h->Pf, (const float*)h->vel[0],
                                                                (const float*)h->vel[1], T, pops);
        break;
    }
    CLB_CUDA(cudaGetLastError());
    return CLB_OK;
}

}  // namespace

extern "C" clb_status clb_thermal_create(int nx, int ny, const clb_params* p, void* stream, clb_thermal** out)
{
    if (!out) return set_error(CLB_EINVAL, "out is NULL");
    *out = nullptr;
    CLB_TRY(validate(nx, ny, p));
    auto* h = new (std::nothrow) clb_thermal;
    if (!h) return host_alloc_failed();
    h->nx = nx;
    h->ny = ny;
    h->p = *p;
    h->stream = (cudaStream_t)stream;
    cudaGetDevice(&h->device);
    const size_t bb = thermal_buffer_bytes(nx, ny, p->storage);
    const size_t N = (size_t)nx * ny;
    const size_t vb = align256(N * (p->storage == CLB_F64 ? 8 : 4));
    cudaError_t e = cudaStreamCreateWithFlags(&h->cap, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMalloc((void**)&h->mem, thermal_footprint(nx, ny, p->storage));
    if (e != cudaSuccess) {
        clb_thermal_destroy(h);
        return set_error(e == cudaErrorMemoryAllocation ? CLB_ENOMEM : CLB_ECUDA, "thermal create: %s", cudaGetErrorString(e));
    }
    h->buf[0] = h->mem;
    h->buf[1] = h->mem + bb;
    h->vel[0] = h->mem + 2 * bb;
    h->vel[1] = h->mem + 2 * bb + vb;
    h->stage = (double*)(h->mem + 2 * bb + 2 * vb);
    h->Pd = make_lat_params<double>(nx, ny, *p);
    h->Pf = make_lat_params<float>(nx, ny, *p);
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
    h->march = thermal_rows_rule(nx, ny, *p, std::max(1, sms));
    e = cudaMemsetAsync(h->mem, 0, 2 * bb, h->stream);
    if (e != cudaSuccess) {
        clb_thermal_destroy(h);
        return set_error(CLB_ECUDA, "thermal memset: %s", cudaGetErrorString(e));
    }
    clb_status st = clb_thermal_init(h, nullptr, nullptr, nullptr);
    if (st != CLB_OK) {
        clb_thermal_destroy(h);
        return st;
    }
    *out = h;
    return CLB_OK;
}

extern "C" void clb_thermal_destroy(clb_thermal* h)
{
    if (!h) return;
    if (h->mem) cudaStreamSynchronize(h->stream);
    for (auto& g : h->graph)
        if (g) cudaGraphExecDestroy(g);
    if (h->mem) cudaFree(h->mem);
    if (h->cap) cudaStreamDestroy(h->cap);
    delete h;
}

extern "C" clb_status clb_thermal_init(clb_thermal* h, const double* T, const double* ux, const double* uy)
{
    if (!h) return set_error(CLB_EINVAL, "handle is NULL");
    const size_t N = (size_t)h->nx * h->ny;
    const double* src[3] = {T, ux, uy};
    const double* dev[3] = {nullptr, nullptr, nullptr};
    for (int k = 0; k < 3; ++k)
        if (src[k]) {
            CLB_CUDA(cudaMemcpyAsync(h->stage + k * N, src[k], N * sizeof(double), cudaMemcpyHostToDevice, h->stream));
            dev[k] = h->stage + k * N;
        }
    const dim3 block(128, 1), grid((h->nx + 127) / 128, h->ny);  // one node per thread
    void* d = h->buf[h->cur];
    switch (h->p.storage) {
    case CLB_F64: k_thermal_init<ST_F64><<<grid, block, 0, h->stream>>>((double*)d, (double*)h->vel[0], (double*)h->vel[1], h->Pd, dev[0], dev[1], dev[2]); break;
    case CLB_F32: k_thermal_init<ST_F32><<<grid, block, 0, h->stream>>>((float*)d, (float*)h->vel[0], (float*)h->vel[1], h->Pf, dev[0], dev[1], dev[2]); break;
    default: k_thermal_init<ST_F16DEV><<<grid, block, 0, h->stream>>>((__half*)d, (float*)h->vel[0], (float*)h->vel[1], h->Pf, dev[0], dev[1], dev[2]); break;
    }
    CLB_CUDA(cudaGetLastError());
    CLB_CUDA(cudaStreamSynchronize(h->stream));
    h->steps = 0;
    return CLB_OK;
}

extern "C" clb_status clb_thermal_set_steps_per_launch(clb_thermal* h, int steps)
{
    if (!h) return set_error(CLB_EINVAL, "handle is NULL");
    if (steps != 0 && steps != 1) return set_error(CLB_EINVAL, "steps per launch %d: 1, or 0 for the library's choice", steps);
    int march = 0;
    if (steps == 0) {
        int sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device);
        march = thermal_rows_rule(h->nx, h->ny, h->p, std::max(1, sms));
    }
    if (march == h->march) return CLB_OK;
    CLB_CUDA(cudaStreamSynchronize(h->stream));
    for (auto& g : h->graph)
        if (g) {
            cudaGraphExecDestroy(g);
            g = nullptr;
        }
    h->march = march;
    return CLB_OK;
}

extern "C" clb_status clb_thermal_get_steps_per_launch(clb_thermal* h, int* steps)
{
    if (!h) return set_error(CLB_EINVAL, "handle is NULL");
    if (!steps) return set_error(CLB_EINVAL, "steps is NULL");
    *steps = h->march > 0 ? kSteps : 1;
    return CLB_OK;
}

extern "C" clb_status clb_thermal_step(clb_thermal* h, long n)
{
    if (!h) return set_error(CLB_EINVAL, "handle is NULL");
    if (n < 0) return set_error(CLB_EINVAL, "n < 0");
    // both parities are captured on the first chunk (no capture later, mid-stepping)
    for (int par = 0; n >= kChunkT && par < 2; ++par) {
        if (h->graph[par]) continue;
        CLB_CUDA(cudaStreamBeginCapture(h->cap, cudaStreamCaptureModeThreadLocal));
        clb_status st = CLB_OK;
        const int per = h->march > 0 ? kSteps : 1;  // steps per launch; kChunkT / per launches are an even number
        for (int k = 0; k < kChunkT / per && st == CLB_OK; ++k)
            st = per > 1 ? thermal_launch_steps(h, par ^ (k & 1), h->cap) : thermal_launch(h, par ^ (k & 1), h->cap);
        cudaGraph_t g = nullptr;
        cudaError_t e = cudaStreamEndCapture(h->cap, &g);
        if (st != CLB_OK) {
            if (g) cudaGraphDestroy(g);
            return st;
        }
        if (e != cudaSuccess) return set_error(CLB_ECUDA, "capture: %s", cudaGetErrorString(e));
        e = cudaGraphInstantiate(&h->graph[par], g, 0);
        cudaGraphDestroy(g);
        if (e != cudaSuccess) return set_error(CLB_ECUDA, "instantiate: %s", cudaGetErrorString(e));
    }
    while (n >= kChunkT) {
        CLB_CUDA(cudaGraphLaunch(h->graph[h->cur], h->stream));
        n -= kChunkT;
        h->steps += kChunkT;
    }
    for (; h->march > 0 && n >= kSteps; n -= kSteps) {
        CLB_TRY(thermal_launch_steps(h, h->cur, h->stream));
        h->cur ^= 1;
        h->steps += kSteps;
    }
    for (; n > 0; --n) {
        CLB_TRY(thermal_launch(h, h->cur, h->stream));
        h->cur ^= 1;
        h->steps++;
    }
    return CLB_OK;
}

extern "C" clb_status clb_thermal_fields(clb_thermal* h, double* T)
{
    if (!h || !T) return set_error(CLB_EINVAL, "handle and T must not be NULL");
    const size_t N = (size_t)h->nx * h->ny;
    CLB_TRY(thermal_out(h, h->stage, nullptr));
    CLB_CUDA(cudaMemcpyAsync(T, h->stage, N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CLB_CUDA(cudaStreamSynchronize(h->stream));
    return CLB_OK;
}

extern "C" clb_status clb_thermal_populations(clb_thermal* h, double* g)
{
    if (!h || !g) return set_error(CLB_EINVAL, "handle and g must not be NULL");
    const size_t N = (size_t)h->nx * h->ny;
    CLB_TRY(thermal_out(h, nullptr, h->stage));
    CLB_CUDA(cudaMemcpyAsync(g, h->stage, 5 * N * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
    CLB_CUDA(cudaStreamSynchronize(h->stream));
    return CLB_OK;
}

extern "C" clb_status clb_thermal_sync(clb_thermal* h)
{
    if (!h) return set_error(CLB_EINVAL, "handle is NULL");
    CLB_CUDA(cudaStreamSynchronize(h->stream));
    return CLB_OK;
}
