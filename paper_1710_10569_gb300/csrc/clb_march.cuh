// clb_march.cuh -- two time steps of a coupled FP32 lattice per launch.
//
// What bounds it. One step reads and writes every population once, and the one-step kernel runs at
// the copy bandwidth doing so (2048 x 1024: 34.8 us, 0.997 of it) with the issue slots half idle:
// the only way past it is to move fewer bytes per step. A warp here takes a window of 64 columns (two
// nodes per lane) and marches along y. At row r it pulls row r from the source buffer and collides
// it (the first step), then pulls row r - 1 of that intermediate state and collides it (the second
// step), so a population crosses HBM once for two steps. Every node's arithmetic is that of the
// one-step kernels (collide_dev on packed pairs, the same pull and wall rules), so the results are
// bitwise the same. It is then bound by the FP32 pipe (73% busy; HBM 62% at 4096 x 2048), and on
// lattices that fill one round of resident warps by the wait for a row's loads (FP32 pipe 53%, HBM 61% at
// 2048 x 1024).
//
// Where the intermediate state lives. The second step at row q needs, of the intermediate state, the
// populations with e_y = 0 of row q, those with e_y = +1 of row q - 1 and those with e_y = -1 of row
// q + 1 (just computed). A lane only ever needs its own two columns and, through a warp shuffle, its
// neighbour lanes': so the rows are kept in shared memory in slots private to the thread, and no
// barrier is needed. One warp per block, so that a block's place is free as soon as its warp ends.
//
// The price. The outermost column of a window is lost at each step (its neighbour lies outside the
// window), so of 64 columns a warp stores the inner 60 at most (lanes 1 to 30); and a segment of R
// rows takes R + 2 rows of the first step. Windows and segments overlap by that much and repeat the
// work (6.7% and 1/R); no two warps exchange anything.
//
// Measured (us per step, one step per launch -> two): 2048 x 1024 34.8 -> 23.9 (87.8 GLUPS), 4096 x
// 2048 131.8 -> 86.5 (97 GLUPS). The FP16 form moves half the bytes and is at the FP32 pipe's limit
// with one step per launch (72.9 us at 4096 x 2048, 80.5 with two): it keeps that. Tried: the next
// row staged by cp.async (2048 x 1024: 35.8; two more shared-memory passes per population) and by
// L2 prefetches one or two rows ahead (24.4 - 24.6); four warps per block (26.6); 24 warps per SM
// instead of 20 (24.8).
#pragma once

#include "clb_kernels.cuh"

namespace clb {

constexpr int kMarchOut = 60;        // columns a window stores at most
constexpr int kMarchSlots = 18;      // pairs of values per thread: rows of the intermediate state
constexpr int kMarchResident = 20;   // warps per SM that the register bound of k_step_two leaves

// The strips (windows along x, `width` stored columns each, even) and segments (along y, `rows`
// rows each) that cover a lattice.
struct MarchGeom {
    int width, strips, rows, segs;
    __host__ __device__ int warps() const { return strips * segs; }
};

// Strips and segments of the two-step kernel with segments of `rows` rows.
inline MarchGeom march_geom(int nx, int ny, int rows)
{
    MarchGeom G;
    G.strips = (nx + kMarchOut - 1) / kMarchOut;
    G.width = ((nx + G.strips - 1) / G.strips + 1) & ~1;
    G.strips = (nx + G.width - 1) / G.width;
    G.rows = rows;
    G.segs = (ny + rows - 1) / rows;
    return G;
}

// The rows per segment for which the warps (a function of it) take the least time, in us per step: a
// round of w warps per SM takes 0.5 + 0.068 w us per row and step (fitted to 1 to 20 warps per SM), a
// segment of R rows is R + 1 of these. 0 if none takes less than `one_step`, the time of one step per
// launch.
constexpr int kMarchRowsMin = 4, kMarchRowsMax = 64;
template <typename Warps>
inline int march_rows_for(const Warps& warps_of, int sms, double one_step)
{
    int best = 0;
    double least = one_step;
    for (int rows = kMarchRowsMin; rows <= kMarchRowsMax; ++rows) {
        const long long warps = warps_of(rows), resident = (long long)sms * kMarchResident, rest = warps % resident;
        const double t = (rows + 1) * ((warps / resident) * (0.5 + 0.068 * kMarchResident) +
                                       (rest ? 0.5 + 0.068 * rest / sms : 0.0));
        if (t < least) {
            least = t;
            best = rows;
        }
    }
    return best;
}

// The pair of values pulled from x - 1 (shr) or x + 1 (shl): one from the neighbour lane.
__device__ __forceinline__ F2 pull_shr(F2 v)
{
    float a, b;
    v.split(a, b);
    return F2(lane_up(b), a);
}
__device__ __forceinline__ F2 pull_shl(F2 v)
{
    float a, b;
    v.split(a, b);
    return F2(b, lane_down(a));
}
__device__ __forceinline__ F2 as_pair(unsigned long long u)
{
    F2 r;
    r.u = u;
    return r;
}

// Wall state of one row of a warp's window.
struct MarchWalls {
    bool bottom, top;  // the row lies next to the bottom (top) wall: warp-uniform
    bool any_x;        // some lane's node lies next to an x wall: warp-uniform
    int m0, m1;        // bits 1 (left wall), 2 (right wall) of this lane's two nodes
};

// The columns a lane loads, and which of its nodes lie next to an x wall.
struct MarchCols {
    int xa, xb;
    bool pairs;  // every lane's two columns load as one aligned pair: warp-uniform
    MarchWalls w;
};
// Columns start + 2 lane and the next (start even).
__device__ __forceinline__ MarchCols march_cols(const LatParams<float>& P, int start, int lane)
{
    MarchCols M;
    const int x0 = start + 2 * lane;
    // its own two where they exist (a periodic row wraps); lanes beyond an x wall, whose values reach
    // no stored node, load columns 0 and 1
    int xa = x0, xb = x0 + 1;
    if (P.per_x) {
        xa = (xa % P.nx + P.nx) % P.nx;
        xb = (xb % P.nx + P.nx) % P.nx;
    } else if (xa < 0 || xa >= P.nx) {
        xa = 0;
        xb = 1;
    } else if (xb >= P.nx) {
        xb = xa;
    }
    M.xa = xa;
    M.xb = xb;
    // not where an odd row wraps or ends (and in the lanes after a wrap of it)
    M.pairs = __all_sync(0xffffffffu, xb == xa + 1 && (xa & 1) == 0);
    M.w.bottom = M.w.top = false;
    M.w.m0 = P.per_x ? 0 : (x0 == 0 ? 1 : 0) | (x0 == P.nx - 1 ? 2 : 0);
    M.w.m1 = P.per_x ? 0 : (x0 + 1 == P.nx - 1 ? 2 : 0);
    M.w.any_x = __any_sync(0xffffffffu, (M.w.m0 | M.w.m1) != 0);
    return M;
}

// Pull and collide one row. Before the shift along x, v[i] holds population i of this lane's two
// nodes on the row it is pulled from (for a pull across a y wall the opposite plane of the node's
// own row); d5..d8 hold the diagonals of the node's own row (read only next to an x wall). v receives
// the post-collision populations.
template <bool HI1, bool WALLS>
__device__ __forceinline__ void march_row(const LatParams<float>& P, F2 v[NPOP], const MarchWalls& w, F2 d5, F2 d6,
                                          F2 d7, F2 d8, float Tb)
{
    // shifts along x; next to an x wall the node's own opposite value comes in instead
    const bool left = WALLS && (w.m0 & 1), right0 = WALLS && (w.m0 & 2), right1 = WALLS && (w.m1 & 2);
    const auto from_left = [&](F2 x, F2 own) {
        float a, b, o0, o1;
        x.split(a, b);
        own.split(o0, o1);
        const float up = lane_up(b);
        return F2(left ? o0 : up, a);
    };
    const auto from_right = [&](F2 x, F2 own) {
        float a, b, o0, o1;
        x.split(a, b);
        own.split(o0, o1);
        const float down = lane_down(a);
        return F2(right0 ? o0 : b, right1 ? o1 : down);
    };
    F2 f[9], g[5];
    f[0] = v[0];
    f[2] = v[2];
    f[4] = v[4];
    f[1] = from_left(v[1], v[3]);
    f[3] = from_right(v[3], v[1]);
    f[5] = from_left(v[5], d7);
    f[6] = from_right(v[6], d8);
    f[7] = from_right(v[7], d5);
    f[8] = from_left(v[8], d6);
    g[0] = v[9];
    g[1] = from_left(v[10], WALLS && P.kind[0] == WALL_DIRICHLET ? F2(P.Tw_c2[0]) - v[12] : v[12]);
    g[2] = v[11];
    g[3] = from_right(v[12], WALLS && P.kind[1] == WALL_DIRICHLET ? F2(P.Tw_c2[1]) - v[10] : v[10]);
    g[4] = v[13];
    // next to a y wall (whole rows): bounced values, not shifted; elsewhere g2 and g4 are re-based to
    // this row (see finish_pull)
    if (WALLS && w.bottom) {
        f[5] = v[5];
        f[6] = v[6];
        if (P.kind[2] == WALL_DIRICHLET) g[2] = F2(P.Tw_c2[2]) - g[2];
    } else {
        g[2] = g[2] - F2(P.T_dyw);
    }
    if (WALLS && w.top) {
        f[7] = v[7];
        f[8] = v[8];
        if (P.kind[3] == WALL_DIRICHLET) g[4] = F2(P.Tw_c2[3]) - g[4];
    } else {
        g[4] = g[4] + F2(P.T_dyw);
    }
    if (WALLS && P.moving) {
        // momentum of a moving wall; a diagonal that crosses two takes the y wall's
        const auto add = [&](int i, bool x0, bool x1, int x_side, bool y, int y_side) {
            const float c = y ? P.fbb[y_side][i] : P.fbb[x_side][i];
            f[i] = f[i] + F2(x0 || y ? c : 0.0f, x1 || y ? c : 0.0f);
        };
        add(1, left, false, 0, false, 0);
        add(3, right0, right1, 1, false, 0);
        add(2, false, false, 0, w.bottom, 2);
        add(4, false, false, 0, w.top, 3);
        add(5, left, false, 0, w.bottom, 2);
        add(6, right0, right1, 1, w.bottom, 2);
        add(7, right0, right1, 1, w.top, 3);
        add(8, left, false, 0, w.top, 3);
    }
    collide_dev<HI1>(P, f, g, F2(Tb));
#pragma unroll
    for (int i = 0; i < NPOP; ++i) v[i] = i < 9 ? f[i] : g[i - 9];
}

// Two time steps of rows [ya, yb), columns [xo, xe) (xo even, xe - xo <= kMarchOut, xe even or nx)
// from src into dst, by one warp; slots: this thread's shared-memory slots, `stride` apart. WALLS =
// false is for windows and segments none of whose rows (ya - 1 to yb) or columns lies next to a wall
// and whose columns all load as aligned pairs: compiled together with the wall rules, the moves
// between the two paths cost the interior 90 of 450 instructions per pair of nodes.
template <bool HI1, bool WALLS>
__device__ __forceinline__ void march_rows(const float* __restrict__ src, float* __restrict__ dst,
                                           const LatParams<float>& P, const MarchCols& M, int xo, int xe, int ya,
                                           int yb, int lane, unsigned long long* __restrict__ slots, int stride)
{
    using Two = unsigned long long;
    const int x0 = xo - 2 + 2 * lane;
    const int oa = (int)chunk_off(M.xa), ob = (int)chunk_off(M.xb);
    const bool pairs = !WALLS || M.pairs;
    MarchWalls w = M.w;
    const bool store = lane >= 1 && lane <= 30 && x0 < xe;
    const bool store2 = x0 + 1 < P.nx;
    const int os = (int)chunk_off(max(x0, 0));
    // populations by the row they are pulled from: the node's own (C), the one below (U), above (D)
    const int C[6] = {0, 1, 3, 9, 10, 12}, U[4] = {2, 5, 6, 11}, D[4] = {4, 7, 8, 13};
    const int ROWSEL[NPOP] = {0, 0, 1, 0, 2, 1, 1, 2, 2, 0, 0, 1, 0, 2};
    // slots, of the intermediate state: C of row q, U of rows q and q - 1, and D of row q
    const auto keepC = [&](int k) -> Two& { return slots[k * stride]; };
    const auto keepU = [&](int row, int k) -> Two& { return slots[(6 + (row & 1) * 4 + k) * stride]; };
    const auto keepD = [&](int k) -> Two& { return slots[(14 + k) * stride]; };

    for (int r = (!WALLS || P.per_y || ya > 0) ? ya - 1 : 0; r <= yb; ++r) {
        F2 v[NPOP];
        if (!WALLS || P.per_y || r < P.ny) {
            // first step, row r (wrapped)
            const int y = r < 0 ? r + P.ny : r >= P.ny ? r - P.ny : r;
            w.bottom = WALLS && !P.per_y && y == 0;
            w.top = WALLS && !P.per_y && y == P.ny - 1;
            const float* sc = src + (long long)y * P.crow;
            // a pull across a y wall reads the node's own opposite plane: two planes further (2, 5, 6,
            // 11 -> 4, 7, 8, 13) at the bottom, two back at the top
            const float* su = w.bottom ? sc + 2 * kRowChunk : src + (long long)(y > 0 ? y - 1 : P.ny - 1) * P.crow;
            const float* sd = w.top ? sc - 2 * kRowChunk : src + (long long)(y < P.ny - 1 ? y + 1 : 0) * P.crow;
            if (pairs) {
                const float *lc = sc + oa, *lu = su + oa, *ld = sd + oa;
#pragma unroll
                for (int i = 0; i < NPOP; ++i)
                    v[i] = as_pair(*reinterpret_cast<const Two*>((ROWSEL[i] == 0 ? lc : ROWSEL[i] == 1 ? lu : ld) + i * kRowChunk));
            } else {
#pragma unroll
                for (int i = 0; i < NPOP; ++i) {
                    const float* p = (ROWSEL[i] == 0 ? sc : ROWSEL[i] == 1 ? su : sd) + i * kRowChunk;
                    v[i] = F2(p[oa], p[ob]);
                }
            }
            F2 d5 = v[0], d6 = v[0], d7 = v[0], d8 = v[0];
            if (WALLS && (w.m0 | w.m1)) {
                const auto own = [&](int i) { return F2(sc[i * kRowChunk + oa], sc[i * kRowChunk + ob]); };
                d5 = own(5);
                d6 = own(6);
                d7 = own(7);
                d8 = own(8);
            }
            march_row<HI1, WALLS>(P, v, w, d5, d6, d7, d8, row_base(P, y));
        }
        // what row q pulls of the intermediate state: U from row q - 1 (bounced at the bottom: its own
        // D), D from row r just computed (bounced at the top: its own U); row r takes the slots
        const int q = r - 1;
        w.bottom = WALLS && !P.per_y && q == 0;
        w.top = WALLS && !P.per_y && q == P.ny - 1;
        F2 d5 = v[0], d6 = v[0], d7 = v[0], d8 = v[0];
        if (WALLS && (w.m0 | w.m1)) {
            d5 = as_pair(keepU(q, 1));
            d6 = as_pair(keepU(q, 2));
            d7 = as_pair(keepD(1));
            d8 = as_pair(keepD(2));
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const Two old = keepC(k);
            keepC(k) = v[C[k]].u;
            v[C[k]] = as_pair(old);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const Two old = w.bottom ? keepD(k) : keepU(r, k);
            keepU(r, k) = v[U[k]].u;
            v[U[k]] = as_pair(old);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const Two now = v[D[k]].u;
            if (WALLS && w.top) v[D[k]] = as_pair(keepU(q, k));
            if (WALLS && (w.any_x || (!P.per_y && r == 0))) keepD(k) = now;
        }
        if (q < ya) continue;
        // second step, row q
        march_row<HI1, WALLS>(P, v, w, d5, d6, d7, d8, row_base(P, q));
        if (store) {
            float* dc = dst + (long long)q * P.crow + os;
            if (store2) {
#pragma unroll
                for (int i = 0; i < NPOP; ++i) *reinterpret_cast<Two*>(dc + i * kRowChunk) = v[i].u;
            } else {
#pragma unroll
                for (int i = 0; i < NPOP; ++i) {
                    float a, b;
                    v[i].split(a, b);
                    dc[i * kRowChunk] = a;
                }
            }
        }
    }
}

// Two time steps of one strip and segment, by one warp.
template <bool HI1>
__device__ __forceinline__ void march_two(const float* __restrict__ src, float* __restrict__ dst,
                                          const LatParams<float>& P, int xo, int xe, int ya, int yb, int lane,
                                          unsigned long long* __restrict__ slots, int stride)
{
    const MarchCols M = march_cols(P, xo - 2, lane);
    if (M.pairs && !M.w.any_x && (P.per_y || (ya >= 2 && yb <= P.ny - 2)))
        march_rows<HI1, false>(src, dst, P, M, xo, xe, ya, yb, lane, slots, stride);
    else
        march_rows<HI1, true>(src, dst, P, M, xo, xe, ya, yb, lane, slots, stride);
}

// Two time steps over a lattice: block (one warp) g takes strip g % strips of segment g / strips.
template <bool HI1>
__global__ void __launch_bounds__(32, kMarchResident)
    k_step_two(const float* __restrict__ src, float* __restrict__ dst, const LatParams<float> P, const MarchGeom G)
{
    step_prologue();
    __shared__ unsigned long long slots[kMarchSlots * 32];
    const int strip = blockIdx.x % G.strips, seg = blockIdx.x / G.strips;
    const int xo = strip * G.width, ya = seg * G.rows;
    march_two<HI1>(src, dst, P, xo, min(P.nx, xo + G.width), ya, min(P.ny, ya + G.rows), threadIdx.x,
                   slots + threadIdx.x, 32);
}

}  // namespace clb
