// Exact signed distance to a height field (Sec. 3.1 of Liu & Stevens,
// arXiv:2006.03343: phi = +d in the fluid, -d in the solid, d the minimum
// distance to the immersed boundary), for terrain given as heights h[j][i] at
// the column nodes.  The boundary is the piecewise-linear surface through the
// samples, each cell split along its (i, j)-(i+1, j+1) diagonal into two flat
// triangles, periodic in x and y.
//
// A block takes a row segment of 32 columns.  Only levels within `reach` of the
// heights around a column can be nearer than `reach` to the surface; every other
// level keeps z - h[j][i], which has the right sign and a magnitude above the
// reach.  The nodes that can be nearer go into a list in shared memory and the
// block's threads search them, one node per thread, whatever columns and levels
// they come from.  A search starts at |z - h[j][i]| (the vertex straight below or
// above is on the surface) and visits the window of cells within `reach`
// horizontally in ascending horizontal distance (a list built on the host and
// passed in the kernel's parameters), stopping once that distance alone exceeds
// the best so far; a cell is skipped when the horizontal gap and the vertical gap
// to its height range together exceed it.  The distances of that pass are FP32;
// only the triangles that can hold the nearest point are evaluated in FP64, and
// of them only the features that can: the result feeds the FP64 classification
// of wmibm_init.
#include "internal.cuh"

#include <algorithm>
#include <vector>

using namespace wmibm;

namespace {

constexpr int kSdfCols = 32;     // columns per block: one row segment
constexpr int kSdfWarps = 8;     // warps per block, each taking every 8th level
constexpr int kSdfBlocks = 3;    // resident blocks per SM (80 registers)
constexpr int kSdfRound = 16;    // levels listed between two searches (both grids)
constexpr int kSdfList = 2 * kSdfCols * kSdfRound;
constexpr int kSdfTasks = 2 * kSdfList;  // FP64 evaluations queued in a round (more are done on the spot)
constexpr int kSdfMaxCells = 1024;
constexpr int kSdfMaxSpan = 160;         // window cell columns and rows: at most 2 (64 + 4)
constexpr int kSdfSmemCap = 20 * 1024;           // bytes for each of the z table and the height tiles

struct SdfParams {
    const double *h;
    double *phi_uv, *phi_w;
    int32_t nx, ny, nz, ncells;
    int32_t wx, wy, segs, tw;    // window half-widths in cells, row segments per row, tile width
    double dx, dy, dz, rdx, rdy, rdz, reach;
    float reachf, rdzf;
    float dxf, dyf, rdxf, rdyf, spanf;   // spanf: horizontal extent of the window, (wx + wy + 2) cells
    int8_t ca[kSdfMaxCells], cb[kSdfMaxCells];   // window cells (i + ca, j + cb), nearest first
};

__device__ __forceinline__ int wrap_index(int q, int n)
{
    if (q >= 0 && q < n) return q;
    q %= n;
    return q < 0 ? q + n : q;
}

__device__ __forceinline__ float quotient(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double quotient(double a, double b) { return a / b; }

// squared distance from the origin to the segment P -> Q (nearest point
// P + t (Q - P), t the projection parameter clamped to [0, 1])
template <typename T>
__device__ __forceinline__ T seg2(T px, T py, T pz, T qx, T qy, T qz)
{
    const T wx = -px, wy = -py, wz = -pz;
    const T ex = qx - px, ey = qy - py, ez = qz - pz;
    const T we = wx * ex + wy * ey + wz * ez;
    T t = T(0);
    if (we > T(0)) {
        const T ee = ex * ex + ey * ey + ez * ez;
        t = we >= ee ? T(1) : quotient(we, ee);
    }
    const T rx = wx - t * ex, ry = wy - t * ey, rz = wz - t * ez;
    return rx * rx + ry * ry + rz * rz;
}

// A cell's corners relative to the node: A = (x0, y0), B = (x1, y0), C = (x1, y1),
// D = (x0, y1), heights e00, e10, e11, e01.  Lower triangle A B C, upper A C D.
template <typename T>
struct CellAt {
    T x0, y0, x1, y1, dx, dy, rdx, rdy, e00, e10, e01, e11;
};

// Squared distance from the node, at the origin, to the plane of the lower
// (U = false) or upper triangle; inside: whether the projection falls in it.
template <typename T, bool U>
__device__ __forceinline__ T face2(const CellAt<T> &q, bool &inside)
{
    // plane e00 + sx (x - x0) + sy (y - y0); c = the node's height above it
    const T sx = U ? (q.e11 - q.e01) * q.rdx : (q.e10 - q.e00) * q.rdx;
    const T sy = U ? (q.e01 - q.e00) * q.rdy : (q.e11 - q.e10) * q.rdy;
    const T c = sx * q.x0 + sy * q.y0 - q.e00;
    const T t = quotient(c, T(1) + sx * sx + sy * sy);
    const T u = t * sx - q.x0, v = t * sy - q.y0;           // the projection, relative to A
    inside = U ? (u >= T(0) && v <= q.dy && v * q.dx >= u * q.dy) : (u <= q.dx && v >= T(0) && v * q.dx <= u * q.dy);
    return c * t;
}

// Squared distance to edge n of a triangle: 0 the diagonal A C (both triangles),
// 1 A B or A D, 2 B C or D C.
template <typename T>
__device__ __forceinline__ T edge2(const CellAt<T> &q, bool upper, int n)
{
    const T mx = upper ? q.x0 : q.x1, my = upper ? q.y1 : q.y0, mz = upper ? q.e01 : q.e10;   // D or B
    const bool from_m = n == 2, to_m = n == 1;
    return seg2<T>(from_m ? mx : q.x0, from_m ? my : q.y0, from_m ? mz : q.e00, to_m ? mx : q.x1, to_m ? my : q.y1,
                   to_m ? mz : q.e11);
}

// FP32 squared distances of a cell's two triangles.
__device__ __forceinline__ void cell2(const CellAt<float> &q, float &lower, float &upper)
{
    bool in1, in2;
    lower = face2<float, false>(q, in1);
    upper = face2<float, true>(q, in2);
    if (!in1 || !in2) {
        const float diag = edge2(q, false, 0);
        if (!in1) lower = fminf(diag, fminf(edge2(q, false, 1), edge2(q, false, 2)));
        if (!in2) upper = fminf(diag, fminf(edge2(q, true, 1), edge2(q, true, 2)));
    }
}

// Heights around one column: from the block's shared tiles (TILE) or from
// global memory.  Offsets (a, b) are relative to the column, |a| <= wx, |b| <= wy.
// The FP32 heights are relative to a height of the block (href; 0 without tiles),
// so that they keep the differences that the distances are made of.
template <bool TILE>
struct Heights {
    const SdfParams &p;
    const double *dt;
    const float *ft;
    int c, i, j;
    __device__ double d(int a, int b) const
    {
        if (TILE) return dt[(b + p.wy) * p.tw + c + a + p.wx];
        return __ldg(p.h + (int64_t)wrap_index(j + b, p.ny) * p.nx + wrap_index(i + a, p.nx));
    }
    __device__ float f(int a, int b) const
    {
        if (TILE) return ft[(b + p.wy) * p.tw + c + a + p.wx];
        return (float)d(a, b);
    }
};

__device__ __forceinline__ float horizontal2(const SdfParams &p, int a, int b)
{
    const float rx = a > 0 ? a * p.dxf : (a < -1 ? -(a + 1) * p.dxf : 0.0f);
    const float ry = b > 0 ? b * p.dyf : (b < -1 ? -(b + 1) * p.dyf : 0.0f);
    return rx * rx + ry * ry;
}

// Corners of window cell (a, b) relative to the node.
template <bool TILE>
__device__ __forceinline__ CellAt<float> corners_f(const SdfParams &p, const Heights<TILE> &H, int a, int b, float zf)
{
    const float x0 = a * p.dxf, y0 = b * p.dyf;
    return CellAt<float>{x0, y0, x0 + p.dxf, y0 + p.dyf, p.dxf, p.dyf, p.rdxf, p.rdyf, H.f(a, b) - zf, H.f(a + 1, b) - zf,
                         H.f(a, b + 1) - zf, H.f(a + 1, b + 1) - zf};
}

// Whether cell q, at horizontal distance sqrt(rh2), can be nearer than lim.
__device__ __forceinline__ bool reachable(const CellAt<float> &q, float rh2, float lim)
{
    const float gap = fmaxf(fmaxf(-fmaxf(fmaxf(q.e00, q.e10), fmaxf(q.e01, q.e11)),
                                  fminf(fminf(q.e00, q.e10), fminf(q.e01, q.e11))), 0.0f);
    return rh2 + gap * gap <= lim * lim;
}

// What an FP64 evaluation is of: a triangle's face whose projection certainly falls
// inside, one whose FP32 projection is too near a side to tell, or one edge.
enum SdfTask { kFace = 0, kFaceOrEdges = 1, kEdge = 2 };     // kEdge + n: edge n

// Corners of window cell (a, b) relative to the node in FP64; xy: the cells'
// (x0, x1), then (y0, y1).  mid: the corner that only this triangle has (both the
// B and the D slot take it; the other is not read).
template <bool TILE>
__device__ __forceinline__ CellAt<double> corners_d(const SdfParams &p, const Heights<TILE> &H, const double2 *xy,
                                                    int a, int b, bool upper, double z)
{
    CellAt<double> q;
    const double2 x = xy[a + p.wx], y = xy[2 * p.wx + b + p.wy];
    q.x0 = x.x;
    q.x1 = x.y;
    q.y0 = y.x;
    q.y1 = y.y;
    q.e00 = __dsub_rn(H.d(a, b), z);
    q.e11 = __dsub_rn(H.d(a + 1, b + 1), z);
    q.e01 = q.e10 = __dsub_rn(upper ? H.d(a, b + 1) : H.d(a + 1, b), z);
    return q;
}

// FP64 squared distance to a triangle's face (kind kFace), or to its face or
// edges (kFaceOrEdges).
__device__ __forceinline__ double face_d(const SdfParams &p, const CellAt<double> &q, bool upper, int kind)
{
    // both triangles' planes by one sequence: sx, sy from the corners each has
    const double mid = q.e01;
    const double sx = (upper ? q.e11 - mid : mid - q.e00) * p.rdx;
    const double sy = (upper ? mid - q.e00 : q.e11 - mid) * p.rdy;
    const double c = sx * q.x0 + sy * q.y0 - q.e00;
    const double t = c / (1.0 + sx * sx + sy * sy);
    if (kind == kFaceOrEdges) {
        const double u = t * sx - q.x0, v = t * sy - q.y0;  // the projection, relative to A
        const double vx = v * p.dx, uy = u * p.dy;
        if (!(upper ? (u >= 0.0 && v <= p.dy && vx >= uy) : (u <= p.dx && v >= 0.0 && vx <= uy)))
            return fmin(edge2(q, upper, 0), fmin(edge2(q, upper, 1), edge2(q, upper, 2)));
    }
    return c * t;
}

template <bool TILE>
__device__ __noinline__ double evaluate(const SdfParams &p, const Heights<TILE> &H, const double2 *xy, int n, int kind,
                                        double z)
{
    const bool upper = n & 1;
    const CellAt<double> q = corners_d<TILE>(p, H, xy, p.ca[n >> 1], p.cb[n >> 1], upper, z);
    return kind >= kEdge ? edge2(q, upper, kind - kEdge) : face_d(p, q, upper, kind);
}

// The FP64 evaluations that triangle n needs (a bit per SdfTask), given that it is
// within lim in FP32: its face where the projection falls inside, else those of
// its edges that are within lim (the nearest point is on one of them).  Inside or
// not is decided in FP32 where that is clear of its rounding: u and v carry the
// error of the slopes (a fifth of tol over a cell, at most) times t and times the
// window's cells, tol bounding the errors of lengths.
template <bool TILE>
__device__ __forceinline__ unsigned tasks_of(const SdfParams &p, const Heights<TILE> &H, int n, float zf, float lim,
                                             float tol)
{
    const bool upper = n & 1;
    const CellAt<float> f = corners_f<TILE>(p, H, p.ca[n >> 1], p.cb[n >> 1], zf);
    const float fx = upper ? (f.e11 - f.e01) * p.rdxf : (f.e10 - f.e00) * p.rdxf;
    const float fy = upper ? (f.e01 - f.e00) * p.rdyf : (f.e11 - f.e10) * p.rdyf;
    const float ft = quotient(fx * f.x0 + fy * f.y0 - f.e00, 1.0f + fx * fx + fy * fy);
    const float fu = ft * fx - f.x0, fv = ft * fy - f.y0;
    // distance of the projection to the triangle's sides, positive inside
    const float diag = quotient(fv * p.dxf - fu * p.dyf, fmaxf(p.dxf, p.dyf));
    const float side = upper ? fminf(fminf(fu, p.dyf - fv), diag) : fminf(fminf(p.dxf - fu, fv), -diag);
    const float eps = tol * ((float)(2 + p.wx + p.wy) + fabsf(ft) * fmaxf(p.rdxf, p.rdyf));
    if (side > eps) return 1u << kFace;
    if (!(side < -eps)) return 1u << kFaceOrEdges;
    const float lim2 = lim * lim;
    unsigned m = 0;
    for (int e = 0; e < 3; ++e)
        if (edge2(f, upper, e) <= lim2) m |= 1u << (kEdge + e);
    return m;
}

// The search of one node in FP32.  On this part FP64 runs at a small fraction of
// the FP32 rate, so this pass finds the smallest distance m over the window's
// triangles (and the vertex straight below or above, |vertf|), and the two nearest
// triangles; those within m + tol are handed on for FP64 evaluation, tol a bound
// on twice the FP32 error.  Where even
// the third is within m + tol, a second pass hands on every triangle that is,
// except around the column's own vertex, where it can tell more.
// The triangle holding the nearest point is always among them, so the least of
// the FP64 values and of the vertex's is the FP64 distance.  Returns the bound that
// the vertex's distance has to be within (by tol) to count, or infinity when m
// exceeds the reach by more than tol: such a node needs no FP64.  herr bounds the
// error of an FP32 height difference.
template <bool TILE, typename Hand>
__device__ __forceinline__ float search(const SdfParams &p, const Heights<TILE> &H, float zf, float vertf, float tol,
                                        float herr, Hand hand)
{
    float m = fabsf(vertf);
    float d1 = INFINITY, d2 = INFINITY, d3 = INFINITY;      // the three least distances, ascending
    int n1 = 0, n2 = 0;                                     // the first two's triangles: 2 * cell + (1: upper)
    auto insert = [&](float d, int n) {
        if (d < d3) {
            d3 = fmaxf(d, d2);
            if (d < d2) {
                d2 = d;
                n2 = n;
                if (d2 < d1) {
                    d2 = d1;
                    d1 = d;
                    n2 = n1;
                    n1 = n;
                }
            }
        }
    };
    for (int e = 0; e < p.ncells; ++e) {
        const int a = p.ca[e], b = p.cb[e];
        const float rh2 = horizontal2(p, a, b);
        const float lim = m + tol;
        if (rh2 > lim * lim) break;
        const CellAt<float> q = corners_f<TILE>(p, H, a, b, zf);
        if (!reachable(q, rh2, lim)) continue;
        float lower, upper;
        cell2(q, lower, upper);
        lower = sqrtf(lower);
        upper = sqrtf(upper);
        m = fminf(m, fminf(lower, upper));
        insert(lower, 2 * e);
        insert(upper, 2 * e + 1);
    }
    if (m - tol > p.reachf) return INFINITY;
    const float lim = m + tol;
    float slope2;
    if (!(d3 <= lim)) {
        if (d1 <= lim) hand(n1, tasks_of<TILE>(p, H, n1, zf, lim, tol));
        if (d2 <= lim) hand(n2, tasks_of<TILE>(p, H, n2, zf, lim, tol));
        return m;
    }
    // The triangles around the column's own vertex.  A point of one of their faces or
    // of an edge through the vertex is nearer than the vertex by vert^2 g^2 (in
    // squares), g the sine of the slope in that direction: where the ground is so
    // nearly level that all of them are within tol, g still tells them apart, as the
    // slopes are as exact as the height differences are (herr).  A face holds its
    // projection when its gradient, taken uphill for a node above the ground, points
    // into its sector.  rise: a lower bound of the largest g whose point certainly exists.
    const float sign = vertf < 0.0f ? -1.0f : 1.0f, h = H.f(0, 0), away = fabsf(vertf);
    const float gerr = 2.0f * herr * fmaxf(p.rdxf, p.rdyf), cerr = 2.0f * gerr * fmaxf(p.dxf, p.dyf);
    // height differences along the edges to (1, 0), (1, 1), (0, 1), (-1, 0), (-1, -1), (0, -1)
    const float zE = sign * (H.f(1, 0) - h), zC = sign * (H.f(1, 1) - h), zN = sign * (H.f(0, 1) - h);
    const float zW = sign * (H.f(-1, 0) - h), zD = sign * (H.f(-1, -1) - h), zS = sign * (H.f(0, -1) - h);
    // the triangles between consecutive edges: 2 * cell + (1: upper), the edge opposite the vertex, the gradient and
    // the two sides of its sector
    constexpr int kTriangle[6] = {6, 7, 4, 1, 0, 3}, kOpposite[6] = {2, 2, 0, 1, 1, 0};
    const float gx[6] = {zE, zC - zN, -zW, -zW, zS - zD, zE}, gy[6] = {zC - zE, zN, zN, zW - zD, -zS, -zS};
    const float edge_z[6] = {zE, zC, zN, zW, zD, zS};
    constexpr int kEdgeOf[6] = {6, 6, 7, 4, 0, 3}, kEdgeNo[6] = {1, 0, 1, 1, 0, 1};
    float rise = 0.0f, g_face[6], g_edge[6];
    int in[6];                                              // 1: the face holds its projection, 0: it may, -1: it does not
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const float sx = gx[i] * p.rdxf, sy = gy[i] * p.rdyf, slope2 = sx * sx + sy * sy;
        const float t = quotient(away, 1.0f + slope2);
        const float right = p.dyf * sx, up = p.dxf * sy, turn = right - up;
        // sides of the sector: E .. C, C .. N, N .. W, W .. (-1, -1), .. S, S .. E
        const float side1 = i == 0 ? up : i == 1 ? -turn : i == 2 ? -right : i == 3 ? -up : i == 4 ? turn : right;
        const float side2 = i == 0 ? turn : i == 1 ? right : i == 2 ? up : i == 3 ? -turn : i == 4 ? -right : -up;
        const float side = fminf(side1, side2);
        const bool near = t * (fabsf(sx) * p.rdxf + fabsf(sy) * p.rdyf) < 0.9f;
        in[i] = side < -cerr ? -1 : (side > cerr && near ? 1 : 0);
        g_face[i] = sqrtf(quotient(slope2, 1.0f + slope2));
        if (in[i] == 1) rise = fmaxf(rise, g_face[i]);
        const bool dx1 = i != 2 && i != 5, dy1 = i != 0 && i != 3;
        const float e2 = (dx1 ? p.dxf * p.dxf : 0.0f) + (dy1 ? p.dyf * p.dyf : 0.0f) + edge_z[i] * edge_z[i];
        g_edge[i] = edge_z[i] > 0.0f ? edge_z[i] * rsqrtf(e2) : -1.0f;
        if (away * edge_z[i] < 0.9f * e2) rise = fmaxf(rise, g_edge[i]);
    }
    rise -= 3.0f * gerr + 1e-5f * rise;                     // either g is off by sqrt 2 gerr and some ulps at most
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const int n = kTriangle[i];
        unsigned k = 0;
        if (in[i] == 0) {
            k = 1u << kFaceOrEdges;
        } else {
            if (in[i] == 1 && g_face[i] >= rise) k = 1u << kFace;
            const CellAt<float> f = corners_f<TILE>(p, H, p.ca[n >> 1], p.cb[n >> 1], zf);
            if (edge2(f, n & 1, kOpposite[i]) <= lim * lim) k |= 1u << (kEdge + kOpposite[i]);
        }
        hand(n, k);
        if (g_edge[i] >= fmaxf(rise, 0.0f)) hand(kEdgeOf[i], 1u << (kEdge + kEdgeNo[i]));
    }
    for (int e = 0; e < p.ncells; ++e) {
        const int a = p.ca[e], b = p.cb[e];
        const float rh2 = horizontal2(p, a, b);
        if (rh2 > lim * lim) break;
        const CellAt<float> q = corners_f<TILE>(p, H, a, b, zf);
        if (!reachable(q, rh2, lim)) continue;
        float lower, upper;
        cell2(q, lower, upper);
        for (int u = 0; u < 2; ++u) {
            const int n = 2 * e + u;
            if (n < 8 && (0xdbu >> n & 1u)) continue;       // around the vertex
            if (sqrtf(u ? upper : lower) <= lim) hand(n, tasks_of<TILE>(p, H, n, zf, lim, tol));
        }
    }
    return rise > 0.0f ? m - 2.0f * tol : m;                // the vertex itself is then not the nearest point
}

// Order of finite doubles as integers and back (the FP64 unit takes 16 cycles a
// warp for a comparison too).
__device__ __forceinline__ int64_t key_of(double v)
{
    const int64_t b = __double_as_longlong(v);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double of_key(int64_t k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}

// z of level k on the uv-grid (g = 0) or the w-grid (g = 1), rounded once, as written
__device__ __forceinline__ double level_z(const SdfParams &p, int g, int k)
{
    return __dmul_rn(k + (g ? 0.0 : 0.5), p.dz);
}

// On rolling terrain bound by the FP64 unit (58 % of its cycles; the subtractions z - h
// alone take 110 us of it at 512 x 256 x 256) and by the FP32 search beside it.  A single
// hill is bound by the spread of the work: the ground around it is flat (one table for
// all columns of a segment, and stores), and the some 290 of 4096 segments whose window
// meets the hill do all the searching, round after round in one block each.
// The first form gave every thread its column's near levels and evaluated whole
// cells in FP64, so a warp paid for the union of what its lanes needed, and setting
// up the ranges cost every thread some 60 FP64 operations.  Now the searches are
// dense over a block, hand on single faces and edges, and those are evaluated dense
// as well.  512 x 256 x 256, reach 4 dz: hill 855 -> 192 us, Gaussian hills 2774 ->
// 567 us; 256 x 128 x 64 ridge, reach 2 dz: 499 -> 70 us (one GB300).
//
// A block owns one row segment of 32 columns; its 8 warps share them, warp q
// taking levels q, q + 8, ... of each, so that every warp's store covers 32
// consecutive nodes.  ZTAB: the levels' z sit in a shared table (2 nz doubles), so
// that a level outside the reach costs one subtraction and a store, or the store
// alone where the segment is flat.  TILE: the heights the segment's windows touch sit in shared tiles, in
// FP64 and in FP32.
template <bool ZTAB, bool TILE>
__global__ void __launch_bounds__(kSdfCols * kSdfWarps, kSdfBlocks) k_heightfield_sdf(const __grid_constant__ SdfParams p)
{
    extern __shared__ double smem[];
    // the warps' height ranges (as keys), then the round's queue of FP64 evaluations: faces from the front, edges from
    // the back (node | triangle << 10 | SdfTask << 21)
    __shared__ union {
        struct {
            int64_t min[kSdfWarps][kSdfCols], max[kSdfWarps][kSdfCols];
        } part;
        uint32_t task[kSdfTasks];
    } sh;
    // the round's nodes: column | grid << 5 | level in the round << 6; their least squared distances (as bits: positive
    // doubles are ordered alike)
    __shared__ uint16_t list[kSdfList];
    __shared__ unsigned long long best[kSdfList];
    __shared__ float scales[kSdfCols];                      // per column: the size of its FP32 heights
    __shared__ int listed, faces, edges;
    // (x0, x1) of the window's cell columns, then (y0, y1) of its cell rows, relative to the node
    __shared__ double2 cell_xy[kSdfMaxSpan];
    double *const ztab = smem;
    double *const dtile = smem + (ZTAB ? 2 * p.nz : 0);
    const int th = 2 * p.wy + 1;
    float *const ftile = reinterpret_cast<float *>(dtile + (TILE ? th * p.tw : 0));
    const int seg = blockIdx.x % p.segs, j = blockIdx.x / p.segs;
    const int i_first = seg * kSdfCols;
    const double href = TILE ? __ldg(p.h + (int64_t)j * p.nx + i_first) : 0.0;
    if (ZTAB) {
        for (int q = threadIdx.x; q < 2 * p.nz; q += kSdfCols * kSdfWarps) ztab[q] = level_z(p, q >= p.nz, q % p.nz);
    }
    if (TILE) {
        for (int q = threadIdx.x; q < th * p.tw; q += kSdfCols * kSdfWarps) {
            const int r = q / p.tw, cc = q % p.tw;
            const double v = __ldg(p.h + (int64_t)wrap_index(j - p.wy + r, p.ny) * p.nx +
                                   wrap_index(i_first - p.wx + cc, p.nx));
            dtile[q] = v;
            ftile[q] = (float)__dsub_rn(v, href);
        }
    }
    for (int q = threadIdx.x; q < 2 * (p.wx + p.wy); q += kSdfCols * kSdfWarps) {
        const bool x = q < 2 * p.wx;
        const double step = x ? p.dx : p.dy, at = (x ? q - p.wx : q - 2 * p.wx - p.wy) * step;
        cell_xy[q] = make_double2(at, at + step);
    }
    if (threadIdx.x == 0) listed = faces = edges = 0;
    __syncthreads();
    const int c = threadIdx.x % kSdfCols, warp = threadIdx.x / kSdfCols;
    const int i = i_first + c;
    const bool live = i < p.nx;
    const Heights<TILE> H{p, dtile, ftile, c, live ? i : 0, j};
    // height range of every vertex a window cell touches, the window's rows
    // shared out over the warps
    int64_t lo = INT64_MAX, hi = INT64_MIN;
    if (live) {
        for (int b = -p.wy + warp; b <= p.wy; b += kSdfWarps)
            for (int a = -p.wx; a <= p.wx; ++a) {
                const int64_t q = key_of(H.d(a, b));
                lo = min(lo, q);
                hi = max(hi, q);
            }
    }
    sh.part.min[warp][c] = lo;
    sh.part.max[warp][c] = hi;
    __syncthreads();
    const int64_t plane = (int64_t)p.nx * p.ny;
    const int64_t col = (int64_t)j * p.nx + i;
    const double hv = live ? H.d(0, 0) : 0.0;
    const int64_t hkey = key_of(hv);
    lo = hi = hkey;
    if (live)
        for (int q = 0; q < kSdfWarps; ++q) {
            lo = min(lo, sh.part.min[q][c]);
            hi = max(hi, sh.part.max[q][c]);
        }
    const bool top = hkey >= hi, bottom = hkey <= lo;
    const float hminf = (float)of_key(lo), hmaxf = (float)of_key(hi);
    const float hsize = fmaxf(fabsf(hminf), fabsf(hmaxf));
    // largest of the column's FP32 heights
    if (warp == 0)
        scales[c] = fmaxf(fabsf((float)(of_key(lo) - href)), fabsf((float)(of_key(hi) - href)));
    // levels with hmin - reach <= z <= hmax + reach, widened on each side by a level
    // and by the rounding of these FP32 operations: only these can lie within the
    // reach (a level taken in needlessly still gets z - h, as its distance exceeds the
    // reach).  A window whose slopes are below 1e-8 has none: over ground of slope s
    // the distance is between |z - h| and |z - h| (1 - s^2 / 2), half an ulp lower.
    const bool level = (float)(of_key(hi) - of_key(lo)) * (p.rdxf + p.rdyf) <= 1e-8f;
    int klo[2], khi[2];
    for (int g = 0; g < 2; ++g) {
        const float off = g ? 0.0f : 0.5f, size = 1e-6f * (hsize + p.reachf) * p.rdzf;
        const float vlo = (hminf - p.reachf) * p.rdzf - off, vhi = (hmaxf + p.reachf) * p.rdzf - off;
        const float flo = fminf(fmaxf(floorf(vlo - size) - 1.0f, 0.0f), 2147483520.0f);
        const float fhi = fminf(fmaxf(ceilf(vhi + size) + 1.0f, -1.0f), 2147483520.0f);
        klo[g] = min((int)flo, p.nz);
        khi[g] = min((int)fhi, p.nz - 1);
        if (!live || level || khi[g] < klo[g]) {
            klo[g] = p.nz;
            khi[g] = -1;
        }
    }
    // a flat segment (all its columns of one height): the table takes z - h, once for all columns
    const int64_t h0 = __shfl_sync(0xffffffffu, hkey, 0);
    const bool flat = ZTAB && __all_sync(0xffffffffu, !live || hkey == h0);
    if (ZTAB && flat) {
        const double h = of_key(h0);
        for (int q = threadIdx.x; q < 2 * p.nz; q += kSdfCols * kSdfWarps) ztab[q] = __dsub_rn(ztab[q], h);
        __syncthreads();
    }
    // the segment's levels that may hold a listed node: [blo, bhi], the same in every warp
    const int blo = __reduce_min_sync(0xffffffffu, min(klo[0], klo[1]));
    const int bhi = __reduce_max_sync(0xffffffffu, max(khi[0], khi[1]));
    // z - h of level k of grid g: one FP64 subtraction (FP64 is the scarce unit here), or none in a flat segment
    auto vertical = [&](int g, int k) -> double {
        const double z = ZTAB ? ztab[g * p.nz + k] : level_z(p, g, k);
        return flat ? z : __dsub_rn(z, hv);
    };
    // levels outside
    if (live)
        for (int g = 0; g < 2; ++g) {
            double *const out = (g ? p.phi_w : p.phi_uv) + col;
            for (int part = 0; part < 2; ++part) {
                if (bhi < 0 && part) break;                 // no near level: the first part was all of them
                const int first = part ? bhi + 1 : 0, end = part ? p.nz : blo;
                int k = first + ((warp - first) & (kSdfWarps - 1));
                double *o = out + k * plane;
                if (flat) {
#pragma unroll 4
                    for (; k < end; k += kSdfWarps, o += kSdfWarps * plane) *o = ztab[g * p.nz + k];
                } else {
#pragma unroll 4
                    for (; k < end; k += kSdfWarps, o += kSdfWarps * plane) *o = vertical(g, k);
                }
            }
        }
    if (bhi >= blo) __syncthreads();                        // the queue takes the ranges' place
    for (int base = blo; base <= bhi; base += kSdfRound) {
        const int end = min(base + kSdfRound, bhi + 1);
        for (int g = 0; g < 2; ++g) {
            double *const out = (g ? p.phi_w : p.phi_uv) + col;
            for (int k = base + warp; k < end; k += kSdfWarps) {
                const double vert = vertical(g, k);
                // the column's own vertex is the nearest surface point when it is the
                // highest of the window and the node lies above it (every other surface
                // point is lower, so farther), or the lowest with the node below it
                const bool above = __double_as_longlong(vert) >= 0;
                const bool wanted = live && k >= klo[g] && k <= khi[g] && !(above ? top : bottom);
                const unsigned mask = __ballot_sync(0xffffffffu, wanted);
                if (mask) {
                    int at = 0;
                    if (c == 0) at = atomicAdd(&listed, __popc(mask));
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if (wanted)
                        list[at + __popc(mask & ((1u << c) - 1u))] = (uint16_t)(c | g << 5 | (k - base) << 6);
                }
                if (live && !wanted) out[(int64_t)k * plane] = vert;
            }
        }
        __syncthreads();
        const int count = listed;
        auto node = [&](int q, int &cc, int &g, int &k) {
            const int e = list[q];
            cc = e & 31;
            g = (e >> 5) & 1;
            k = base + (e >> 6);
        };
        auto z_of = [&](int g, int k) -> double { return ZTAB && !flat ? ztab[g * p.nz + k] : level_z(p, g, k); };
        // FP32 searches: what they hand on goes into the queue
        for (int q = threadIdx.x; q < count; q += kSdfCols * kSdfWarps) {
            int cc, g, k;
            node(q, cc, g, k);
            const Heights<TILE> N{p, dtile, ftile, cc, i_first + cc, j};
            const double z = z_of(g, k);
            const float zf = (float)(TILE ? __dsub_rn(z, href) : z), vertf = zf - N.f(0, 0);
            // twice the FP32 error of a distance: the heights and coordinates are off by 3 ulps (of 2^-24) of their size,
            // which moves a distance by no more, and the arithmetic adds 6 of the lengths in it and 8 of the distance:
            // less than 1.3e-6 of the sizes together
            const float tol = 2e-6f * (2.0f * scales[cc] + p.spanf + 2.0f * fabsf(zf));
            unsigned long long mine = (unsigned long long)__double_as_longlong(INFINITY);
            const float m = search<TILE>(p, N, zf, vertf, tol, 2.5e-7f * scales[cc], [&](int n, unsigned kinds) {
                for (; kinds; kinds &= kinds - 1u) {
                    const int kind = __ffs((int)kinds) - 1;
                    const bool face = kind < kEdge;
                    const int at = atomicAdd(face ? &faces : &edges, 1);
                    if (at < kSdfTasks / 2)
                        sh.task[face ? at : kSdfTasks - 1 - at] = (uint32_t)(q | n << 10 | kind << 21);
                    else
                        mine = min(mine, (unsigned long long)__double_as_longlong(
                                             evaluate<TILE>(p, N, cell_xy, n, kind, z)));
                }
            });
            // the vertex straight below or above counts where it is within the same bound
            if (m < INFINITY && fabsf(vertf) <= m + tol) {
                const double vert = __dsub_rn(z, N.d(0, 0));
                mine = min(mine, (unsigned long long)__double_as_longlong(vert * vert));
            }
            best[q] = mine;
        }
        __syncthreads();
        const int nf = min(faces, kSdfTasks / 2), ne = min(edges, kSdfTasks / 2);
        for (int half = 0; half < 2; ++half)
            for (int t = threadIdx.x; t < (half ? ne : nf); t += kSdfCols * kSdfWarps) {
                const uint32_t task = sh.task[half ? kSdfTasks - 1 - t : t];
                const int q = task & 1023, n = (task >> 10) & 2047, kind = task >> 21;
                int cc, g, k;
                node(q, cc, g, k);
                const Heights<TILE> N{p, dtile, ftile, cc, i_first + cc, j};
                const bool upper = n & 1;
                const CellAt<double> at = corners_d<TILE>(p, N, cell_xy, p.ca[n >> 1], p.cb[n >> 1], upper, z_of(g, k));
                const double d2 = half ? edge2(at, upper, kind - kEdge) : face_d(p, at, upper, kind);
                atomicMin(&best[q], (unsigned long long)__double_as_longlong(d2));
            }
        __syncthreads();
        for (int q = threadIdx.x; q < count; q += kSdfCols * kSdfWarps) {
            int cc, g, k;
            node(q, cc, g, k);
            const Heights<TILE> N{p, dtile, ftile, cc, i_first + cc, j};
            const double vert = __dsub_rn(z_of(g, k), N.d(0, 0)), b2 = __longlong_as_double((long long)best[q]);
            double phi = vert;
            if (b2 < INFINITY) {
                const double d = sqrt(b2);
                if (d <= p.reach) phi = copysign(d, vert);
            }
            (g ? p.phi_w : p.phi_uv)[k * plane + (int64_t)j * p.nx + i_first + cc] = phi;
        }
        if (threadIdx.x == 0) listed = faces = edges = 0;
        __syncthreads();
    }
}

}  // namespace

extern "C" int wmibm_heightfield_sdf(const wmibm_grid *g, const double *height, double reach, double *phi_uv,
                                     double *phi_w, void *stream)
{
    ApiRange nvtx_range("wmibm_heightfield_sdf");
    if (!g || !height || !phi_uv || !phi_w) return set_error(nullptr, WMIBM_EINVAL, "NULL grid or field pointer");
    if (g->nx < 1 || g->ny < 1 || g->nz < 3) return set_error(nullptr, WMIBM_EINVAL, "bad grid sizes");
    const int64_t n = (int64_t)g->nx * g->ny * g->nz;
    if (n >= ((int64_t)1 << 31)) return set_error(nullptr, WMIBM_EINVAL, "nx*ny*nz must be < 2^31");
    if (!(g->lx > 0.0) || !(g->ly > 0.0) || !(g->lz > 0.0) || !std::isfinite(g->lx) || !std::isfinite(g->ly) ||
        !std::isfinite(g->lz))
        return set_error(nullptr, WMIBM_EINVAL, "domain lengths must be finite and > 0");
    if (!(reach > 0.0) || !std::isfinite(reach)) return set_error(nullptr, WMIBM_EINVAL, "reach must be finite and > 0");
    if (phi_uv == phi_w) return set_error(nullptr, WMIBM_EINVAL, "phi_uv and phi_w must be distinct");
    SdfParams p = {};
    p.h = height;
    p.phi_uv = phi_uv;
    p.phi_w = phi_w;
    p.nx = g->nx;
    p.ny = g->ny;
    p.nz = g->nz;
    p.dx = g->lx / g->nx;
    p.dy = g->ly / g->ny;
    p.dz = g->lz / (g->nz - 1);
    p.rdx = 1.0 / p.dx;
    p.rdy = 1.0 / p.dy;
    p.rdz = 1.0 / p.dz;
    p.reach = reach;
    const double wxd = std::ceil(reach / p.dx), wyd = std::ceil(reach / p.dy);
    if (wxd * wyd * 4.0 > kSdfMaxCells || wxd > 64 || wyd > 64)
        return set_error(nullptr, WMIBM_EINVAL,
                         "reach spans %.0f x %.0f cells; at most %d window cells and 128 in each direction", 2 * wxd,
                         2 * wyd, kSdfMaxCells);
    p.wx = (int32_t)wxd;
    p.wy = (int32_t)wyd;
    // window cells a in [-wx, wx - 1], b in [-wy, wy - 1]: every cell that meets
    // the disc of radius reach around the column; nearest (horizontally) first
    struct Cell {
        double r2;
        int a, b;
    };
    std::vector<Cell> cells;
    for (int b = -p.wy; b < p.wy; ++b)
        for (int a = -p.wx; a < p.wx; ++a) {
            const double rx = a > 0 ? a * p.dx : (a < -1 ? -(a + 1) * p.dx : 0.0);
            const double ry = b > 0 ? b * p.dy : (b < -1 ? -(b + 1) * p.dy : 0.0);
            const double r2 = rx * rx + ry * ry;
            if (r2 <= reach * reach * (1.0 + 1e-12)) cells.push_back({r2, a, b});
        }
    std::stable_sort(cells.begin(), cells.end(), [](const Cell &l, const Cell &r) { return l.r2 < r.r2; });
    p.ncells = (int32_t)cells.size();
    for (size_t e = 0; e < cells.size(); ++e) {
        p.ca[e] = (int8_t)cells[e].a;
        p.cb[e] = (int8_t)cells[e].b;
    }
    p.segs = (g->nx + kSdfCols - 1) / kSdfCols;
    p.tw = kSdfCols + 2 * p.wx;
    p.dxf = (float)p.dx;
    p.dyf = (float)p.dy;
    p.reachf = (float)reach;
    p.rdzf = (float)p.rdz;
    p.rdxf = (float)(1.0 / p.dx);
    p.rdyf = (float)(1.0 / p.dy);
    p.spanf = (float)((p.wx + 1) * p.dx + (p.wy + 1) * p.dy);
    const int64_t blocks = (int64_t)p.segs * g->ny;
    if (blocks >= ((int64_t)1 << 31)) return set_error(nullptr, WMIBM_EINVAL, "too many row segments");
    const size_t zbytes = (size_t)2 * g->nz * sizeof(double);
    const size_t tbytes = (size_t)(2 * p.wy + 1) * p.tw * (sizeof(double) + sizeof(float));
    const bool ztab = zbytes <= (size_t)kSdfSmemCap, tile = tbytes <= (size_t)kSdfSmemCap;
    const size_t smem = (ztab ? zbytes : 0) + (tile ? tbytes : 0);
    const dim3 grid((unsigned)blocks), block(kSdfCols * kSdfWarps);
    cudaStream_t st = (cudaStream_t)stream;
    auto *const kernel = ztab ? (tile ? k_heightfield_sdf<true, true> : k_heightfield_sdf<true, false>)
                              : (tile ? k_heightfield_sdf<false, true> : k_heightfield_sdf<false, false>);
    // with the static arrays more than the 48 KB that need no asking
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * kSdfSmemCap);
    if (e != cudaSuccess) return cuda_status(nullptr, e, "k_heightfield_sdf shared memory");
    kernel<<<grid, block, smem, st>>>(p);
    return cuda_status(nullptr, cudaGetLastError(), "k_heightfield_sdf launch");
}
