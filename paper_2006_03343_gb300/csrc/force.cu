// The forcing f = -div(tau) on the vertically staggered grid (Eq. 2 and Eq. 18
// of Liu & Stevens, arXiv:2006.03343; vertical differences of Eqs. 15-16,
// horizontal derivatives by periodic second-order central differences):
//   f_x(uv k) = -[(txx[i+1]-txx[i-1])/2dx + (txy[j+1]-txy[j-1])/2dy + (txz[k+1]-txz[k])/dz]
//   f_y(uv k) = -[(txy[i+1]-txy[i-1])/2dx + (tyy[j+1]-tyy[j-1])/2dy + (tyz[k+1]-tyz[k])/dz]
//   f_z(w k)  = -[(txz[i+1]-txz[i-1])/2dx + (tyz[j+1]-tyz[j-1])/2dy + (tzz[k]-tzz[k-1])/dz]
// with f_x = f_y = 0 on the ghost uv level and f_z = 0 on the floor and lid.
//
// The direct-load form, for rows that the bulk-copy pipeline (stencil.cu) does not
// take: each thread owns V consecutive x-points of one (j) row and marches up a
// chunk of z levels, carrying txz, tyz (level k+1 -> k) and tzz (k -> k-1) in
// registers.  Centre values come in as vector loads of the widest type that the
// rows' alignment allows; the x-neighbours at the vector edges and the j +- 1 rows
// are re-read through L1 (they are the neighbouring threads' lines), so DRAM sees
// each array once.  Bound by the loads' latency: all of a level's loads are issued
// before the first is used, with 32-bit offsets from the array bases.  The whole
// step (one GB300, FP32; before: 64-bit addresses, one value a thread, 32 x 8
// threads): 150 x 90 x 75 35.4 -> 20.7 us, 151 x 90 x 75 35.4 -> 22.8, 490 x 130 x
// 101 128 -> 54.  Loading a level ahead took registers worth more as resident
// blocks (22.7, 24.8 and 68 us).
#include "internal.cuh"

using namespace wmibm;

namespace {

template <typename T, int V>
struct Pack {
    T v[V];
};

template <typename T, int V>
__device__ __forceinline__ Pack<T, V> ldp(const T *p);

template <>
__device__ __forceinline__ Pack<float, 4> ldp<float, 4>(const float *p)
{
    float4 a = __ldg(reinterpret_cast<const float4 *>(p));
    return Pack<float, 4>{{a.x, a.y, a.z, a.w}};
}
template <>
__device__ __forceinline__ Pack<float, 2> ldp<float, 2>(const float *p)
{
    float2 a = __ldg(reinterpret_cast<const float2 *>(p));
    return Pack<float, 2>{{a.x, a.y}};
}
template <>
__device__ __forceinline__ Pack<float, 1> ldp<float, 1>(const float *p)
{
    return Pack<float, 1>{{__ldg(p)}};
}
template <>
__device__ __forceinline__ Pack<double, 2> ldp<double, 2>(const double *p)
{
    double2 a = __ldg(reinterpret_cast<const double2 *>(p));
    return Pack<double, 2>{{a.x, a.y}};
}
template <>
__device__ __forceinline__ Pack<double, 1> ldp<double, 1>(const double *p)
{
    return Pack<double, 1>{{__ldg(p)}};
}

template <typename T, int V>
__device__ __forceinline__ void stp(T *p, const Pack<T, V> &x);
template <>
__device__ __forceinline__ void stp<float, 4>(float *p, const Pack<float, 4> &x)
{
    *reinterpret_cast<float4 *>(p) = make_float4(x.v[0], x.v[1], x.v[2], x.v[3]);
}
template <>
__device__ __forceinline__ void stp<float, 2>(float *p, const Pack<float, 2> &x)
{
    *reinterpret_cast<float2 *>(p) = make_float2(x.v[0], x.v[1]);
}
template <>
__device__ __forceinline__ void stp<float, 1>(float *p, const Pack<float, 1> &x) { *p = x.v[0]; }
template <>
__device__ __forceinline__ void stp<double, 2>(double *p, const Pack<double, 2> &x)
{
    *reinterpret_cast<double2 *>(p) = make_double2(x.v[0], x.v[1]);
}
template <>
__device__ __forceinline__ void stp<double, 1>(double *p, const Pack<double, 1> &x) { *p = x.v[0]; }

template <typename T>
struct ForceParams {
    const T *txx, *txy, *tyy, *tzz, *txz, *tyz;
    T *fx, *fy, *fz;
    int32_t nx, ny, nz, kc;
    T cx, cy, cz;       // 1/(2 dx), 1/(2 dy), 1/dz
};

// What a thread loads for level k: the vectors of its row and of the rows beside it,
// the values beyond the vector's ends, txz and tyz of the level above.
template <typename T, int V>
struct Level {
    Pack<T, V> xx, xy, xyjm, xyjp, yyjm, yyjp, yzjm, yzjp, zz, xz_kp, yz_kp;
    T xxl, xxr, xyl, xyr, xzl, xzr;
};

// Resident blocks per SM that the registers are held to: latency-bound, so as many
// as need no spills.
template <typename T, int V>
constexpr int kForceBlocks = sizeof(T) == 4 && V <= 2 ? 4 : 3;

template <typename T, int V>
__global__ void __launch_bounds__(256, (kForceBlocks<T, V>)) k_force(ForceParams<T> p)
{
    const int32_t nq = p.nx / V;
    const int32_t q = blockIdx.x * blockDim.x + threadIdx.x;
    const int32_t j = blockIdx.y * blockDim.y + threadIdx.y;
    if (q >= nq || j >= p.ny) return;
    const int32_t k0 = blockIdx.z * p.kc;
    const int32_t k1 = min(k0 + p.kc, p.nz);

    const int32_t i = q * V;
    const int32_t im = (i == 0) ? p.nx - 1 : i - 1;
    const int32_t ip = (i + V == p.nx) ? 0 : i + V;
    const int32_t jm = (j == 0) ? p.ny - 1 : j - 1;
    const int32_t jp = (j + 1 == p.ny) ? 0 : j + 1;
    const int64_t plane = (int64_t)p.nx * p.ny;
    const int64_t row = (int64_t)j * p.nx, rowm = (int64_t)jm * p.nx, rowp = (int64_t)jp * p.nx;

    // the row, the rows beside it and the values beyond the vector's ends, within a plane (node indices fit 32 bits)
    const int32_t at = (int32_t)row + i, atm = (int32_t)rowm + i, atp = (int32_t)rowp + i;
    const int32_t left = (int32_t)row + im, right = (int32_t)row + ip;
    auto load = [&](int32_t k) {
        Level<T, V> l;
        const int32_t o = k * (int32_t)plane;
        l.xx = ldp<T, V>(p.txx + o + at);
        l.xxl = __ldg(p.txx + o + left);
        l.xxr = __ldg(p.txx + o + right);
        l.xy = ldp<T, V>(p.txy + o + at);
        l.xyl = __ldg(p.txy + o + left);
        l.xyr = __ldg(p.txy + o + right);
        l.xyjm = ldp<T, V>(p.txy + o + atm);
        l.xyjp = ldp<T, V>(p.txy + o + atp);
        l.yyjm = ldp<T, V>(p.tyy + o + atm);
        l.yyjp = ldp<T, V>(p.tyy + o + atp);
        l.yzjm = ldp<T, V>(p.tyz + o + atm);
        l.yzjp = ldp<T, V>(p.tyz + o + atp);
        l.xzl = __ldg(p.txz + o + left);
        l.xzr = __ldg(p.txz + o + right);
        l.zz = ldp<T, V>(p.tzz + o + at);
        const int32_t up = k == p.nz - 1 ? o : o + (int32_t)plane;
        l.xz_kp = ldp<T, V>(p.txz + up + at);
        l.yz_kp = ldp<T, V>(p.tyz + up + at);
        return l;
    };
    const int32_t first = k0 * (int32_t)plane + at;
    Pack<T, V> xz_k = ldp<T, V>(p.txz + first);
    Pack<T, V> yz_k = ldp<T, V>(p.tyz + first);
    Pack<T, V> zz_km;
    for (int e = 0; e < V; ++e) zz_km.v[e] = T(0);
    if (k0 > 0) zz_km = ldp<T, V>(p.tzz + first - (int32_t)plane);

    for (int32_t k = k0; k < k1; ++k) {
        const Level<T, V> l = load(k);
        const int32_t o = k * (int32_t)plane + at;
        const bool top = (k == p.nz - 1);
        Pack<T, V> Fx, Fy, Fz;
#pragma unroll
        for (int e = 0; e < V; ++e) {
            const T xxm = e == 0 ? l.xxl : l.xx.v[e - 1], xxp = e == V - 1 ? l.xxr : l.xx.v[e + 1];
            const T xym = e == 0 ? l.xyl : l.xy.v[e - 1], xyp = e == V - 1 ? l.xyr : l.xy.v[e + 1];
            const T xzm = e == 0 ? l.xzl : xz_k.v[e - 1], xzp = e == V - 1 ? l.xzr : xz_k.v[e + 1];
            const T fx = -((xxp - xxm) * p.cx + (l.xyjp.v[e] - l.xyjm.v[e]) * p.cy + (l.xz_kp.v[e] - xz_k.v[e]) * p.cz);
            const T fy = -((xyp - xym) * p.cx + (l.yyjp.v[e] - l.yyjm.v[e]) * p.cy + (l.yz_kp.v[e] - yz_k.v[e]) * p.cz);
            const T fz = -((xzp - xzm) * p.cx + (l.yzjp.v[e] - l.yzjm.v[e]) * p.cy + (l.zz.v[e] - zz_km.v[e]) * p.cz);
            Fx.v[e] = top ? T(0) : fx;
            Fy.v[e] = top ? T(0) : fy;
            Fz.v[e] = (top || k == 0) ? T(0) : fz;
        }
        stp<T, V>(p.fx + o, Fx);
        stp<T, V>(p.fy + o, Fy);
        stp<T, V>(p.fz + o, Fz);
        xz_k = l.xz_kp;
        yz_k = l.yz_kp;
        zz_km = l.zz;
    }
}

template <typename T, int V>
int launch(wmibm_handle *h, const void *const tau[6], void *fx, void *fy, void *fz, cudaStream_t stream, int bx,
           int by, int kc)
{
    ForceParams<T> p;
    p.txx = (const T *)tau[0]; p.txy = (const T *)tau[1]; p.tyy = (const T *)tau[2];
    p.tzz = (const T *)tau[3]; p.txz = (const T *)tau[4]; p.tyz = (const T *)tau[5];
    p.fx = (T *)fx; p.fy = (T *)fy; p.fz = (T *)fz;
    p.nx = h->nx; p.ny = h->ny; p.nz = h->nz; p.kc = kc;
    p.cx = (T)(1.0 / (2.0 * h->dx));
    p.cy = (T)(1.0 / (2.0 * h->dy));
    p.cz = (T)(1.0 / h->dz);
    const int nq = h->nx / V;
    if (bx <= 0) {
        // default: blocks of equal width, at most a warp, and as many rows as 256 threads hold
        const int across = (nq + 31) / 32;
        bx = (nq + across - 1) / across;
        by = by > 0 ? by : 256 / bx;
    }
    if (by <= 0) by = 8;
    if (bx > nq) bx = nq;
    if (bx * by > 256) by = 256 / bx;
    if (by < 1) by = 1;
    dim3 block(bx, by, 1);
    dim3 grid((nq + bx - 1) / bx, (h->ny + by - 1) / by, (h->nz + kc - 1) / kc);
    if (grid.y > 65535 || grid.z > 65535) return set_error(h, WMIBM_EINVAL, "grid too large for the force launch");
    k_force<T, V><<<grid, block, 0, stream>>>(p);
    return cuda_status(h, cudaGetLastError(), "k_force launch");
}

bool aligned16(const void *p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace

namespace wmibm {

// Tile of the force launch: bx vectors along x, by rows, kc levels per thread.
int force_impl(wmibm_handle *h, const void *const tau[6], void *fx, void *fy, void *fz, cudaStream_t stream, int bx,
               int by, int kc)
{
    if (kc < 1) kc = 1;
    bool al = aligned16(fx) && aligned16(fy) && aligned16(fz);
    for (int c = 0; c < 6; ++c) al = al && aligned16(tau[c]);
    if (h->dtype == WMIBM_F64) {
        if (al && h->nx % 2 == 0) return launch<double, 2>(h, tau, fx, fy, fz, stream, bx, by, kc);
        return launch<double, 1>(h, tau, fx, fy, fz, stream, bx, by, kc);
    }
    if (al && h->nx % 4 == 0) return launch<float, 4>(h, tau, fx, fy, fz, stream, bx, by, kc);
    bool al8 = h->nx % 2 == 0 && ((uintptr_t)fx % 8) == 0 && ((uintptr_t)fy % 8) == 0 && ((uintptr_t)fz % 8) == 0;
    for (int c = 0; c < 6; ++c) al8 = al8 && ((uintptr_t)tau[c] % 8) == 0;
    if (al8) return launch<float, 2>(h, tau, fx, fy, fz, stream, bx, by, kc);
    return launch<float, 1>(h, tau, fx, fy, fz, stream, bx, by, kc);
}

void force_default_tile(const wmibm_handle *h, int *bx, int *by, int *kc)
{
    *bx = h->tuning.direct_bx;                              // 0: chosen at the launch
    *by = h->tuning.direct_by;
    *kc = h->tuning.direct_kc > 0 ? h->tuning.direct_kc : 4;
}

bool stencil_config(const wmibm_handle *h, const void *const tau[6], void *const f[3], StencilConfig *out);
int stencil_force(wmibm_handle *h, const void *const tau[6], void *const f[3], const StencilConfig &c,
                  cudaStream_t stream, wmibm_band_stats *emit);

// f = -div(tau): the bulk-copy pipeline where it applies, else the direct-load kernel.
int force_any(wmibm_handle *h, const void *const tau[6], void *fx, void *fy, void *fz, cudaStream_t stream)
{
    void *const f[3] = {fx, fy, fz};
    StencilConfig c;
    if (stencil_config(h, tau, f, &c)) return stencil_force(h, tau, f, c, stream, nullptr);
    int bx, by, kc;
    force_default_tile(h, &bx, &by, &kc);
    return force_impl(h, tau, fx, fy, fz, stream, bx, by, kc);
}

}  // namespace wmibm

extern "C" int wmibm_force(wmibm_handle *h, const void *const tau[6], void *fx, void *fy, void *fz, void *stream)
{
    ApiRange nvtx_range("wmibm_force");
    if (!h) return set_error(nullptr, WMIBM_EINVAL, "NULL handle");
    if (!tau || !fx || !fy || !fz) return set_error(h, WMIBM_EINVAL, "NULL stress or force pointer");
    for (int c = 0; c < 6; ++c)
        if (!tau[c]) return set_error(h, WMIBM_EINVAL, "NULL stress pointer %d", c);
    int st = check_device(h);
    if (st) return st;
    return force_any(h, tau, fx, fy, fz, (cudaStream_t)stream);
}
