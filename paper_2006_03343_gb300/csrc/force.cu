// The forcing f = -div(tau) on the vertically staggered grid (Eq. 2 and Eq. 18
// of Liu & Stevens, arXiv:2006.03343; vertical differences of Eqs. 15-16,
// horizontal derivatives by periodic second-order central differences):
//   f_x(uv k) = -[(txx[i+1]-txx[i-1])/2dx + (txy[j+1]-txy[j-1])/2dy + (txz[k+1]-txz[k])/dz]
//   f_y(uv k) = -[(txy[i+1]-txy[i-1])/2dx + (tyy[j+1]-tyy[j-1])/2dy + (tyz[k+1]-tyz[k])/dz]
//   f_z(w k)  = -[(txz[i+1]-txz[i-1])/2dx + (tyz[j+1]-tyz[j-1])/2dy + (tzz[k]-tzz[k-1])/dz]
// with f_x = f_y = 0 on the ghost uv level and f_z = 0 on the floor and lid.
//
// The kernels are in stencil.cu.
#include "internal.cuh"

using namespace wmibm;

namespace wmibm {

bool use_direct(const wmibm_handle *h, const void *const tau[6], void *const f[3], StencilConfig *c);
int direct_stage(wmibm_handle *h, const void *const tau[6], const void *const own[6], void *const f[3], void *u,
                 void *v, void *w, const void *const gradp[3], double dt, int do_mask, bool after, bool pdl,
                 cudaStream_t stream, wmibm_band_stats *emit);
int stencil_force(wmibm_handle *h, const void *const tau[6], void *const f[3], const StencilConfig &c,
                  cudaStream_t stream);

// f = -div(tau): the direct-load kernel, or the bulk-copy pipeline where the tuning asks for it.
int force_any(wmibm_handle *h, const void *const tau[6], void *fx, void *fy, void *fz, cudaStream_t stream)
{
    void *const f[3] = {fx, fy, fz};
    StencilConfig c;
    if (use_direct(h, tau, f, &c))
        return direct_stage(h, tau, tau, f, nullptr, nullptr, nullptr, nullptr, 0.0, 0, false, false, stream, nullptr);
    return stencil_force(h, tau, f, c, stream);
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
