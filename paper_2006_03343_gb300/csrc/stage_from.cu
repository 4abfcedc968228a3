// The stage of wmibm_wall_stress_force on stresses that stay as they are: the
// entries that the wall model writes go to a work buffer.  Only the levels that
// hold band or solid nodes, and those that the stencil reads beside them, are
// copied there; every other level's units read the caller's stresses.
#include <algorithm>

#include "internal.cuh"

using namespace wmibm;

namespace wmibm {
int wall_model(wmibm_handle *h, const void *u, const void *v, const void *w, void *const tau[6],
               wmibm_band_stats *stats, const void *logz0, cudaStream_t stream, bool emit);
int direct_stage(wmibm_handle *h, const void *const tau[6], const void *const own[6], void *const f[3], void *u,
                 void *v, void *w, const void *const gradp[3], double dt, int do_mask, bool after, bool pdl,
                 cudaStream_t stream, wmibm_band_stats *emit);
}  // namespace wmibm

namespace {

struct CopyParams {
    const char *src[6];
    char *dst[6];
    int64_t bytes;              // per field
};

// Six contiguous copies in one launch.  V: the unit that every address and the size
// are multiples of.  HBM-bound: four independent 16-byte loads in flight per thread.
template <typename V>
__global__ void __launch_bounds__(kThreads) k_copy_levels(const __grid_constant__ CopyParams p)
{
    const int64_t n = p.bytes / (int64_t)sizeof(V), stride = (int64_t)gridDim.x * kThreads;
    const V *const src = reinterpret_cast<const V *>(p.src[blockIdx.y]);
    V *const dst = reinterpret_cast<V *>(p.dst[blockIdx.y]);
    int64_t q = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    for (; q + 3 * stride < n; q += 4 * stride) {
        const V a = src[q], b = src[q + stride], c = src[q + 2 * stride], d = src[q + 3 * stride];
        dst[q] = a;
        dst[q + stride] = b;
        dst[q + 2 * stride] = c;
        dst[q + 3 * stride] = d;
    }
    for (; q < n; q += stride) dst[q] = src[q];
}

// Levels [lo, hi) that the work buffer holds: those that the stencil reads for dirty
// levels (the one below, and the one above, too).
void work_levels(const wmibm_handle *h, int32_t *lo, int32_t *hi)
{
    *lo = *hi = 0;
    if (h->dirty_hi <= h->dirty_lo) return;
    *lo = std::max(h->dirty_lo - 1, 0);
    *hi = std::min(h->dirty_hi + 1, h->nz);
}

// Bytes of one field of the work buffer, padded so that each field starts on a 16-byte boundary.
int64_t field_bytes(const wmibm_handle *h, int32_t levels)
{
    const int64_t b = (int64_t)levels * h->nx * h->ny * (int64_t)elem_size(h->dtype);
    return (b + 15) / 16 * 16;
}

}  // namespace

extern "C" int64_t wmibm_stage_work_bytes(const wmibm_handle *h, const void *const tau[6], const void *fx,
                                          const void *fy, const void *fz)
{
    if (!h || !tau || !fx || !fy || !fz) return -1;
    for (int c = 0; c < 6; ++c)
        if (!tau[c]) return -1;
    int32_t lo, hi;
    work_levels(h, &lo, &hi);
    return 6 * field_bytes(h, hi - lo);
}

extern "C" int wmibm_wall_stress_force_from(wmibm_handle *h, const void *u, const void *v, const void *w,
                                            const void *const tau[6], void *work, int64_t work_bytes, void *fx, void *fy,
                                            void *fz, wmibm_band_stats *stats, void *stream)
{
    ApiRange nvtx_range("wmibm_wall_stress_force_from");
    if (!h) return set_error(nullptr, WMIBM_EINVAL, "NULL handle");
    if (!u || !v || !w || !tau || !fx || !fy || !fz)
        return set_error(h, WMIBM_EINVAL, "NULL velocity, stress or force pointer");
    for (int c = 0; c < 6; ++c)
        if (!tau[c]) return set_error(h, WMIBM_EINVAL, "NULL stress pointer %d", c);
    int st = check_device(h);
    if (st) return st;
    void *const f[3] = {fx, fy, fz};
    int32_t lo, hi;
    work_levels(h, &lo, &hi);
    const int64_t field = field_bytes(h, hi - lo);
    if (work_bytes < 6 * field || (field > 0 && (!work || ((uintptr_t)work & 15u) != 0)))
        return set_error(h, WMIBM_EINVAL, "the work buffer must be 16-byte aligned and hold %lld bytes",
                         (long long)(6 * field));
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t es = (int64_t)elem_size(h->dtype), level = (int64_t)h->nx * h->ny * es;
    CopyParams p;
    p.bytes = (int64_t)(hi - lo) * level;
    void *at[6];                // where a field of the buffer would start if it held level 0
    bool v16 = p.bytes % 16 == 0;
    for (int a = 0; a < 6; ++a) {
        p.src[a] = (const char *)tau[a] + (int64_t)lo * level;
        p.dst[a] = (char *)work + a * field;
        at[a] = (void *)((uintptr_t)p.dst[a] - (uintptr_t)((int64_t)lo * level));
        v16 = v16 && ((uintptr_t)p.src[a] & 15u) == 0;
    }
    if (p.bytes > 0) {
        const int64_t unit = v16 ? 16 : es, per = 4 * kThreads * unit;
        const int64_t blocks = std::min<int64_t>((p.bytes + per - 1) / per, 4 * (int64_t)h->sm_count);
        const dim3 grid((unsigned)blocks, 6);
        if (v16)
            k_copy_levels<uint4><<<grid, kThreads, 0, s>>>(p);
        else if (es == 8)
            k_copy_levels<uint2><<<grid, kThreads, 0, s>>>(p);
        else
            k_copy_levels<uint32_t><<<grid, kThreads, 0, s>>>(p);
        st = cuda_status(h, cudaGetLastError(), "k_copy_levels launch");
        if (st) return st;
    }
    st = wall_model(h, u, v, w, at, stats, h->logz0, s, false);
    if (st) return st;
    return direct_stage(h, tau, (const void *const *)at, f, nullptr, nullptr, nullptr, nullptr, 0.0, 0, true, true, s,
                        stats);
}
