// Adjoint of one stage (wall stress of Sec. 3.3 of Liu & Stevens,
// arXiv:2006.03343, then f = -div tau of Eqs. 15-16 and Eq. 18) for the linear
// functional L = sum over nodes of (gx fx + gy fy + gz fz), with the per-cell
// roughness s = ln z0 as a parameter (C = kappa^2 / (ln phi_c - s)^2).
//
//   1. per band record: gam = dL/dtau at the node's stored components (the
//      transpose of the divergence, gathered from g around the node); with
//      r = U_r, rho = |r|, m = G n and q = r . m (G the symmetric matrix of gam),
//      L_node = -2 C rho q, so
//        dL/du_hat = P (-2 C (q r / rho + rho m)),  P = I - n n^T
//        dL/ds     = -2 rho q * 2 C / (ln phi_c - s)
//   2. per touched velocity node: dL/du = sum over the (record, corner) pairs of
//      the transpose map of (trilinear weight) * dL/du_hat, in ascending
//      (record, corner) order; per band cell: dL/ds = w-band part + uv-band part.
// No atomics: every output element is written by one thread in a fixed order,
// so the result is deterministic.
#include <algorithm>

#include "band.cuh"

using namespace wmibm;

namespace {

template <typename T>
struct AdjParams {
    const void *rec;
    int64_t nb_w, nrec;
    const T *gx, *gy, *gz;
    const void *u, *v, *w;
    const T *logz0;
    T log_phi_c, kappa, kappa2;
    int32_t nx, ny, nz;
    T hx, hy, hz;                 // 1 / (2 dx), 1 / (2 dy), 1 / dz
    T *grad;                      // [nrec][4]: dL/du_hat (3), dL/ds
    // gather
    const int32_t *keys, *offs, *ent;
    int64_t m_uv, m_w;
    const int32_t *band_w, *band_uv;   // ascending node lists of the two bands
    T *du, *dv, *dw, *ds;
    // zeroing of the gradient fields, by the blocks after the records' blocks
    int64_t n;                    // nodes per field
    int64_t record_blocks;
    int32_t vec16;                // the fields are 16-byte aligned and n * sizeof(T) is a multiple of 16
};

// Clears du, dv, dw (and ds) before the gather writes the touched nodes: zeroing
// block zb of nzb, grid-stride, 16-byte stores where the fields allow.
template <typename T>
__device__ void zero_gradients(const AdjParams<T> &p, int64_t zb, int64_t nzb)
{
    T *const outs[4] = {p.du, p.dv, p.dw, p.ds};
    const int64_t first = zb * kThreads + threadIdx.x, stride = nzb * kThreads;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        T *o = outs[f];
        if (!o) continue;
        if (p.vec16) {
            const int64_t n4 = p.n * (int64_t)sizeof(T) / 16;
            for (int64_t q = first; q < n4; q += stride) reinterpret_cast<float4 *>(o)[q] = make_float4(0, 0, 0, 0);
        } else {
            for (int64_t q = first; q < p.n; q += stride) o[q] = T(0);
        }
    }
}

// Blocks [0, record_blocks): one band record per thread.  The blocks after them
// clear the gradient fields meanwhile (the gather, next in the stream, writes the
// touched nodes after both).
template <typename T, typename VEL>
__global__ void __launch_bounds__(kThreads) k_adjoint_records(AdjParams<T> p)
{
    using Rec = typename RecOf<T>::type;
    if ((int64_t)blockIdx.x >= p.record_blocks) {
        zero_gradients(p, (int64_t)blockIdx.x - p.record_blocks, (int64_t)gridDim.x - p.record_blocks);
        return;
    }
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= p.nrec) return;
    T nxv, nyv, nzv, C, ax, ay, azu, azw;
    int4 ix;
    unpack(reinterpret_cast<const Rec *>(p.rec), t, nxv, nyv, nzv, C, ax, ay, azu, azw, ix);
    const bool is_w = t < p.nb_w;
    const int32_t nx = p.nx, ny = p.ny, nz = p.nz;
    const int64_t plane = (int64_t)nx * ny;
    const int64_t di = (ix.w & 1) ? 1 - nx : 1;
    const int64_t dj = (ix.w & 2) ? (int64_t)(1 - ny) * nx : nx;
    const T uc = trilinear<VEL, T>(reinterpret_cast<const VEL *>(p.u), ix.y, di, dj, plane, ax, ay, azu);
    const T vc = trilinear<VEL, T>(reinterpret_cast<const VEL *>(p.v), ix.y, di, dj, plane, ax, ay, azu);
    const T wc = trilinear<VEL, T>(reinterpret_cast<const VEL *>(p.w), ix.z, di, dj, plane, ax, ay, azw);
    T lg;
    if (p.logz0) {
        lg = p.log_phi_c - __ldg(p.logz0 + ix.x);
        C = p.kappa2 / (lg * lg);
    } else {
        lg = p.kappa / sqrt(C);             // C = kappa^2 / lg^2 with lg = ln(phi_c / z0) > 0
    }

    // node coordinates and its horizontal neighbours (periodic)
    const int64_t idx = ix.x;
    const int32_t k = (int32_t)(idx / plane);
    const int64_t rem = idx - (int64_t)k * plane;
    const int32_t j = (int32_t)(rem / nx);
    const int32_t i = (int32_t)(rem - (int64_t)j * nx);
    const int64_t row = idx - i, lev = idx - rem;
    const int64_t ip = row + (i + 1 == nx ? 0 : i + 1), im = row + (i == 0 ? nx - 1 : i - 1);
    const int64_t jp = lev + (int64_t)(j + 1 == ny ? 0 : j + 1) * nx + i;
    const int64_t jm = lev + (int64_t)(j == 0 ? ny - 1 : j - 1) * nx + i;
    const bool fx_on = k <= nz - 2;                  // f_x, f_y at uv level k (not the ghost level)
    const bool fz_on = k >= 1 && k <= nz - 2;        // f_z at w level k (not floor or lid)

    T mx, my, mz;                                     // m = G n
    if (is_w) {
        // txz at w level k enters f_x at uv levels k-1 and k, and f_z at w level k
        T gxz = p.hz * ((fx_on ? __ldg(p.gx + idx) : T(0)) - (k >= 1 ? __ldg(p.gx + idx - plane) : T(0)));
        T gyz = p.hz * ((fx_on ? __ldg(p.gy + idx) : T(0)) - (k >= 1 ? __ldg(p.gy + idx - plane) : T(0)));
        if (fz_on) {
            gxz += p.hx * (__ldg(p.gz + ip) - __ldg(p.gz + im));
            gyz += p.hy * (__ldg(p.gz + jp) - __ldg(p.gz + jm));
        }
        mx = T(0.5) * gxz * nzv;
        my = T(0.5) * gyz * nzv;
        mz = T(0.5) * (gxz * nxv + gyz * nyv);
    } else {
        T gxx = T(0), gxy = T(0), gyy = T(0);
        if (fx_on) {
            gxx = p.hx * (__ldg(p.gx + ip) - __ldg(p.gx + im));
            gxy = p.hy * (__ldg(p.gx + jp) - __ldg(p.gx + jm)) + p.hx * (__ldg(p.gy + ip) - __ldg(p.gy + im));
            gyy = p.hy * (__ldg(p.gy + jp) - __ldg(p.gy + jm));
        }
        // tzz at uv level k enters f_z at w levels k and k+1
        const T gzz = p.hz * ((k <= nz - 3 ? __ldg(p.gz + idx + plane) : T(0)) - (fz_on ? __ldg(p.gz + idx) : T(0)));
        mx = gxx * nxv + T(0.5) * gxy * nyv;
        my = T(0.5) * gxy * nxv + gyy * nyv;
        mz = gzz * nzv;
    }

    const T un = uc * nxv + vc * nyv + wc * nzv;
    const T rx = uc - un * nxv, ry = vc - un * nyv, rz = wc - un * nzv;
    const T rho = sqrt(rx * rx + ry * ry + rz * rz);
    T o0 = T(0), o1 = T(0), o2 = T(0), o3 = T(0);
    if (rho > T(0)) {
        const T q = rx * mx + ry * my + rz * mz;
        const T a = -T(2) * C;
        const T dx_ = a * (q * rx / rho + rho * mx);
        const T dy_ = a * (q * ry / rho + rho * my);
        const T dz_ = a * (q * rz / rho + rho * mz);
        const T nd = nxv * dx_ + nyv * dy_ + nzv * dz_;
        o0 = dx_ - nd * nxv;
        o1 = dy_ - nd * nyv;
        o2 = dz_ - nd * nzv;
        o3 = -T(2) * rho * q * (T(2) * C / lg);
    }
    T *g = p.grad + 4 * t;
    g[0] = o0;
    g[1] = o1;
    g[2] = o2;
    g[3] = o3;
}

// Position of node idx in an ascending list, or -1.
__device__ __forceinline__ int64_t find_node(const int32_t *list, int64_t n, int32_t idx)
{
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (__ldg(list + mid) < idx)
            lo = mid + 1;
        else
            hi = mid;
    }
    return (lo < n && __ldg(list + lo) == idx) ? lo : -1;
}

template <typename T>
__device__ __forceinline__ T corner_weight(int c, T ax, T ay, T az)
{
    const T wx = (c & 1) ? ax : T(1) - ax;
    const T wy = (c & 2) ? ay : T(1) - ay;
    const T wz = (c & 4) ? az : T(1) - az;
    return wx * wy * wz;
}

// Threads [0, m_uv): touched uv-grid nodes (du, dv); [m_uv, m_uv + m_w): touched
// w-grid nodes (dw); then one thread per band record for dL/ds (if wanted).
template <typename T>
__global__ void __launch_bounds__(kThreads) k_adjoint_gather(AdjParams<T> p)
{
    using Rec = typename RecOf<T>::type;
    const Rec *rec = reinterpret_cast<const Rec *>(p.rec);
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const int64_t m = p.m_uv + p.m_w;
    if (t < m) {
        const bool uv = t < p.m_uv;
        const int32_t node = __ldg(p.keys + t);
        T s0 = T(0), s1 = T(0);
        for (int32_t e = __ldg(p.offs + t); e < __ldg(p.offs + t + 1); ++e) {
            const int32_t code = __ldg(p.ent + e);
            const int64_t r = code >> 3;
            T nxv, nyv, nzv, C, ax, ay, azu, azw;
            int4 ix;
            unpack(rec, r, nxv, nyv, nzv, C, ax, ay, azu, azw, ix);
            const T wt = corner_weight<T>(code & 7, ax, ay, uv ? azu : azw);
            if (uv) {
                s0 += wt * p.grad[4 * r + 0];
                s1 += wt * p.grad[4 * r + 1];
            } else {
                s0 += wt * p.grad[4 * r + 2];
            }
        }
        if (uv) {
            p.du[node] = s0;
            p.dv[node] = s1;
        } else {
            p.dw[node] = s0;
        }
        return;
    }
    const int64_t r = t - m;
    if (!p.ds || r >= p.nrec) return;
    const int32_t idx = __ldg(&rec[r].ix).x;
    if (r < p.nb_w) {
        // the cell's uv-band record, if any, writes the sum
        if (find_node(p.band_uv, p.nrec - p.nb_w, idx) >= 0) return;
        p.ds[idx] = p.grad[4 * r + 3];
    } else {
        const int64_t tw = find_node(p.band_w, p.nb_w, idx);
        const T a = tw >= 0 ? p.grad[4 * tw + 3] : T(0);
        p.ds[idx] = a + p.grad[4 * r + 3];    // w-band part first, then the uv-band part
    }
}

// ---------------------------------------------------------------------------
// The transpose of the trilinear gathers, built once per handle: every node that
// some record's stencil touches (uv-grid nodes, then w-grid nodes, ascending in
// each), and for each its (record * 8 + corner) entries, ascending.  A slot per node
// and grid counts the entries, a scan over the slots lays out the keys and offsets,
// the entries go to their node in any order and each node's few are sorted.  (Sorting
// all entries on the host took 32 ms for the 131,072 records of 256 x 128 x 128
// hills; this form, with its allocations, under 2 ms.)
// The slots take 8 bytes a node while the map is built.  Where that is not to be had, the
// chunks of slots are gone through in windows, whose entries are counted once for the
// totals and once more for the places: a window of 4 MB is asked for at last.
constexpr int kMapChunk = 4096;                 // slots per block of the scan
constexpr int kMapPer = kMapChunk / kThreads;   // and per thread
constexpr int64_t kMapWindow = 256;             // chunks of the smallest window

// Slot of corner c of record r on grid g (0: uv, 1: w), each grid's from a new chunk on.
template <typename T>
__device__ __forceinline__ int64_t map_slot(const void *rec, int64_t r, int g, int c, int32_t nx, int32_t ny,
                                            int64_t per_grid)
{
    const int4 ix = __ldg(&reinterpret_cast<const typename RecOf<T>::type *>(rec)[r].ix);
    const int64_t plane = (int64_t)nx * ny;
    const int64_t di = (ix.w & 1) ? 1 - nx : 1;
    const int64_t dj = (ix.w & 2) ? (int64_t)(1 - ny) * nx : nx;
    return g * per_grid * kMapChunk + (g ? ix.z : ix.y) + ((c & 1) ? di : 0) + ((c & 2) ? dj : 0) +
           ((c & 4) ? plane : 0);
}

// One thread per record, grid and corner; slots holds those of chunks [c0, c1).
// FILL = false: counts the entries of each slot; true: takes the slot's next place for
// the entry.
template <typename T, bool FILL>
__global__ void __launch_bounds__(kThreads) k_map_entries(const void *rec, int64_t nrec, int32_t nx, int32_t ny,
                                                          int64_t per_grid, int64_t c0, int64_t c1, int32_t *slots,
                                                          int32_t *ent)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= 16 * nrec) return;
    const int c = (int)(t & 7), g = (int)((t >> 3) & 1);
    const int64_t r = t >> 4;
    const int64_t slot = map_slot<T>(rec, r, g, c, nx, ny, per_grid) - c0 * kMapChunk;
    if (slot < 0 || slot >= (c1 - c0) * kMapChunk) return;
    const int32_t at = atomicAdd(slots + slot, 1);
    if (FILL) ent[at] = (int32_t)(r * 8 + c);
}

// A thread's nodes of chunk c, [first, first + count) of its grid's n.
__device__ __forceinline__ void map_range(int64_t n, int64_t per_grid, int64_t c, int64_t &first, int &count)
{
    first = (c >= per_grid ? c - per_grid : c) * kMapChunk + threadIdx.x * kMapPer;
    count = (int)min((int64_t)kMapPer, max((int64_t)0, n - first));
}

// Exclusive prefix of v over the block (x: touched slots, y: entries); total: the block's sum.
__device__ __forceinline__ int2 block_prefix(int2 v, int2 &total)
{
    __shared__ int2 warps[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    int2 s = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, s.x, o), y = __shfl_up_sync(0xffffffffu, s.y, o);
        if (lane >= o) {
            s.x += x;
            s.y += y;
        }
    }
    if (lane == 31) warps[warp] = s;
    __syncthreads();
    int2 before = make_int2(s.x - v.x, s.y - v.y);
    total = make_int2(0, 0);
    for (int w = 0; w < nwarps; ++w) {
        if (w < warp) {
            before.x += warps[w].x;
            before.y += warps[w].y;
        }
        total.x += warps[w].x;
        total.y += warps[w].y;
    }
    __syncthreads();
    return before;
}

// One block per chunk from c0 on.  WRITE = false: the chunk's touched slots and entries
// into sums; true: from the chunk's prefix in sums, the keys and offsets of its touched
// slots, whose counts become the places of their first entries.
template <bool WRITE>
__global__ void __launch_bounds__(kThreads) k_map_scan(int32_t *slots, int64_t n, int64_t per_grid, int64_t c0,
                                                       int2 *sums, int32_t *keys, int32_t *offs)
{
    const int64_t c = c0 + blockIdx.x;
    int32_t *const own = slots + (int64_t)blockIdx.x * kMapChunk + threadIdx.x * kMapPer;
    int64_t first;
    int count;
    map_range(n, per_grid, c, first, count);
    int2 v = make_int2(0, 0), total;
    for (int q = 0; q < count; ++q) {
        const int e = own[q];
        v.x += e != 0;
        v.y += e;
    }
    const int2 before = block_prefix(v, total);
    if (!WRITE) {
        if (threadIdx.x == 0) sums[c] = total;
        return;
    }
    int2 at = make_int2(sums[c].x + before.x, sums[c].y + before.y);
    for (int q = 0; q < count; ++q) {
        const int e = own[q];
        if (e == 0) continue;
        keys[at.x] = (int32_t)(first + q);
        offs[at.x] = at.y;
        own[q] = at.y;
        ++at.x;
        at.y += e;
    }
}

// Exclusive prefix over the chunks' sums, in one block; sums[count] receives the totals.
__global__ void __launch_bounds__(1024) k_map_totals(int2 *sums, int count)
{
    int2 carry = make_int2(0, 0);
    for (int base = 0; base < count; base += 1024) {
        const int q = base + threadIdx.x;
        const int2 v = q < count ? sums[q] : make_int2(0, 0);
        int2 total;
        const int2 before = block_prefix(v, total);
        if (q < count) sums[q] = make_int2(carry.x + before.x, carry.y + before.y);
        carry.x += total.x;
        carry.y += total.y;
    }
    if (threadIdx.x == 0) sums[count] = carry;
}

// Restores the heap of a[0 .. end) below root.
__device__ __forceinline__ void sift(int32_t *a, int root, int end)
{
    const int32_t v = a[root];
    for (int child = 2 * root + 1; child < end; child = 2 * root + 1) {
        if (child + 1 < end && a[child + 1] > a[child]) ++child;
        if (a[child] <= v) break;
        a[root] = a[child];
        root = child;
    }
    a[root] = v;
}

// Each touched node's entries, ascending: insertion for the usual few, a heap for many.
__global__ void __launch_bounds__(kThreads) k_map_sort(const int32_t *offs, int64_t m, int32_t total, int32_t *ent)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= m) return;
    int32_t *const a = ent + offs[t];
    const int len = (t + 1 < m ? offs[t + 1] : total) - offs[t];
    if (len <= 48) {
        for (int i = 1; i < len; ++i) {
            const int32_t v = a[i];
            int j = i;
            for (; j > 0 && a[j - 1] > v; --j) a[j] = a[j - 1];
            a[j] = v;
        }
        return;
    }
    for (int i = len / 2 - 1; i >= 0; --i) sift(a, i, len);
    for (int end = len - 1; end > 0; --end) {
        const int32_t v = a[0];
        a[0] = a[end];
        a[end] = v;
        sift(a, 0, end);
    }
}

// The map with a window of `window` chunks' slots at a time.
template <typename T>
cudaError_t build_map(wmibm_handle *h, int64_t window, cudaStream_t stream)
{
    const int64_t n = h->n, entries = 16 * h->nrec, per_grid = (n + kMapChunk - 1) / kMapChunk, chunks = 2 * per_grid;
    const unsigned eblocks = (unsigned)((entries + kThreads - 1) / kThreads);
    int32_t *slots = nullptr;
    int2 *sums = nullptr;
    int2 ends[2];                               // touched slots of the uv-grid; of both, and the entries
    cudaError_t e = dev_alloc(&slots, window * kMapChunk * sizeof(int32_t));
    if (e == cudaSuccess) e = dev_alloc(&sums, (chunks + 1) * sizeof(int2));
    auto count = [&](int64_t c0, int64_t c1) {
        e = cudaMemsetAsync(slots, 0, (c1 - c0) * kMapChunk * sizeof(int32_t), stream);
        if (e != cudaSuccess) return;
        k_map_entries<T, false><<<eblocks, kThreads, 0, stream>>>(h->rec, h->nrec, h->nx, h->ny, per_grid, c0, c1, slots,
                                                                  nullptr);
        e = cudaGetLastError();
    };
    for (int64_t c0 = 0; e == cudaSuccess && c0 < chunks; c0 += window) {
        const int64_t c1 = std::min(c0 + window, chunks);
        count(c0, c1);
        if (e != cudaSuccess) break;
        k_map_scan<false><<<(unsigned)(c1 - c0), kThreads, 0, stream>>>(slots, n, per_grid, c0, sums, nullptr, nullptr);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        k_map_totals<<<1, 1024, 0, stream>>>(sums, (int)chunks);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&ends[0], sums + per_grid, sizeof(int2), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&ends[1], sums + chunks, sizeof(int2), cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    const int64_t m = e == cudaSuccess ? ends[1].x : 0;
    if (e == cudaSuccess) e = dev_alloc(&h->adj_keys, m * sizeof(int32_t));
    if (e == cudaSuccess) e = dev_alloc(&h->adj_offs, (m + 1) * sizeof(int32_t));
    if (e == cudaSuccess) e = dev_alloc(&h->adj_ent, entries * sizeof(int32_t));
    if (e == cudaSuccess) e = dev_alloc(&h->adj_grad, (size_t)h->nrec * 4 * sizeof(T));
    for (int64_t c0 = 0; e == cudaSuccess && c0 < chunks; c0 += window) {
        const int64_t c1 = std::min(c0 + window, chunks);
        if (window < chunks) count(c0, c1);     // else the counts are still there
        if (e != cudaSuccess) break;
        k_map_scan<true><<<(unsigned)(c1 - c0), kThreads, 0, stream>>>(slots, n, per_grid, c0, sums, h->adj_keys,
                                                                       h->adj_offs);
        k_map_entries<T, true><<<eblocks, kThreads, 0, stream>>>(h->rec, h->nrec, h->nx, h->ny, per_grid, c0, c1, slots,
                                                                 h->adj_ent);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        const int32_t total = (int32_t)entries;
        k_map_sort<<<(unsigned)((m + kThreads - 1) / kThreads), kThreads, 0, stream>>>(h->adj_offs, m, total, h->adj_ent);
        e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(h->adj_offs + m, &total, sizeof(int32_t), cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    }
    cudaFree(slots);
    cudaFree(sums);
    if (e != cudaSuccess) {
        cudaFree(h->adj_keys);
        cudaFree(h->adj_offs);
        cudaFree(h->adj_ent);
        cudaFree(h->adj_grad);
        h->adj_keys = h->adj_offs = h->adj_ent = nullptr;
        h->adj_grad = nullptr;
        return e;
    }
    h->adj_m[0] = ends[0].x;
    h->adj_m[1] = m - ends[0].x;
    return cudaSuccess;
}

// Builds the transpose map of the trilinear gathers (once per handle).
int ensure_adjoint_map(wmibm_handle *h, cudaStream_t stream)
{
    if (h->adj_grad || h->nrec == 0) return WMIBM_OK;
    // entry codes (record * 8 + corner) and offsets (16 entries per record) stay below 2^31
    if (h->nrec >= (int64_t(1) << 27)) return set_error(h, WMIBM_EINVAL, "too many band records for the adjoint map");
    cudaError_t e = cudaErrorMemoryAllocation;
    for (int64_t window = 2 * ((h->n + kMapChunk - 1) / kMapChunk);; window = std::max(window / 4, kMapWindow)) {
        e = h->dtype == WMIBM_F64 ? build_map<double>(h, window, stream) : build_map<float>(h, window, stream);
        if (e != cudaErrorMemoryAllocation || window <= kMapWindow) break;
        (void)cudaGetLastError();
    }
    return e == cudaSuccess ? WMIBM_OK : cuda_status(h, e, "adjoint map");
}

template <typename T, typename VEL>
int backward_impl(wmibm_handle *h, const void *const g[3], const void *const uvw[3], void *du, void *dv, void *dw,
                  void *dlogz0, cudaStream_t stream)
{
    AdjParams<T> p = {};
    p.rec = h->rec;
    p.nb_w = h->lists.n[WMIBM_LIST_BAND_W];
    p.nrec = h->nrec;
    p.gx = (const T *)g[0];
    p.gy = (const T *)g[1];
    p.gz = (const T *)g[2];
    p.u = uvw[0];
    p.v = uvw[1];
    p.w = uvw[2];
    p.logz0 = (const T *)h->logz0;
    p.log_phi_c = (T)log(h->phi_c);
    p.kappa = (T)h->kappa;
    p.kappa2 = (T)(h->kappa * h->kappa);
    p.nx = h->nx;
    p.ny = h->ny;
    p.nz = h->nz;
    p.hx = (T)(1.0 / (2.0 * h->dx));
    p.hy = (T)(1.0 / (2.0 * h->dy));
    p.hz = (T)(1.0 / h->dz);
    p.grad = (T *)h->adj_grad;
    p.keys = h->adj_keys;
    p.offs = h->adj_offs;
    p.ent = h->adj_ent;
    p.m_uv = h->adj_m[0];
    p.m_w = h->adj_m[1];
    p.band_w = h->lists.p[WMIBM_LIST_BAND_W];
    p.band_uv = h->lists.p[WMIBM_LIST_BAND_UV];
    p.du = (T *)du;
    p.dv = (T *)dv;
    p.dw = (T *)dw;
    p.ds = (T *)dlogz0;
    p.n = h->n;
    bool al = (h->n * (int64_t)sizeof(T)) % 16 == 0;
    const void *const outs[4] = {du, dv, dw, dlogz0};
    for (int f = 0; f < 4; ++f) al = al && ((uintptr_t)outs[f] & 15u) == 0;
    p.vec16 = al ? 1 : 0;
    // records' blocks, then zeroing blocks: about two per SM, at most one per 1024 vectors
    const int64_t b1 = (h->nrec + kThreads - 1) / kThreads;
    int64_t bz = (h->n * (int64_t)sizeof(T) / 16 + 4 * kThreads - 1) / (4 * kThreads);
    if (bz > 2 * (int64_t)h->sm_count) bz = 2 * (int64_t)h->sm_count;
    if (bz < 1) bz = 1;
    p.record_blocks = b1;
    k_adjoint_records<T, VEL><<<(unsigned)(b1 + bz), kThreads, 0, stream>>>(p);
    int st = cuda_status(h, cudaGetLastError(), "k_adjoint_records launch");
    if (st) return st;
    if (h->nrec == 0) return WMIBM_OK;
    const int64_t total = p.m_uv + p.m_w + (dlogz0 ? h->nrec : 0);
    const unsigned b2 = (unsigned)((total + kThreads - 1) / kThreads);
    k_adjoint_gather<T><<<b2, kThreads, 0, stream>>>(p);
    return cuda_status(h, cudaGetLastError(), "k_adjoint_gather launch");
}

}  // namespace

extern "C" int wmibm_set_log_z0(wmibm_handle *h, const void *logz0, void *stream)
{
    ApiRange nvtx_range("wmibm_set_log_z0");
    if (!h) return set_error(nullptr, WMIBM_EINVAL, "NULL handle");
    int st = check_device(h);
    if (st) return st;
    if (logz0 && ((uintptr_t)logz0 % elem_size(h->dtype)) != 0)
        return set_error(h, WMIBM_EINVAL, "logz0 is not aligned to its element size");
    st = ensure_adjoint_map(h, (cudaStream_t)stream);
    if (st) return st;
    h->logz0 = logz0;
    return WMIBM_OK;
}

extern "C" int wmibm_backward(wmibm_handle *h, const void *const g[3], const void *const uvw[3], void *du,
                              void *dv, void *dw, void *dlogz0, void *stream)
{
    ApiRange nvtx_range("wmibm_backward");
    if (!h) return set_error(nullptr, WMIBM_EINVAL, "NULL handle");
    if (!g || !g[0] || !g[1] || !g[2]) return set_error(h, WMIBM_EINVAL, "NULL forcing weight g");
    if (!uvw || !uvw[0] || !uvw[1] || !uvw[2]) return set_error(h, WMIBM_EINVAL, "NULL velocity pointer");
    if (!du || !dv || !dw) return set_error(h, WMIBM_EINVAL, "NULL velocity gradient pointer");
    int st = check_device(h);
    if (st) return st;
    st = ensure_adjoint_map(h, (cudaStream_t)stream);
    if (st) return st;
    if (h->dtype == WMIBM_F64) return backward_impl<double, double>(h, g, uvw, du, dv, dw, dlogz0, (cudaStream_t)stream);
    if (h->vel_dtype == WMIBM_BF16)
        return backward_impl<float, __nv_bfloat16>(h, g, uvw, du, dv, dw, dlogz0, (cudaStream_t)stream);
    return backward_impl<float, float>(h, g, uvw, du, dv, dw, dlogz0, (cudaStream_t)stream);
}
