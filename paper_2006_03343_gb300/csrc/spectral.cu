// The forcing f = -div(tau) with the paper's own horizontal scheme (Eq. 2 /
// Eq. 18 of Liu & Stevens, arXiv:2006.03343): x and y derivatives
// pseudo-spectral (Eqs. 13-14), vertical ones the staggered differences of
// Eqs. 15-16,
//   f_x(uv k) = -[d_x txx + d_y txy + (txz[k+1] - txz[k])/dz]
//   f_y(uv k) = -[d_x txy + d_y tyy + (tyz[k+1] - tyz[k])/dz]
//   f_z(w k)  = -[d_x txz + d_y tyz + (tzz[k] - tzz[k-1])/dz]
// with f_x = f_y = 0 on the ghost uv level and f_z = 0 on the floor and lid.
//
// The 2-D transform of Eqs. 13-14 factors by direction: multiplying the plane's
// amplitudes by i k_x touches the x index only, so d_x is the 1-D spectral
// derivative of every x-row and d_y that of every y-column.  The Nyquist bin of
// each direction carries no first derivative.  One persistent launch works
// through two kinds of unit:
//   row unit    (level k, rx rows): d_x of txx, txy, txz plus the vertical
//               terms -> writes the partial forcing into f
//   column unit (level k, wy columns): d_y of txy, tyy, tyz, subtracted from f
// Each unit stages its lines in shared memory, two real lines per complex
// sequence (z = a + i b; the derivative operator is real, so D z = D a + i D b), runs
// a decimation-in-frequency FFT in place (radix up to 16), whose last pass leaves the
// bins in digit-reversed order, multiplies them there by i k / N and conjugates them
// (IFFT(y) = conj(FFT(conj y))/N), and runs the transposed network, whose first pass
// takes the same elements: the two passes are one, no reordering is needed, and the
// result is in natural order.  Units are dispensed by an atomic ticket in chunks of kc levels:
// the row units of chunk c, then the column units of chunk c-1.  A column unit
// on level k waits (bounded) until all row units of level k have finished, so
// the partial forcing and the stresses the two unit kinds share are re-read
// from L2 while DRAM streams each array once.  Row units never wait, and every
// row unit a column unit depends on was dispensed earlier to a running block,
// so the waits end whatever the grid size.
#include <algorithm>
#include <math.h>
#include <stdlib.h>

#include "internal.cuh"
#include "tma.cuh"

namespace wmibm {

constexpr int kSpecMaxLog = 11;         // lines of up to 2048 points (FP32; 1024 for FP64)
constexpr int kSpecThreads = 192;
constexpr int kSpecBudget = 3300;       // complex elements per shared buffer aimed at (FP32; half for FP64)
// L2 footprint of one chunk of levels: below it the column units wait for their row
// units, above it their second reads miss L2 (hill, FP32: 12 / 24 / 32 / 48 / 72 MB: 967 /
// 742 / 761 / 789 / 797 us).
constexpr double kSpecChunkBytes = 24.0 * 1024 * 1024;
// limit of a block's shared memory: one value for every grid, as the limit belongs to the
// process and other threads may be launching
constexpr int kSpecSmemMax = 224 * 1024;

struct SpecState {
    int lognx, logny;
    int rx, wy;                 // rows per row unit, columns per column unit
    int ldx, ldy;               // shared-memory stride of a sequence (complex elements, skewed and padded)
    int kc, nchunks;
    int xpl, ypl;               // units per level
    int64_t total;
    int64_t buf;                // complex elements of the FFT buffer
    size_t smem;
    void *twx, *twy;            // twiddles of the passes (dtype complex)
    void *knx, *kny;            // k_m / N per bin in the FFT's digit-reversed order, Nyquist bin 0 (dtype)
    unsigned int *ctr;          // [0] ticket, [1] exit ticket, [2 + k] row units finished on level k
};

}  // namespace wmibm

using namespace wmibm;

namespace {

template <typename T>
struct Cx;
template <>
struct Cx<float> {
    using type = float2;
};
template <>
struct Cx<double> {
    using type = double2;
};

template <typename T>
struct SpecParams {
    const T *txx, *txy, *tyy, *tzz, *txz, *tyz;
    T *fx, *fy, *fz;
    const typename Cx<T>::type *twx, *twy;
    const T *knx, *kny;
    unsigned int *ctr;
    int *status;
    int32_t nx, ny, nz;
    int32_t lognx, logny, logrx, logwy;
    int32_t ldx, ldy;
    int32_t kc, nchunks, xpl, ypl;
    int64_t total;
    int32_t buf;              // complex elements of the FFT buffer
    int32_t wide;             // 16-byte runs in the epilogues as well (every run of the forcing 16-byte aligned)
    int32_t v16;              // stage with 16-byte copies (every staged segment 16-byte aligned)
    T rdz;
};

template <typename C>
__device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C>
__device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C>
__device__ __forceinline__ C cmul(C a, C b) { return C{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
template <typename C>
__device__ __forceinline__ C cmi(C a) { return C{a.y, -a.x}; }       // -i a

// Element e of a sequence sits at e + e/16 in shared memory: passes of stride 16 and
// more read 16 consecutive elements to a half-warp, and the middle pass, whose
// butterflies take R consecutive elements each, a different bank for each of them.
__device__ __forceinline__ int sk(int e) { return e + (e >> 4); }

// The passes of an N = 2^logn point transform: outer ones of radix 2^outer_log, each on
// the blocks that the ones before it left, then the middle one of radix 2^mid_log on
// consecutive elements, as large as maxlog allows (it does two DFTs on one trip through
// shared memory); as few outer ones as maxlog allows, as even as possible, and at least
// one (FP32, radix up to 16: 256 = 16 x 16, 512 = 8 x 4 x 16; FP64, whose values take
// twice the registers: up to 8).
__host__ __device__ constexpr int mid_log(int logn, int maxlog) { return logn <= maxlog ? logn - 1 : maxlog; }
__host__ __device__ constexpr int outer_log(int logn, int used, int maxlog)
{
    const int left = logn - mid_log(logn, maxlog) - used;
    const int passes = (left + maxlog - 1) / maxlog;
    return left <= 0 ? 0 : (left + passes - 1) / passes;
}
template <typename T>
constexpr int kMaxPassLog = sizeof(T) == 4 ? 4 : 3;

// R-point forward DFT in registers, natural order in and out:
// V[q] = sum_r v[r] exp(-2 pi i r q / R).
template <typename T, int R>
struct Dft;

template <typename T>
struct Dft<T, 1> {
    template <typename C>
    __device__ __forceinline__ static void run(C *)
    {
    }
};

template <typename T>
struct Dft<T, 2> {
    template <typename C>
    __device__ __forceinline__ static void run(C *v)
    {
        const C a = v[0];
        v[0] = cadd(a, v[1]);
        v[1] = csub(a, v[1]);
    }
};

template <typename T>
struct Dft<T, 4> {
    template <typename C>
    __device__ __forceinline__ static void run(C *v)
    {
        const C s0 = cadd(v[0], v[2]), d0 = csub(v[0], v[2]);
        const C s1 = cadd(v[1], v[3]), d1 = cmi(csub(v[1], v[3]));
        v[0] = cadd(s0, s1);
        v[2] = csub(s0, s1);
        v[1] = cadd(d0, d1);
        v[3] = csub(d0, d1);
    }
};

template <typename T>
struct Dft<T, 16> {
    // four 4-point DFTs over the stride-4 subsequences, the twiddles
    // exp(-2 pi i r2 q1 / 16), then four 4-point DFTs across them:
    // V[q1 + 4 q2] = sum_r2 w4^(r2 q2) w16^(r2 q1) sum_r1 v[4 r1 + r2] w4^(r1 q1)
    template <typename C>
    __device__ __forceinline__ static void run(C *v)
    {
        const T c = T(0.92387953251128675613), s = T(0.38268343236508977173), h = T(0.70710678118654752440);
        C a[4][4];
#pragma unroll
        for (int r2 = 0; r2 < 4; ++r2) {
            C x[4] = {v[r2], v[4 + r2], v[8 + r2], v[12 + r2]};
            Dft<T, 4>::run(x);
#pragma unroll
            for (int q1 = 0; q1 < 4; ++q1) a[r2][q1] = x[q1];
        }
        const C w1{c, -s}, w2{h, -h}, w3{s, -c}, w6{-h, -h}, w9{-c, s};
        a[1][1] = cmul(a[1][1], w1);
        a[1][2] = cmul(a[1][2], w2);
        a[1][3] = cmul(a[1][3], w3);
        a[2][1] = cmul(a[2][1], w2);
        a[2][2] = cmi(a[2][2]);                                       // w16^4 = -i
        a[2][3] = cmul(a[2][3], w6);
        a[3][1] = cmul(a[3][1], w3);
        a[3][2] = cmul(a[3][2], w6);
        a[3][3] = cmul(a[3][3], w9);
#pragma unroll
        for (int q1 = 0; q1 < 4; ++q1) {
            C y[4] = {a[0][q1], a[1][q1], a[2][q1], a[3][q1]};
            Dft<T, 4>::run(y);
#pragma unroll
            for (int q2 = 0; q2 < 4; ++q2) v[q1 + 4 * q2] = y[q2];
        }
    }
};

template <typename T>
struct Dft<T, 8> {
    // even / odd halves by two 4-point DFTs, joined with exp(-2 pi i q / 8)
    template <typename C>
    __device__ __forceinline__ static void run(C *v)
    {
        C e[4] = {v[0], v[2], v[4], v[6]};
        C o[4] = {v[1], v[3], v[5], v[7]};
        Dft<T, 4>::run(e);
        Dft<T, 4>::run(o);
        const T h = T(0.70710678118654752440);
        o[1] = C{h * (o[1].x + o[1].y), h * (o[1].y - o[1].x)};      // (1 - i)/sqrt 2
        o[2] = cmi(o[2]);                                             // -i
        o[3] = C{h * (o[3].y - o[3].x), -h * (o[3].x + o[3].y)};     // (-1 - i)/sqrt 2
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            v[q] = cadd(e[q], o[q]);
            v[q + 4] = csub(e[q], o[q]);
        }
    }
};

// One outer pass, in place, after passes of radices that multiply to 2^USED: on every
// block of M = N / 2^USED elements, butterfly j < M / R takes the elements j + r M / R.
// FORWARD: DFT, then the twiddles omega_M^(j q) on its outputs; the transposed pass:
// the same twiddles on its inputs, then the DFT.  The pass's twiddles are a table of
// its own, tw[(q - 1) M / R + j], so that a warp's loads of one q are contiguous.
// Every shared address is a base plus an immediate: M / R divides 16 or is a multiple
// of it, so sk(e + r M / R) = sk(e) + r M / R + (r M / R) / 16.
template <typename T, int LOGN, int USED, bool FORWARD>
__device__ __forceinline__ void outer_pass(typename Cx<T>::type *a, int S, int ld,
                                           const typename Cx<T>::type *__restrict__ tw)
{
    using C = typename Cx<T>::type;
    constexpr int LOGR = outer_log(LOGN, USED, kMaxPassLog<T>), R = 1 << LOGR;
    constexpr int LOGNB = LOGN - LOGR, LOGSTEP = LOGN - USED - LOGR, STEP = 1 << LOGSTEP;
    const int total = S << LOGNB;
    for (int t = threadIdx.x; t < total; t += kSpecThreads) {
        const int s = t >> LOGNB, jj = t & ((1 << LOGNB) - 1);
        const int j = jj & (STEP - 1), block = jj >> LOGSTEP;
        C *const at = a + s * ld + sk((block << (LOGN - USED)) + j);
        const C *const w = tw + j;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = at[r * STEP + ((r * STEP) >> 4)];
        if (!FORWARD) {
#pragma unroll
            for (int q = 1; q < R; ++q) v[q] = cmul(v[q], __ldg(w + (q - 1) * STEP));
        }
        Dft<T, R>::run(v);
        if (FORWARD) {
#pragma unroll
            for (int q = 1; q < R; ++q) v[q] = cmul(v[q], __ldg(w + (q - 1) * STEP));
        }
#pragma unroll
        for (int r = 0; r < R; ++r) at[r * STEP + ((r * STEP) >> 4)] = v[r];
    }
}

// The middle pass, in place: on R consecutive elements the forward transform's last
// DFT, the bins' i k / N and conjugation, v -> (-kn v.y, -kn v.x), and the first DFT
// of the second transform.  kn: in the order of the elements.
template <typename T, int LOGN>
__device__ __forceinline__ void mid_pass(typename Cx<T>::type *a, int S, int ld, const T *__restrict__ kn)
{
    using C = typename Cx<T>::type;
    constexpr int LOGR = mid_log(LOGN, kMaxPassLog<T>), R = 1 << LOGR, LOGNB = LOGN - LOGR;
    const int total = S << LOGNB;
    for (int t = threadIdx.x; t < total; t += kSpecThreads) {
        const int s = t >> LOGNB, e = (t & ((1 << LOGNB) - 1)) << LOGR;
        C *const at = a + s * ld + sk(e);
        const T *const k = kn + e;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = at[r];
        Dft<T, R>::run(v);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const T kr = __ldg(k + r);
            v[r] = C{-kr * v[r].y, -kr * v[r].x};
        }
        Dft<T, R>::run(v);
#pragma unroll
        for (int r = 0; r < R; ++r) at[r] = v[r];
    }
}

// The passes from the one after 2^USED on to the same one of the transposed network,
// with a block barrier after each.  tw points at the table of the pass after 2^USED.
template <typename T, int LOGN, int USED, bool MID>
struct Passes {
    using C = typename Cx<T>::type;
    __device__ __forceinline__ static void run(C *a, int S, int ld, const C *tw, const T *kn)
    {
        constexpr int LOGR = outer_log(LOGN, USED, kMaxPassLog<T>), NEXT = USED + LOGR;
        outer_pass<T, LOGN, USED, true>(a, S, ld, tw);
        __syncthreads();
        inner(a, S, ld, tw + (((1 << LOGR) - 1) << (LOGN - NEXT)), kn);
        outer_pass<T, LOGN, USED, false>(a, S, ld, tw);
        __syncthreads();
    }
    __device__ __forceinline__ static void inner(C *a, int S, int ld, const C *tw, const T *kn)
    {
        constexpr int NEXT = USED + outer_log(LOGN, USED, kMaxPassLog<T>);
        Passes<T, LOGN, NEXT, (NEXT + mid_log(LOGN, kMaxPassLog<T>) == LOGN)>::run(a, S, ld, tw, kn);
    }
};
template <typename T, int LOGN, int USED>
struct Passes<T, LOGN, USED, true> {
    using C = typename Cx<T>::type;
    __device__ __forceinline__ static void run(C *a, int S, int ld, const C *, const T *kn)
    {
        mid_pass<T, LOGN>(a, S, ld, kn);
        __syncthreads();
    }
};

// The first outer pass, read straight from the planar staging P (planes of n = L x N
// values): sequence s < L is plane0 + i plane1 of line s, sequence L + q is plane 2 of
// lines 2q and 2q + 1.  ROWS: the staging is [line][pos] and consecutive threads take
// consecutive butterflies of one sequence; otherwise it is [pos][line] and consecutive
// threads take consecutive sequences of one butterfly, so that both the staging reads
// and the skewed sequence writes stay spread over the banks.
template <typename T, int LOGN, bool ROWS>
__device__ __forceinline__ void first_pass(const T *__restrict__ P, typename Cx<T>::type *__restrict__ b, int logL,
                                           int ld, const typename Cx<T>::type *__restrict__ tw)
{
    using C = typename Cx<T>::type;
    constexpr int LOGR = outer_log(LOGN, 0, kMaxPassLog<T>);
    constexpr int R = 1 << LOGR;
    constexpr int LOGNB = LOGN - LOGR;
    constexpr int NB = 1 << LOGNB;
    const int L = 1 << logL;
    const int S = L + L / 2;
    const int n = L << LOGN;
    const int total = S << LOGNB;
    for (int t = threadIdx.x; t < total; t += kSpecThreads) {
        int s, j;
        if (ROWS) {
            s = t >> LOGNB;
            j = t & (NB - 1);
        } else if (t < L << LOGNB) {            // the line sequences, then the plane-2 ones
            j = t >> logL;
            s = t & (L - 1);
        } else {
            const int u = t - (L << LOGNB);
            j = u >> (logL - 1);
            s = L + (u & (L / 2 - 1));
        }
        C v[R];
        if (s < L) {
            const T *p0 = ROWS ? P + (s << LOGN) + j : P + (j << logL) + s;
            const int step = ROWS ? NB : NB << logL;
#pragma unroll
            for (int r = 0; r < R; ++r) v[r] = C{p0[r * step], p0[n + r * step]};
        } else {
            const int l0 = 2 * (s - L);
            if (ROWS) {
                const T *p0 = P + 2 * n + (l0 << LOGN) + j;
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = C{p0[r * NB], p0[(1 << LOGN) + r * NB]};
            } else {
                const C *p0 = reinterpret_cast<const C *>(P + 2 * n + (j << logL) + l0);
                const int step = (NB << logL) / 2;      // complex elements between r and r + 1
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = p0[r * step];
            }
        }
        Dft<T, R>::run(v);
        const C *const w = tw + j;
#pragma unroll
        for (int q = 1; q < R; ++q) v[q] = cmul(v[q], __ldg(w + (q - 1) * NB));
        C *const out = b + s * ld + sk(j);
#pragma unroll
        for (int q = 0; q < R; ++q) out[q * NB + ((q * NB) >> 4)] = v[q];
    }
}

template <typename T, bool ROWS, int LOGN, typename Next>
__device__ __forceinline__ void derive_n(const T *P, typename Cx<T>::type *A, int logL, int ld,
                                         const typename Cx<T>::type *tw, const T *kn, Next next)
{
    const int S = (1 << logL) + (1 << logL) / 2;
    first_pass<T, LOGN, ROWS>(P, A, logL, ld, tw);
    __syncthreads();
    next();
    Passes<T, LOGN, 0, false>::inner(A, S, ld, tw + (((1 << outer_log(LOGN, 0, kMaxPassLog<T>)) - 1)
                                                    << (LOGN - outer_log(LOGN, 0, kMaxPassLog<T>))), kn);
    outer_pass<T, LOGN, 0, false>(A, S, ld, tw);
    __syncthreads();
}

// Spectral derivative of the staged lines: z = plane0 + i plane1 (and the plane-2
// pairs), conj(FFT(conj(i k/N * FFT(z)))), for N = 2^logN, 2 <= N <= 2048.  The
// first pass reads the planar staging P, then next() runs (P is free); A then holds
// (D a, -D b) for each z = a + i b.
template <typename T, bool ROWS, typename Next>
__device__ __forceinline__ void derive(const T *P, typename Cx<T>::type *A, int logL, int logN, int ld,
                                       const typename Cx<T>::type *tw, const T *kn, Next next)
{
    switch (logN) {
    case 1: return derive_n<T, ROWS, 1>(P, A, logL, ld, tw, kn, next);
    case 2: return derive_n<T, ROWS, 2>(P, A, logL, ld, tw, kn, next);
    case 3: return derive_n<T, ROWS, 3>(P, A, logL, ld, tw, kn, next);
    case 4: return derive_n<T, ROWS, 4>(P, A, logL, ld, tw, kn, next);
    case 5: return derive_n<T, ROWS, 5>(P, A, logL, ld, tw, kn, next);
    case 6: return derive_n<T, ROWS, 6>(P, A, logL, ld, tw, kn, next);
    case 7: return derive_n<T, ROWS, 7>(P, A, logL, ld, tw, kn, next);
    case 8: return derive_n<T, ROWS, 8>(P, A, logL, ld, tw, kn, next);
    case 9: return derive_n<T, ROWS, 9>(P, A, logL, ld, tw, kn, next);
    case 10: return derive_n<T, ROWS, 10>(P, A, logL, ld, tw, kn, next);
    default: return derive_n<T, ROWS, 11>(P, A, logL, ld, tw, kn, next);
    }
}

// Asynchronous global -> shared copies (cp.async; completion by commit groups).
template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst, const void *src)
{
    if (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)), "l"(src), "n"(BYTES)
                     : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Issues the copies of a unit's input lines into the planar staging buffer P:
// three planes of n = lines x line-length values (row unit: txx, txy, txz rows
// j0 .. j0 + rx - 1; column unit: txy, tyy, tyz as [ny][wy] strips), then
// commits the group (an empty group when the unit needs no input).
template <typename T, int VB>
__device__ __forceinline__ void stage_copies(const SpecParams<T> &p, T *P, int kind, int level, int idx)
{
    constexpr int kLogV = VB == (int)sizeof(T) ? 0 : (VB == 2 * (int)sizeof(T) ? 1 : 2);   // log2 of the values per copy
    if (kind == 0 && level < p.nz - 1) {
        const int logn = p.logrx + p.lognx, logper = logn - kLogV;      // every count is a power of two
        const int base = level * p.nx * p.ny + (idx << logn);
        for (int c = threadIdx.x; c < 3 << logper; c += kSpecThreads) {
            const int f = c >> logper, q = (c & ((1 << logper) - 1)) << kLogV;
            const T *src = f == 0 ? p.txx : (f == 1 ? p.txy : p.txz);
            cp_async<VB>(P + (f << logn) + q, src + base + q);
        }
    } else if (kind == 1 && level < p.nz - 1) {
        const int logn = p.logny + p.logwy, logper = logn - kLogV;
        const int base = level * p.nx * p.ny + (idx << p.logwy);
        for (int c = threadIdx.x; c < 3 << logper; c += kSpecThreads) {
            const int f = c >> logper, q = (c & ((1 << logper) - 1)) << kLogV;
            const int j = q >> p.logwy, cc = q & ((1 << p.logwy) - 1);
            const T *src = f == 0 ? p.txy : (f == 1 ? p.tyy : p.tyz);
            cp_async<VB>(P + (f << logn) + q, src + base + (j << p.lognx) + cc);
        }
    }
}

// Bulk prefetch of `bytes` (a multiple of 16, 16-byte aligned) into L2.
__device__ __forceinline__ void prefetch_l2(const void *src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

template <typename T>
__device__ void stage_unit(const SpecParams<T> &p, T *P, int kind, int level, int idx)
{
    if (p.v16) stage_copies<T, 16>(p, P, kind, level, idx);
    else stage_copies<T, (int)sizeof(T)>(p, P, kind, level, idx);
    cp_async_commit();
    // a row unit's epilogue reads the vertical terms of its rows (tzz at k and
    // k - 1, txz and tyz at k + 1, tyz at k), which no unit has staged yet: start
    // them towards L2 now, a unit ahead, so that the epilogue waits on L2, not DRAM
    if (kind == 0 && p.v16 && level < p.nz - 1 && threadIdx.x == 0) {
        const int64_t plane = (int64_t)p.nx * p.ny;
        const int64_t base = (int64_t)level * plane + ((int64_t)idx << (p.logrx + p.lognx));
        const uint32_t bytes = (uint32_t)(sizeof(T) << (p.logrx + p.lognx));
        prefetch_l2(p.tzz + base, bytes);
        if (level > 0) prefetch_l2(p.tzz + base - plane, bytes);
        prefetch_l2(p.tyz + base, bytes);
        prefetch_l2(p.txz + base + plane, bytes);
        prefetch_l2(p.tyz + base + plane, bytes);
    }
}

// V consecutive values of a global array (V > 1: 16-byte aligned); L2: past L1.
template <typename T, int V>
struct Run {
    T v[V];
};
template <bool L2, typename T>
__device__ __forceinline__ T ld(const T *p) { return L2 ? __ldcg(p) : __ldg(p); }
template <int V, bool L2, typename T>
__device__ __forceinline__ Run<T, V> ld_run(const T *p)
{
    Run<T, V> r;
    if constexpr (V == 4) {
        const float4 a = ld<L2>(reinterpret_cast<const float4 *>(p));
        r.v[0] = a.x; r.v[1] = a.y; r.v[2] = a.z; r.v[3] = a.w;
    } else if constexpr (V == 2) {
        const double2 a = ld<L2>(reinterpret_cast<const double2 *>(p));
        r.v[0] = a.x; r.v[1] = a.y;
    } else {
        r.v[0] = ld<L2>(p);
    }
    return r;
}
template <int V, typename T>
__device__ __forceinline__ void st_run(T *p, const Run<T, V> &r)
{
    if constexpr (V == 4) *reinterpret_cast<float4 *>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
    else if constexpr (V == 2) *reinterpret_cast<double2 *>(p) = make_double2(r.v[0], r.v[1]);
    else *p = r.v[0];
}

// The row unit's forcing from its derivatives R and the vertical terms.
template <typename T, int V>
__device__ __forceinline__ void row_forcing(const SpecParams<T> &p, const typename Cx<T>::type *R, int k, int base)
{
    using C = typename Cx<T>::type;
    const int rx = 1 << p.logrx, n = rx << p.lognx, plane = p.nx * p.ny, ld = p.ldx;
#pragma unroll 2
    for (int e = threadIdx.x * V; e < n; e += kSpecThreads * V) {
        const int r = e >> p.lognx, i = e & (p.nx - 1), o = base + e;
        const Run<T, V> xz0 = ld_run<V, false>(p.txz + o), xz1 = ld_run<V, false>(p.txz + o + plane);
        const Run<T, V> yz0 = ld_run<V, false>(p.tyz + o), yz1 = ld_run<V, false>(p.tyz + o + plane);
        const Run<T, V> zz0 = ld_run<V, false>(p.tzz + o);
        Run<T, V> zzm = zz0, fx, fy, fz;
        if (k > 0) zzm = ld_run<V, false>(p.tzz + o - plane);
        // V divides 16: the skew is the same for all of a run
        const C *const d = R + r * ld + sk(i), *const dd = R + (rx + (r >> 1)) * ld + sk(i);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const C a = d[q], b = dd[q];                        // (d_x txx, -d_x txy), d_x txz of two rows
            const T dxz = (r & 1) ? -b.y : b.x;
            fx.v[q] = -(a.x + (xz1.v[q] - xz0.v[q]) * p.rdz);
            fy.v[q] = -(-a.y + (yz1.v[q] - yz0.v[q]) * p.rdz);
            fz.v[q] = (k == 0) ? T(0) : -(dxz + (zz0.v[q] - zzm.v[q]) * p.rdz);
        }
        st_run(p.fx + o, fx);
        st_run(p.fy + o, fy);
        st_run(p.fz + o, fz);
    }
}

// Row unit on level k, rows j0 .. j0 + rx - 1, whose input lines are staged in
// P: d_x of txx, txy (sequences s < rx) and txz (rows 2q, 2q + 1 in rx + q),
// plus the vertical terms -> the partial forcing in f.
template <typename T, typename Next>
__device__ void row_unit(const SpecParams<T> &p, const T *P, typename Cx<T>::type *A, int k, int j0, Next next)
{
    const int n = 1 << (p.logrx + p.lognx), base = k * p.nx * p.ny + j0 * p.nx;
    if (k == p.nz - 1) {                    // ghost uv level / lid: f = 0
        next();
        for (int e = threadIdx.x; e < n; e += kSpecThreads) {
            p.fx[base + e] = T(0);
            p.fy[base + e] = T(0);
            p.fz[base + e] = T(0);
        }
        return;
    }
    derive<T, true>(P, A, p.logrx, p.lognx, p.ldx, p.twx, p.knx, next);
    if (p.wide) row_forcing<T, 16 / (int)sizeof(T)>(p, A, k, base);
    else row_forcing<T, 1>(p, A, k, base);
}

// Waits until *ctr >= target (acquire, GPU scope); bounded by kWaitLimitNs.
__device__ bool wait_level(const unsigned int *ctr, unsigned int target, int *status)
{
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
    if (v >= target) return true;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 1;; ++it) {
        __nanosleep(128);
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
        if (v >= target) return true;
        if ((it & 7u) == 0) {
            if (*(volatile int *)status != 0) return false;
            if (global_timer_ns() - t0 > kWaitLimitNs) {
                atomicExch(status, kDevStatusBarrierTimeout);
                return false;
            }
        }
    }
}

// Subtracts the column unit's derivatives R from the partial forcing.
template <typename T, int V>
__device__ __forceinline__ void column_forcing(const SpecParams<T> &p, const typename Cx<T>::type *R, int k, int base)
{
    using C = typename Cx<T>::type;
    const int wy = 1 << p.logwy, n = wy << p.logny, ld = p.ldy;
#pragma unroll 2
    for (int e = threadIdx.x * V; e < n; e += kSpecThreads * V) {
        const int j = e >> p.logwy, c = e & (wy - 1), o = base + (j << p.lognx) + c;
        Run<T, V> fx = ld_run<V, true>(p.fx + o), fy = ld_run<V, true>(p.fy + o), fz = ld_run<V, true>(p.fz + o);
#pragma unroll
        for (int q = 0; q < V; ++q) {
            const C d = R[(c + q) * ld + sk(j)];                // (d_y txy, -d_y tyy)
            const C dd = R[(wy + ((c + q) >> 1)) * ld + sk(j)];
            const T dyz = ((c + q) & 1) ? -dd.y : dd.x;         // d_y tyz
            fx.v[q] -= d.x;
            fy.v[q] += d.y;
            fz.v[q] -= dyz;
        }
        st_run(p.fx + o, fx);
        st_run(p.fy + o, fy);
        if (k > 0) st_run(p.fz + o, fz);
    }
}

// Column unit on level k, columns i0 .. i0 + wy - 1, staged in P: d_y of txy, tyy
// (sequences c < wy) and tyz (columns 2q, 2q + 1 in wy + q), subtracted from f
// once every row unit of level k has written its partial forcing.
template <typename T, typename Next>
__device__ void column_unit(const SpecParams<T> &p, const T *P, typename Cx<T>::type *A, int k, int i0, int *s_go,
                            Next next)
{
    using C = typename Cx<T>::type;
    if (k == p.nz - 1) {                    // f stays 0 there (written by the row units)
        next();
        return;
    }
    const int base = k * p.nx * p.ny + i0;
    derive<T, false>(P, A, p.logwy, p.logny, p.ldy, p.twy, p.kny, next);
    if (threadIdx.x == 0) *s_go = wait_level(p.ctr + 2 + k, (unsigned)p.xpl, p.status) ? 1 : 0;
    __syncthreads();
    if (!*s_go) return;                     // gave up waiting: skipped, the status says so
    if (p.wide) column_forcing<T, 16 / (int)sizeof(T)>(p, A, k, base);
    else column_forcing<T, 1>(p, A, k, base);
}

// Unit u of the dispense order -> kind (0 row, 1 column), level, index within the level.
// Phase ph (0 .. nchunks): row units of chunk ph, then column units of chunk ph - 1.
template <typename T>
__device__ void decode_unit(const SpecParams<T> &p, int64_t u, int *kind, int *level, int *idx)
{
    auto start = [&](int ph) -> int64_t {
        const int64_t a = min((int64_t)ph * p.kc, (int64_t)p.nz);
        const int64_t b = min((int64_t)max(ph - 1, 0) * p.kc, (int64_t)p.nz);
        return a * p.xpl + b * p.ypl;
    };
    int lo = 0, hi = p.nchunks;             // largest ph with start(ph) <= u
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (start(mid) <= u) lo = mid;
        else hi = mid - 1;
    }
    int64_t o = u - start(lo);
    const int64_t nrow = lo < p.nchunks ? (min((int64_t)(lo + 1) * p.kc, (int64_t)p.nz) - (int64_t)lo * p.kc) * p.xpl
                                        : 0;
    if (o < nrow) {
        *kind = 0;
        *level = lo * p.kc + (int)(o / p.xpl);
        *idx = (int)(o % p.xpl);
    } else {
        o -= nrow;
        *kind = 1;
        *level = (lo - 1) * p.kc + (int)(o / p.ypl);
        *idx = (int)(o % p.ypl);
    }
}

template <typename T>
__device__ __forceinline__ void claim(const SpecParams<T> &p, int *slot)
{
    const int64_t u = (int64_t)atomicAdd(p.ctr, 1u);
    int kind = -1, level = 0, idx = 0;
    if (u < p.total) decode_unit(p, u, &kind, &level, &idx);
    slot[0] = kind;
    slot[1] = level;
    slot[2] = idx;
}

// Bound, FP32: shared-memory accesses, issue and the barriers between passes (hill
// 512 x 256 x 256: 722 us against 178 us for its bytes at the copy peak; 256 x 128 x
// 128 77 us, 64^3 14.7 us); a Stockham pair of transforms with two more buffers, three
// blocks of 256 threads per SM, took 765, 93 and 17 us.  FP64: the FP64 pipe, about 150
// operations a point, 1.09 ms of 1.20 ms on 256 x 128 x 128.  192 threads divide the
// passes of the common tiles evenly (six sequences of 512 points are 192 butterflies
// of radix 16): four blocks of 192 per SM 742 us, of 256 788, three of 256 779, five of
// 192 820, eight of 96 1070 (before the 16-byte epilogues).  FP64: radix 16 or three
// blocks per SM 1211 and 1231 us against 1202.
//
// Persistent loop: each block holds the unit it works on and the next one, whose
// input lines stream into the staging buffer as soon as the unit's first pass has
// read its own from there.  A column unit waits only for the row units of its level,
// which hold smaller tickets; the unfinished unit with the smallest ticket can
// always proceed, so the loop ends.  Shared memory: the FFT buffer A and the staging
// buffer P (a second one would leave the tables and the epilogue's loads a few KB of
// L1).
template <typename T>
__global__ void __launch_bounds__(kSpecThreads, sizeof(T) == 4 ? 4 : 2) k_spectral(SpecParams<T> p)
{
    using C = typename Cx<T>::type;
    extern __shared__ __align__(16) unsigned char spec_smem[];
    C *A = reinterpret_cast<C *>(spec_smem);
    T *const P = reinterpret_cast<T *>(A + p.buf);
    __shared__ int s_u[2][3];
    __shared__ int s_go, s_last;
    int cur = 0;
    if (threadIdx.x == 0) claim(p, s_u[0]);
    __syncthreads();
    stage_unit<T>(p, P, s_u[0][0], s_u[0][1], s_u[0][2]);
    for (;;) {
        const int kind = s_u[cur][0], level = s_u[cur][1], idx = s_u[cur][2];
        if (kind < 0) break;
        if (threadIdx.x == 0) claim(p, s_u[cur ^ 1]);
        cp_async_wait<0>();                 // this unit's lines have landed
        __syncthreads();
        auto next = [&] { stage_unit<T>(p, P, s_u[cur ^ 1][0], s_u[cur ^ 1][1], s_u[cur ^ 1][2]); };
        if (kind == 0) {
            row_unit<T>(p, P, A, level, idx << p.logrx, next);
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                atomicAdd(p.ctr + 2 + level, 1u);
            }
        } else {
            column_unit<T>(p, P, A, level, idx << p.logwy, &s_go, next);
            __syncthreads();
        }
        cur ^= 1;
    }
    cp_async_wait<0>();
    // the last block out re-arms the counters for the next launch: every block
    // has taken its final ticket and passed its waits by then
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = (atomicAdd(p.ctr + 1, 1u) == gridDim.x - 1) ? 1 : 0;
    }
    __syncthreads();
    if (s_last) {
        for (int k = threadIdx.x; k < p.nz; k += kSpecThreads) p.ctr[2 + k] = 0u;
        if (threadIdx.x == 0) p.ctr[0] = 0u;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            p.ctr[1] = 0u;
        }
    }
}

int ilog2_exact(int n)
{
    if (n < 1 || (n & (n - 1))) return -1;
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

template <typename T>
int upload_tables(wmibm_handle *h, SpecState *s, cudaStream_t stream)
{
    using C = typename Cx<T>::type;
    const int n[2] = {h->nx, h->ny};
    const double len[2] = {h->lx, h->ly};
    void **tw[2] = {&s->twx, &s->twy};
    void **kn[2] = {&s->knx, &s->kny};
    for (int d = 0; d < 2; ++d) {
        const int N = n[d];
        C *ht = (C *)host_alloc(sizeof(C) * N);
        T *hk = (T *)host_alloc(sizeof(T) * N);
        if (!ht || !hk) {
            free(ht);
            free(hk);
            return set_error(nullptr, WMIBM_ENOMEM, "host memory for the spectral tables");
        }
        // twiddles of the outer passes: on blocks of M elements, omega_M^(j q) at (q - 1) M / R + j
        const int logN = ilog2_exact(N), maxlog = kMaxPassLog<T>;
        int at = 0, used = 0;
        for (int logR; (logR = outer_log(logN, used, maxlog)) > 0; used += logR) {
            const int M = N >> used, R = 1 << logR, step = M / R;
            for (int q = 1; q < R; ++q)
                for (int j = 0; j < step; ++j) {
                    const double a = 2.0 * M_PI * (double)j * (double)q / (double)M;
                    ht[at].x = (T)cos(a);
                    ht[at].y = (T)(-sin(a));
                    ++at;
                }
        }
        for (int e = 0; e < N; ++e) {
            // the bin that the forward transform leaves at element e: the passes' digits of e, the first one's
            // (the most significant) counting least
            int m = 0, left = e, size = N, weight = 1;
            for (int u = 0; size > 1;) {
                int logR = outer_log(logN, u, maxlog);
                if (logR == 0) logR = ilog2_exact(size);    // the middle pass
                const int R = 1 << logR, step = size / R;
                m += weight * (left / step);
                left %= step;
                weight *= R;
                size = step;
                u += logR;
            }
            // its wavenumber: m below N/2, m - N above, 0 for the Nyquist bin
            const int mm = (2 * m < N) ? m : (2 * m == N ? 0 : m - N);
            hk[e] = (T)(2.0 * M_PI * (double)mm / len[d] / (double)N);
        }
        cudaError_t e = dev_alloc(tw[d], sizeof(C) * N);
        if (e == cudaSuccess) e = dev_alloc(kn[d], sizeof(T) * N);
        if (e == cudaSuccess) e = cudaMemcpyAsync(*tw[d], ht, sizeof(C) * N, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(*kn[d], hk, sizeof(T) * N, cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        free(ht);
        free(hk);
        if (e != cudaSuccess) return cuda_status(nullptr, e, "spectral tables");
    }
    return WMIBM_OK;
}

template <typename T>
int run_spectral(wmibm_handle *h, const SpecParams<T> &p, const SpecState *s, cudaStream_t stream)
{
    cudaError_t e = cudaFuncSetAttribute(k_spectral<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSpecSmemMax);
    if (e != cudaSuccess) return cuda_status(h, e, "k_spectral shared memory");
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_spectral<T>, kSpecThreads, s->smem);
    if (e != cudaSuccess) return cuda_status(h, e, "k_spectral occupancy");
    if (per_sm < 1) return set_error(h, WMIBM_EINVAL, "spectral units do not fit on an SM");
    int64_t grid = (int64_t)per_sm * h->sm_count;
    if (grid > s->total) grid = s->total;
    k_spectral<T><<<(unsigned)grid, kSpecThreads, s->smem, stream>>>(p);
    return cuda_status(h, cudaGetLastError(), "k_spectral launch");
}

template <typename T>
int launch_spectral(wmibm_handle *h, const void *const tau[6], void *fx, void *fy, void *fz, cudaStream_t stream)
{
    const SpecState *s = h->spec;
    SpecParams<T> p;
    p.txx = (const T *)tau[0]; p.txy = (const T *)tau[1]; p.tyy = (const T *)tau[2];
    p.tzz = (const T *)tau[3]; p.txz = (const T *)tau[4]; p.tyz = (const T *)tau[5];
    p.fx = (T *)fx; p.fy = (T *)fy; p.fz = (T *)fz;
    p.twx = (const typename Cx<T>::type *)s->twx;
    p.twy = (const typename Cx<T>::type *)s->twy;
    p.knx = (const T *)s->knx;
    p.kny = (const T *)s->kny;
    p.ctr = s->ctr;
    p.status = h->dev_status;
    p.nx = h->nx; p.ny = h->ny; p.nz = h->nz;
    p.lognx = s->lognx; p.logny = s->logny;
    p.logrx = ilog2_exact(s->rx); p.logwy = ilog2_exact(s->wy);
    p.ldx = s->ldx; p.ldy = s->ldy;
    p.kc = s->kc; p.nchunks = s->nchunks; p.xpl = s->xpl; p.ypl = s->ypl;
    p.total = s->total;
    p.buf = (int)s->buf;
    p.rdz = (T)(1.0 / h->dz);
    // 16-byte copies when every staged line segment starts on a 16-byte boundary
    bool v16 = (h->nx * sizeof(T)) % 16 == 0 && (s->wy * sizeof(T)) % 16 == 0;
    for (int c = 0; c < 6; ++c) v16 = v16 && ((uintptr_t)tau[c] & 15u) == 0;
    p.v16 = v16 ? 1 : 0;
    for (const void *q : {fx, fy, fz}) v16 = v16 && ((uintptr_t)q & 15u) == 0;
    p.wide = v16 ? 1 : 0;
    return run_spectral<T>(h, p, s, stream);
}

}  // namespace

namespace wmibm {

// Called once by wmibm_init: tables, counters and tile shapes of the spectral
// forcing when nx and ny are powers of two in [2, 2048] (FP32) or [2, 1024] (FP64);
// otherwise the handle has no spectral state and wmibm_force_spectral returns
// WMIBM_EINVAL.
// Errors go to the thread's last error (the handle is not returned on failure).
int spectral_setup(wmibm_handle *h, cudaStream_t stream)
{
    h->spec = nullptr;
    const int lx = ilog2_exact(h->nx), ly = ilog2_exact(h->ny);
    const int maxlog = h->dtype == WMIBM_F64 ? kSpecMaxLog - 1 : kSpecMaxLog;
    if (lx < 1 || ly < 1 || lx > maxlog || ly > maxlog) return WMIBM_OK;
    SpecState *s = (SpecState *)host_alloc(sizeof(SpecState));
    if (!s) return set_error(nullptr, WMIBM_ENOMEM, "host memory for the spectral state");
    h->spec = s;
    s->lognx = lx;
    s->logny = ly;
    const bool f64 = h->dtype == WMIBM_F64;
    const size_t cs = f64 ? 16 : 8;
    const int budget = f64 ? kSpecBudget / 2 : kSpecBudget;
    // rows per row unit: even power of two dividing ny, 1.5 rx (nx + 1) within the budget
    s->ldx = h->nx + (h->nx >> 4) + 1;       // skewed sequence (e + e/16) plus one: odd-ish bank offset
    s->rx = 2;
    while (s->rx * 2 <= h->ny && 3 * (s->rx * 2) / 2 * s->ldx <= budget) s->rx *= 2;
    s->ldy = h->ny + (h->ny >> 4) + 1;
    s->wy = 2;
    // FP32: at least a 32-byte sector of columns where shared memory has the room, whatever
    // that leaves of the blocks per SM (columns of 512 points, 4 / 8 of them: 1024 x 512 x 18
    // 332 / 292 us, 512 x 512 x 64 566 / 515; of 1024, 2 / 4 / 8: 512 x 1024 x 20 659 / 451 / 441)
    auto room = [&](int wy) { return !f64 && wy <= 8 && (12 * (size_t)s->ldy + 12 * (size_t)h->ny) * wy <= 220 * 1024; };
    while (s->wy * 2 <= h->nx && (3 * (s->wy * 2) / 2 * s->ldy <= budget || room(s->wy * 2))) s->wy *= 2;
    const int64_t ex = (int64_t)3 * s->rx / 2 * s->ldx, ey = (int64_t)3 * s->wy / 2 * s->ldy;
    s->buf = ((ex > ey ? ex : ey) + 1) & ~(int64_t)1;               // even: 16-byte aligned buffers
    const int64_t px = (int64_t)3 * s->rx * h->nx, py = (int64_t)3 * s->wy * h->ny;
    s->smem = cs * (size_t)s->buf + (cs / 2) * (size_t)(px > py ? px : py);
    s->xpl = h->ny / s->rx;
    s->ypl = h->nx / s->wy;
    const double level_bytes = 9.0 * (double)h->nx * (double)h->ny * (double)elem_size(h->dtype);
    s->kc = (int)(kSpecChunkBytes / level_bytes);
    const int resident = h->sm_count * std::min<int>(f64 ? 2 : 4, (int)(227 * 1024 / (s->smem + 1024)));
    // and at least half the resident blocks' number of row units a chunk: the column units of
    // a shorter one wait (1024 x 512 x 18 with chunks of one and two levels 378 and 335 us,
    // 512 x 512 x 64 of two and three 638 and 569)
    s->kc = std::max(s->kc, (resident / 2 + s->xpl - 1) / s->xpl);
    if (s->kc > h->nz) s->kc = h->nz;
    s->nchunks = (h->nz + s->kc - 1) / s->kc;
    s->total = (int64_t)h->nz * (s->xpl + s->ypl);
    int st = f64 ? upload_tables<double>(h, s, stream) : upload_tables<float>(h, s, stream);
    if (st) return st;
    cudaError_t e = dev_alloc(&s->ctr, sizeof(unsigned int) * (size_t)(h->nz + 2));
    if (e == cudaSuccess) e = cudaMemsetAsync(s->ctr, 0, sizeof(unsigned int) * (size_t)(h->nz + 2), stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_status(nullptr, e, "spectral counters");
    return WMIBM_OK;
}

void spectral_free(wmibm_handle *h)
{
    SpecState *s = h ? h->spec : nullptr;
    if (!s) return;
    if (s->twx) cudaFree(s->twx);
    if (s->twy) cudaFree(s->twy);
    if (s->knx) cudaFree(s->knx);
    if (s->kny) cudaFree(s->kny);
    if (s->ctr) cudaFree(s->ctr);
    free(s);
    h->spec = nullptr;
}

// Shape of the spectral launch, for the bench and the tests: [rows per row unit,
// columns per column unit, levels per chunk, shared bytes per block].
int spectral_shape(const wmibm_handle *h, int64_t out[4])
{
    const SpecState *s = h->spec;
    if (!s) return WMIBM_EINVAL;
    out[0] = s->rx;
    out[1] = s->wy;
    out[2] = s->kc;
    out[3] = (int64_t)s->smem;
    return WMIBM_OK;
}

}  // namespace wmibm

extern "C" int wmibm_force_spectral(wmibm_handle *h, const void *const tau[6], void *fx, void *fy, void *fz,
                                    void *stream)
{
    ApiRange nvtx_range("wmibm_force_spectral");
    if (!h) return set_error(nullptr, WMIBM_EINVAL, "NULL handle");
    if (!tau || !fx || !fy || !fz) return set_error(h, WMIBM_EINVAL, "NULL stress or force pointer");
    for (int c = 0; c < 6; ++c)
        if (!tau[c]) return set_error(h, WMIBM_EINVAL, "NULL stress pointer %d", c);
    if (!h->spec)
        return set_error(h, WMIBM_EINVAL, "spectral derivatives need nx and ny powers of two in [2, %d] (got %d x %d)",
                         h->dtype == WMIBM_F64 ? 1 << (kSpecMaxLog - 1) : 1 << kSpecMaxLog, h->nx, h->ny);
    int st = check_device(h);
    if (st) return st;
    if (h->dtype == WMIBM_F64) return launch_spectral<double>(h, tau, fx, fy, fz, (cudaStream_t)stream);
    return launch_spectral<float>(h, tau, fx, fy, fz, (cudaStream_t)stream);
}

extern "C" int wmibm_spectral_shape(const wmibm_handle *h, int64_t out[4])
{
    if (!h || !out) return WMIBM_EINVAL;
    return wmibm::spectral_shape(h, out);
}
