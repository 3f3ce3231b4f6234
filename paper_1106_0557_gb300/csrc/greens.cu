// greens.cu -- the transform of the doubled-mesh Green's function (Eq. 9),
// built once per (doubled mesh, width ratios) in FP64 on the device.
//
// The Eq. 9 table is real and even in every axis (its inactive regions are
// mirror images), so its DFT is real and even too and is separable over the
// even octant 0 <= p <= Mx/2, 0 <= q <= My/2, 0 <= r <= Mz/2:
//   Gt(kx,ky,kz) = sum w_p w_q w_r G(p,q,r) cos(2 pi kx p/Mx) cos(2 pi ky q/My)
//                  cos(2 pi kz r/Mz),   w = 1 at 0 and M/2, 2 otherwise.
// Each axis's cosine sum is the M-point DFT of the octant line mirrored to
// its full length (c[p] = G[min(p, M - p)]), whose bins 0..M/2 are real.
// One pass per axis transforms every octant line that way in place, with
// the FFT engine of the solve passes in FP64 (O(M^3 log M) in all); FP64 is
// what sets the accuracy floor of the solve.
//
// A spectrum that is stored in FP32 rounds each bin to 24 bits, so its build
// takes two cheaper FP64 forms (PAIRS below: inv_sqrt, and two lines per
// transform).  FP64 and float-pair spectra keep every bit they can: with the
// cheaper forms FP64 potentials lay further from 80-bit ones, by 3 to 6 % on
// random sources (at most 1.42 times) and up to 9 times on sources that
// alternate from cell to cell (36^3 2.7e-15 -> 2.5e-14; allocation-free 4.5e-15
// -> 8.5e-14), float pairs up to 5 times; FP32 ones did not move.
#include <math.h>
#include <stdio.h>

#include <type_traits>
#include <vector>

#include "inv_sqrt.cuh"
#include "launch.h"
#include "passes.cuh"

namespace isofft {

// A thread takes one (x, y) and `zc` planes; block row blockIdx.y.  Bound by
// FP64 arithmetic: the quotient by the square root with 64-bit indices took
// 22.9 us on a 65^3 octant, PAIRS 16.8 us (0.82 -> 0.52 ms at 257^3).
template <bool PAIRS>
static __global__ void k_green_octant(double *__restrict__ g, int X, int Y, int Z, double hx, double hy,
                                      double hz, int zc)
{
    grid_wait();
    const int xy = blockIdx.x * blockDim.x + threadIdx.x;
    if (xy >= X * Y) return;
    const int y = xy / X, x = xy - y * X;
    const double num = -hx * hy * hz / (4.0 * 3.14159265358979323846);
    const double hmin = fmin(hx, fmin(hy, hz));
    const double dx = hx * (double)x, dy = hy * (double)y;
    const int z1 = min((int)(blockIdx.y + 1) * zc, Z);
    for (int z = blockIdx.y * zc; z < z1; ++z) {
        const double dz = hz * (double)z;
        // Eq. 6; at the origin Eq. 9: the largest off-origin magnitude
        double v;
        if (xy == 0 && z == 0) {
            v = num / hmin;
        } else {
            if constexpr (PAIRS)
                v = num * inv_sqrt(fma(dz, dz, fma(dx, dx, dy * dy)));
            else
                v = num / sqrt(dx * dx + dy * dy + dz * dz);
        }
        g[(int64_t)z * X * Y + xy] = v;
    }
}

// One axis of the octant transform, in place: line (a, c) of the octant,
// elements base[q Cc] (q <= L/2, base = oct + a (L/2 + 1) Cc + c), is
// mirrored to L points, transformed, and bins 0..L/2 (real) are written back.
// PAIRS (FP32 spectra): the transform of a real even line is real, so two
// neighbouring lines go through one complex transform as its real and
// imaginary parts: the pass is bound by FP64 arithmetic, and this halves it
// (22.2 -> 15.2 us an axis at 65^3, 1.40 -> 0.82 ms at 257^3).  Each line's
// rounding is then relative to the larger of the two.
// Lines (or pairs) are grouped NL per CTA (one row buffer each, as the x passes use).
template <int L>
struct DctCfg {
    using SH = Shape<double, L>;
    static constexpr int E = SH::E, NT = L / E;
    static constexpr int NL = NT >= 128 ? 1 : 128 / NT;
    static constexpr int THREADS = NL * NT;
    static constexpr size_t SMEM = (size_t)NL * RowPad<double, L>::LP * sizeof(Cx<double>);
};

template <int L, bool PAIRS>
static __global__ void __launch_bounds__(DctCfg<L>::THREADS)
k_cos_lines(double *__restrict__ oct, const Cx<double> *__restrict__ tw, int64_t A, int64_t Cc)
{
    using C = DctCfg<L>;
    constexpr int E = C::E, NT = C::NT, n = L / 2 + 1;
    extern __shared__ __align__(16) unsigned char dct_smem[];
    Cx<double> *row = reinterpret_cast<Cx<double> *>(dct_smem) + (threadIdx.x / NT) * RowPad<double, L>::LP;
    const int l = threadIdx.x / NT, t = threadIdx.x % NT;
    constexpr int PER = PAIRS ? 2 : 1;  // lines per transform
    const int64_t lines = A * Cc, units = (lines + PER - 1) / PER;
    grid_wait();
    for (int64_t u0 = (int64_t)blockIdx.x * C::NL; u0 < units; u0 += (int64_t)gridDim.x * C::NL) {
        const int64_t line = PER * (u0 + l);
        const bool act0 = line < lines, act1 = PAIRS && line + 1 < lines;
        const int64_t a = act0 ? line / Cc : 0, c = act0 ? line % Cc : 0;
        double *base0 = oct + a * n * Cc + c;
        double *base1 = c + 1 < Cc ? base0 + 1 : oct + (a + 1) * n * Cc;  // line + 1
        Cx<double> v[E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int p = t + m * NT;
            const int64_t q = (int64_t)(p <= L / 2 ? p : L - p) * Cc;
            v[m] = {act0 ? base0[q] : 0.0, act1 ? base1[q] : 0.0};
        }
        // every thread has read its lines before the first exchange's barrier,
        // and writes after the last one
        RowXch<double, L, E> xch{row};
        run_stages<double, L, E, false>(v, t, tw, xch, typename C::SH::Rad{});
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int k = t + m * NT;
            if (k <= L / 2) {
                if (act0) base0[(int64_t)k * Cc] = v[m].x;
                if (act1) base1[(int64_t)k * Cc] = v[m].y;
            }
        }
    }
}

// the lengths that kMeshLengths (launch.h) gives FP32 only, the 16-byte types
// only, and both
#define ISOFFT_DCT_LENGTHS_F32(X) X(324) X(432) X(648) X(1296)
#define ISOFFT_DCT_LENGTHS_16B(X) X(144)
#define ISOFFT_DCT_LENGTHS(X) \
    X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(288) X(384) X(512) X(576) X(768) X(1024) X(1152) X(1536) X(2048) \
    X(2304)

template <int L, bool PAIRS>
static cudaError_t run_cos_lines(double *oct, const Cx<double> *tw, int64_t A, int64_t Cc, cudaStream_t st)
{
    using C = DctCfg<L>;
    const int64_t units = PAIRS ? (A * Cc + 1) / 2 : A * Cc, groups = (units + C::NL - 1) / C::NL;
    const int grid = (int)(groups < 152 * 8 ? groups : 152 * 8);
    if (C::SMEM > 48 * 1024) {
        cudaError_t e =
            cudaFuncSetAttribute(k_cos_lines<L, PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
        if (e != cudaSuccess) return e;
    }
    return launch_pass(k_cos_lines<L, PAIRS>, dim3(grid), C::THREADS, C::SMEM, st, oct, tw, A, Cc);
}

// Cosine transform of every octant line along one axis of length M (one of
// the supported doubled lengths); tw = W_M^k, k < M.
template <bool PAIRS>
static cudaError_t cos_axis(int M, double *oct, const Cx<double> *tw, int64_t A, int64_t Cc, cudaStream_t st)
{
#define X_(n) \
    case n: return run_cos_lines<n, PAIRS>(oct, tw, A, Cc, st);
    switch (M) {
        ISOFFT_DCT_LENGTHS(X_)
    default: break;
    }
    if constexpr (PAIRS) {
        switch (M) {
            ISOFFT_DCT_LENGTHS_F32(X_)
        default: break;
        }
    } else {
        switch (M) {
            ISOFFT_DCT_LENGTHS_16B(X_)
        default: break;
        }
    }
#undef X_
    return cudaErrorInvalidValue;
}

// The three axis passes of the octant transform, in place on oct [Z][Y][X];
// tws[a] = W_{M_a}^k.
template <bool PAIRS>
static cudaError_t cos_transform(const int64_t M[3], double *oct, const Cx<double> *const tws[3], cudaStream_t st)
{
    const int64_t X = M[0] / 2 + 1, Y = M[1] / 2 + 1, Z = M[2] / 2 + 1;
    cudaError_t e = cos_axis<PAIRS>((int)M[0], oct, tws[0], Z * Y, 1, st);
    if (e == cudaSuccess) e = cos_axis<PAIRS>((int)M[1], oct, tws[1], Z, X, st);
    if (e == cudaSuccess) e = cos_axis<PAIRS>((int)M[2], oct, tws[2], 1, X * Y, st);
    return e;
}

// oct [Z][Y][X] (X = Mx/2 + 1) -> G in the z pass's tiled layout
// [Y][ntx][blk] with block element kz * tx + c (kx = xt * tx + c, zero past
// Kx = Mx/2, zero in the padding past Z * tx) and Gs [Y][Z], of type T;
// column kx = 0 packs the kx = 0 and kx = Mx/2 planes.
template <typename T>
static __global__ void k_pack(const double *__restrict__ oct, T *__restrict__ G, T *__restrict__ Gs, int X,
                              int Y, int Z, int tx, int ntx, int blk, double scale)
{
    const int Kx = X - 1;
    const int64_t tot = (int64_t)Y * ntx * blk;
    grid_wait();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < tot;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int j = (int)(i % blk);
        if (j >= Z * tx) {
            G[i] = (T)0;
            continue;
        }
        const int c = j % tx;
        const int64_t kz = j / tx;
        const int xt = (int)((i / blk) % ntx);
        const int64_t ky = i / ((int64_t)blk * ntx);
        const int kx = xt * tx + c;
        const double *o = oct + (kz * Y + ky) * X;
        if (kx >= Kx) {
            G[i] = (T)0;
        } else if (kx == 0) {
            const double g0 = o[0], gn = o[Kx];
            G[i] = (T)(0.5 * (g0 + gn) * scale);
            Gs[ky * Z + kz] = (T)(0.5 * (g0 - gn) * scale);
        } else {
            G[i] = (T)(o[kx] * scale);
        }
    }
}

template <typename T>
size_t spectrum_elems(const int64_t M[3])
{
    const int tx = z_tile_for<T>((int)M[2]);
    const size_t Y = M[1] / 2 + 1, Z = M[2] / 2 + 1, Kx = M[0] / 2;
    const size_t ntx = (Kx + tx - 1) / tx;
    return Y * ntx * (size_t)z_spec_block(tx, (int)Z, (int)sizeof(T)) + Y * Z;
}
template size_t spectrum_elems<float>(const int64_t *);
template size_t spectrum_elems<double>(const int64_t *);
template size_t spectrum_elems<df64>(const int64_t *);

void host_roots(int64_t n, int64_t count, double *re, double *im)
{
    // e^{-2 pi i k/n}: the angle, in units of 2 pi / (4 n), is reduced to the
    // first octant by the exact symmetries of the circle.
    for (int64_t k = 0; k < count; ++k) {
        int64_t u = 4 * (((k % n) + n) % n);
        const bool neg_s = u > 2 * n;  // lower half: sin negative
        if (neg_s) u = 4 * n - u;
        const bool neg_c = u > n;  // second quadrant: cos(pi - a) = -cos a, sin same
        if (neg_c) u = 2 * n - u;
        const bool swap = 2 * u > n;  // past the octant: cos and sin of the complement
        if (swap) u = n - u;
        const double a = 2.0 * M_PI * (double)u / (double)(4 * n);
        const double c = swap ? sin(a) : cos(a), s = swap ? cos(a) : sin(a);
        re[k] = neg_c ? -c : c;
        im[k] = neg_s ? s : -s;
    }
}

// Root tables of the three axes, W_{M_a}^k for k < M_a, one after another.
int64_t green_cos_elems(const int64_t M[3]) { return 2 * (M[0] + M[1] + M[2]); }
// The FP64 octant; its element count rounded up to even, so that root
// tables placed after it start on a 16-byte boundary (complex doubles).
int64_t green_octant_elems(const int64_t M[3])
{
    const int64_t n = (M[0] / 2 + 1) * (M[1] / 2 + 1) * (M[2] / 2 + 1);
    return (n + 1) & ~(int64_t)1;
}

size_t green_build_scratch_bytes(const int64_t M[3])
{
    return (size_t)(green_octant_elems(M) + green_cos_elems(M)) * sizeof(double);
}

static int grid_for(int64_t n)
{
    int64_t b = (n + 255) / 256;
    if (b > 152 * 64) b = 152 * 64;
    return (int)(b < 1 ? 1 : b);
}

// G from the transformed octant, in the z pass's layout and dtype.
template <typename T>
static cudaError_t pack_spectrum(const int64_t M[3], const double *oct, T *G, T *Gs, cudaStream_t st)
{
    const int X = (int)(M[0] / 2 + 1), Y = (int)(M[1] / 2 + 1), Z = (int)(M[2] / 2 + 1);
    const double scale = 1.0 / (2.0 * (double)M[0] * (double)M[1] * (double)M[2]);
    const int tx = z_tile_for<T>((int)M[2]);
    const int ntx = (int)((M[0] / 2 + tx - 1) / tx);
    const int blk = z_spec_block(tx, Z, (int)sizeof(T));
    return launch_pass(k_pack<T>, dim3(grid_for((int64_t)Y * ntx * blk)), 256, 0, st, oct, G, Gs, X, Y, Z, tx, ntx, blk,
                       scale);
}

// The octant of Eq. 9 (FP64), its three axis transforms in place, the pack.
// tws: the root tables of the three axes (green_cos_elems doubles).
template <typename T>
static cudaError_t spectrum_steps(const int64_t M[3], const double hn[3], T *G, T *Gs, double *oct,
                                  const double *tws, cudaStream_t st)
{
    const int X = (int)(M[0] / 2 + 1), Y = (int)(M[1] / 2 + 1), Z = (int)(M[2] / 2 + 1);
    if ((reinterpret_cast<uintptr_t>(tws) & 15) || (reinterpret_cast<uintptr_t>(oct) & 7))
        return cudaErrorMisalignedAddress;  // complex-double tables need 16-byte alignment
    constexpr bool PAIRS = std::is_same<T, float>::value;
    const int zc = Z > 128 ? 8 : 2;
    cudaError_t e = launch_pass(k_green_octant<PAIRS>, dim3((unsigned)((X * Y + 255) / 256), (unsigned)((Z + zc - 1) / zc)), 256,
                                0, st, oct, X, Y, Z, hn[0], hn[1], hn[2], zc);
    const Cx<double> *tw[3] = {reinterpret_cast<const Cx<double> *>(tws),
                               reinterpret_cast<const Cx<double> *>(tws) + M[0],
                               reinterpret_cast<const Cx<double> *>(tws) + M[0] + M[1]};
    if (e == cudaSuccess) e = cos_transform<PAIRS>(M, oct, tw, st);
    if (e == cudaSuccess) e = pack_spectrum<T>(M, oct, G, Gs, st);
    return e;
}

template <typename T>
cudaError_t build_green_spectrum(const int64_t M[3], const double hn[3], T *G, T *Gs, cudaStream_t st)
{
    const int64_t n = green_octant_elems(M), nt = green_cos_elems(M);
    // roots W_M^k per axis, by exact reduction to the first octant (host)
    std::vector<double> host(nt);
    int64_t off = 0;
    for (int a = 0; a < 3; ++a) {
        std::vector<double> re(M[a]), im(M[a]);
        host_roots(M[a], M[a], re.data(), im.data());
        for (int64_t k = 0; k < M[a]; ++k) {
            host[off + 2 * k] = re[k];
            host[off + 2 * k + 1] = im[k];
        }
        off += 2 * M[a];
    }
    double *buf = nullptr;
    cudaError_t e = cudaMalloc(&buf, (size_t)(n + nt) * sizeof(double));
    if (e != cudaSuccess) return e;
    e = cudaMemcpyAsync(buf + n, host.data(), nt * sizeof(double), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = spectrum_steps<T>(M, hn, G, Gs, buf, buf + n, st);
    cudaError_t e2 = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = e2;
    cudaFree(buf);
    return e;
}

// Same spectrum as build_green_spectrum, enqueued on `st` without allocating
// or synchronising: the FP64 octant lives in the caller's `oct` scratch
// (green_octant_elems(M) doubles), the FP64 root tables in `ct`
// (green_cos_elems(M) doubles).  k_tables computes these and, from the same
// roots, the solve's own tables: tw_x = W_Lx^k = W_Mx^2k and rtw = W_Mx^k for
// k < Lx = Mx/2, tw_y = W_My^k, tw_z = W_Mz^k.
template <typename T>
static __global__ void k_tables(double *__restrict__ ct, Cx<T> *__restrict__ tw_x, Cx<T> *__restrict__ rtw,
                                Cx<T> *__restrict__ tw_y, Cx<T> *__restrict__ tw_z, int mx, int my, int mz)
{
    grid_wait();
    const int tot = mx + my + mz;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += gridDim.x * blockDim.x) {
        const int axis = i < mx ? 0 : (i < mx + my ? 1 : 2);
        const int k = axis == 0 ? i : (axis == 1 ? i - mx : i - mx - my);
        const int m = axis == 0 ? mx : (axis == 1 ? my : mz);
        double sn, cs;
        sincospi(2.0 * (double)k / (double)m, &sn, &cs);
        ct[2 * i] = cs;
        ct[2 * i + 1] = -sn;
        const Cx<T> w = {(T)cs, (T)-sn};
        if (axis == 0) {
            if (k < mx / 2) rtw[k] = w;
            if ((k & 1) == 0) tw_x[k / 2] = w;
        } else {
            (axis == 1 ? tw_y : tw_z)[k] = w;
        }
    }
}

template <typename T>
cudaError_t enqueue_green_spectrum(const int64_t M[3], const double hn[3], T *G, T *Gs, double *oct, double *ct,
                                   void *tw_x, void *rtw, void *tw_y, void *tw_z, cudaStream_t st)
{
    cudaError_t e = launch_pass(k_tables<T>, dim3(grid_for(M[0] + M[1] + M[2])), 256, 0, st, ct, (Cx<T> *)tw_x,
                                (Cx<T> *)rtw, (Cx<T> *)tw_y, (Cx<T> *)tw_z, (int)M[0], (int)M[1], (int)M[2]);
    if (e == cudaSuccess) e = spectrum_steps<T>(M, hn, G, Gs, oct, ct, st);
    return e;
}
template cudaError_t enqueue_green_spectrum<float>(const int64_t *, const double *, float *, float *, double *,
                                                   double *, void *, void *, void *, void *, cudaStream_t);
template cudaError_t enqueue_green_spectrum<double>(const int64_t *, const double *, double *, double *, double *,
                                                    double *, void *, void *, void *, void *, cudaStream_t);

template cudaError_t build_green_spectrum<float>(const int64_t *, const double *, float *, float *,
                                                 cudaStream_t);
template cudaError_t build_green_spectrum<double>(const int64_t *, const double *, double *, double *,
                                                  cudaStream_t);
template cudaError_t build_green_spectrum<df64>(const int64_t *, const double *, df64 *, df64 *, cudaStream_t);

}  // namespace isofft
