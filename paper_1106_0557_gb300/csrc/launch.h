// launch.h -- host-side launchers of the device passes (internal to the
// library; the public surface is include/isofft.h).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "df64.cuh"

namespace isofft {

// Doubled-mesh lengths.  Any M >= 2N - 1 gives the same cropped result, so a
// plan rounds 2N up, on each axis, to the next length that is worth taking
// there for its dtype.  Powers of two and 3/2 of them (and 2304) serve every
// axis; the lengths between are 9/8, 81/64 and 27/16 of a power of two, which
// the kernels reach in two or three stages of 12 to 48 points a thread.  A
// length that does not beat the next longer one on its axis is left out
// there (times of one pass, us, of 256 x 200 x 128-cell meshes with the axis
// at M/2 cells, half that for the 16-byte types):
//   FP32 z:  288 56, 324 84, 384 90, 432 120, 512 99, 576 107, 648 226,
//            768 199, 1024 230, 1152 298, 1296 469, 1536 577, 2048 841,
//            2304 949: 432 and 648 are left out (y takes them: 37 against
//            42 at 512, 65 + 72 against 72 + 66 at 768, with 16 % fewer z
//            lines);
//   FP32 x:  432 31 + 33 against 22 + 23 at 512: left out; elsewhere a few
//            per cent on the x passes buy 9 to 16 % fewer columns;
//   df64 z:  lines of powers of two hold more warps and no radix 3: 192 70,
//            288 126, 512 154, 576 302, 1024 344, 1152 522, 1536 876, 2048 913,
//            2304 1467; with fewer roundings, which were not kept, 144 took 69
//            (192: 69), 384 194 and 768 401, so those are not
//            taken on z, and 324 319, 432 226 and 648 658, so those on no axis;
//   FP64 z:  144 220, 192 303, 288 509, 324 742, 384 673, 576 1112, 648 1550,
//            768 1457, 1152 2455, 1296 3375, 1536 3373, 2048 4284, 2304 5416.
enum { kDtF32 = 0, kDtF64 = 1, kDtDf64 = 2 };  // = ipf_dtype
struct MeshLength {
    int m;
    unsigned char axes[3];  // by dtype: bit a set where axis a (x, y, z) takes it
};
constexpr MeshLength kMeshLengths[] = {
    {32, {7, 7, 7}},   {48, {7, 7, 7}},   {64, {7, 7, 7}},   {96, {7, 7, 7}},   {128, {7, 7, 7}},  {144, {0, 7, 3}},
    {192, {7, 7, 7}},  {256, {7, 7, 7}},  {288, {7, 7, 7}},  {324, {7, 0, 0}},  {384, {7, 7, 3}},  {432, {2, 0, 0}},
    {512, {7, 7, 7}},  {576, {7, 7, 7}},  {648, {3, 0, 0}},  {768, {7, 7, 3}},  {1024, {7, 7, 7}}, {1152, {7, 7, 7}},
    {1296, {7, 0, 0}}, {1536, {7, 7, 7}}, {2048, {7, 7, 7}}, {2304, {7, 7, 7}}};
constexpr int kMaxM = 2304;
// Whether z lines of length Mz have an instance on a z-blocked workspace (1296
// points would need blocks of 8 planes or less).
constexpr bool z_blocks(int Mz, bool f32)
{
    return Mz == 2304 || (f32 && (Mz == 768 || Mz == 1024 || Mz == 1152 || Mz == 1536 || Mz == 2048));
}

// The doubled length of n cells on an axis (-1 beyond the longest).  `blocked`:
// only the lengths whose y passes also run on a z-blocked workspace.
inline int mesh_length(int64_t n, int dtype, int axis, bool blocked = false)
{
    for (const MeshLength &c : kMeshLengths) {
        const bool basic = (c.m & (c.m - 1)) == 0 ? c.m != 2048 : (c.m % 9 != 0 || c.m == 2304);
        if (c.m >= 2 * n && (c.axes[dtype] >> axis & 1) && (basic || !blocked)) return c.m;
    }
    return -1;
}

// Counts every kernel launch the library makes (ipf_launch_count).
void count_launch();

// All pointers are device pointers of the current device; complex buffers
// are interleaved (re, im) of the arithmetic type T; source and potential
// arrays hold IoReal<T>::type (double for df64).
// `zsh`: the workspace's z planes are grouped in blocks of 2^zsh (w_row in
// passes.cuh; 0 = plain [Nz][My][Kx]).  A launch on a part of the planes
// starts at a block.
// Planes per z block of a blocked workspace, as a shift: 16 (plan_zsh in
// api.cu says which meshes take it).  The z pass then reads each line group
// in runs of 16 rows one Kx row (9 KB at 1152^3) apart instead of rows a whole
// plane (21 MB) apart: 32-byte strided reads measured 3.5 TB/s against 1.5
// TB/s.  Blocks of 4 and 8 planes measured the same within 1 % (36.2 ms
// against 37.1 and 37.2 for K3 at 1152^3).
constexpr int kZBlockShift = 4;
template <typename T>
cudaError_t launch_x_forward(int L, const typename IoReal<T>::type *src, void *W, const void *tw, const void *rtw,
                             int Nx, int Ny, int My, int64_t nrows, int zsh, cudaStream_t st);
template <typename T>
cudaError_t launch_x_inverse(int L, const void *W, typename IoReal<T>::type *phi, const void *tw, const void *rtw,
                             int Nx, int Ny, int My, int64_t nrows, int zsh, cudaStream_t st);
// The y passes come in three forms with bitwise the same arithmetic:
//   kYTile        one CTA per column tile (plain loads; many CTAs per SM),
//   kYStream      persistent CTAs fed by tensor-map copies (see passes.cuh),
//   kYTileNarrow  the tile form on tiles of half the width.
// Plans pick one per pass by timing all three (y_default_variant without).
enum { kYTile = 0, kYStream = 1, kYTileNarrow = 2 };
constexpr int kYForms = 3;
template <typename T>
cudaError_t launch_y_forward(int L, void *W, const void *tw, int Ny, int Kx, int Nz, int zsh, unsigned *status,
                             int variant, cudaStream_t st);
template <typename T>
cudaError_t launch_y_inverse(int L, void *W, const void *tw, int Ny, int Kx, int Nz, int zsh, unsigned *status,
                             int variant, cudaStream_t st);
// The form used without timing: streamed for 8-byte points on lines of 512
// to 1024 points (where it measured faster), tiles elsewhere.
inline int y_default_variant(int L, size_t real_bytes)
{
    return real_bytes == 4 && L >= 512 && L <= 1024 ? kYStream : kYTile;
}
// `status` (device word, may be null) gets bit 0 set when one of the pass's
// bounded waits for its tile copies gave up (ipf_plan_check reads it); the
// y passes and the z pass share it.  `test_extra_tx` (normally 0) is the
// run-out test hook: bytes each CTA's first tile expects beyond its copies.
template <typename T>
cudaError_t launch_z_convolve(int L, void *W, const void *tw, const T *G, const T *Gs, T gscale, int Nz,
                              int My, int Kx, int zsh, unsigned *status, unsigned test_extra_tx, cudaStream_t st);

// Width (kx columns per tile) of the z pass for line length L; the cached
// Green's spectrum is stored in tiles of this width (0: unsupported L).
template <typename T>
int z_tile_for(int L);

// The lengths between powers of two and 3/2 of them (passes_inst.cu, part
// 2); the launchers above call these for lengths of their own that they lack.
template <typename T>
cudaError_t launch_x_forward_more(int L, const typename IoReal<T>::type *src, void *W, const void *tw, const void *rtw,
                                  int Nx, int Ny, int My, int64_t nrows, int zsh, cudaStream_t st);
template <typename T>
cudaError_t launch_x_inverse_more(int L, const void *W, typename IoReal<T>::type *phi, const void *tw, const void *rtw,
                                  int Nx, int Ny, int My, int64_t nrows, int zsh, cudaStream_t st);
template <typename T>
cudaError_t launch_y_forward_more(int L, void *W, const void *tw, int Ny, int Kx, int Nz, int zsh, unsigned *status,
                                  int variant, cudaStream_t st);
template <typename T>
cudaError_t launch_y_inverse_more(int L, void *W, const void *tw, int Ny, int Kx, int Nz, int zsh, unsigned *status,
                                  int variant, cudaStream_t st);
template <typename T>
cudaError_t launch_z_convolve_more(int L, void *W, const void *tw, const T *G, const T *Gs, T gscale, int Nz, int My,
                                   int Kx, int zsh, unsigned *status, unsigned test_extra_tx, cudaStream_t st);
template <typename T>
int z_tile_for_more(int L);

// Elements of one (k_y', kx tile) block of the cached spectrum: nkz x tx
// values, padded so that every block starts on a 16-byte boundary (the z pass
// copies a block with one bulk copy).
constexpr int z_spec_block(int tx, int nkz, int elem_bytes)
{
    return (nkz * tx + 16 / elem_bytes - 1) / (16 / elem_bytes) * (16 / elem_bytes);
}

// Device bytes of the cached Green's spectrum of a doubled mesh M.
template <typename T>
size_t spectrum_elems(const int64_t M[3]);

// Green's spectrum (FP64 build).  M = doubled mesh, hn = widths divided by
// their minimum.  Writes G [My/2+1][Mz/2+1][Mx/2] and Gs [My/2+1][Mz/2+1] of
// type T in the z pass's tiled layout, pre-divided by 2 Mx My Mz (see
// passes.cuh).  Allocates and frees its FP64 scratch; synchronises `st`
// before returning.
template <typename T>
cudaError_t build_green_spectrum(const int64_t M[3], const double hn[3], T *G, T *Gs, cudaStream_t st);

// The same spectrum enqueued without allocating or synchronising, in caller
// scratch: `oct` holds green_octant_elems(M) doubles (the FP64 octant,
// transformed in place), `ct` holds green_cos_elems(M) doubles (the root
// tables of the three axes, computed on the device).  The solve's root tables
// (complex T: tw_x and rtw of Mx/2 points, tw_y of My, tw_z of Mz) are filled
// by the same launch.
template <typename T>
cudaError_t enqueue_green_spectrum(const int64_t M[3], const double hn[3], T *G, T *Gs, double *oct, double *ct,
                                   void *tw_x, void *rtw, void *tw_y, void *tw_z, cudaStream_t st);
int64_t green_octant_elems(const int64_t M[3]);
int64_t green_cos_elems(const int64_t M[3]);

// Device bytes of the FP64 scratch build_green_spectrum needs for mesh M.
size_t green_build_scratch_bytes(const int64_t M[3]);

// One grid of a batch run in one launch per pass (batch.cu): the plan's
// buffers and sizes.
struct BatchGridDesc {
    const void *src;
    void *phi;
    void *W;
    const void *tw_x, *rtw, *tw_y, *tw_z;
    const void *G, *Gs;
    double gscale;
    int Nx, Ny, Nz, Mx, My, Mz;
    int runout;  // test hook (IPF_FLAG_TEST_WAIT_RUNOUT): in one launch, the z items' wait runs out
};
// Whether a grid of this dtype and doubled mesh can join a batched launch
// (FP32, every doubled length at most 256).
bool batch_fits(int dtype_is_f32, const int64_t M[3]);
// The five passes of `count` such grids on `st`: mode 1, one launch per
// pass; mode 2, one persistent launch for all five (per-(grid, pass)
// completion counters; a wait that runs out sets bit 0 of *status, which
// may be null).  The first call for a given set of grids builds and uploads
// its work tables (synchronously); later calls only launch.
cudaError_t batch_enqueue(const BatchGridDesc *grids, int count, int mode, unsigned *status, cudaStream_t st);

// e^{-2 pi i k / n} for 0 <= k < count, by exact reduction to the first
// octant (host, libm in double).
void host_roots(int64_t n, int64_t count, double *re, double *im);

}  // namespace isofft
