// dispatch.h -- entry points of the per-lattice kernel translation units.
#pragma once
#include <cuda_runtime.h>
#include <cstddef>
#include <cstdint>

namespace rr {

struct StepParams;

enum { PREC_FP64 = 0, PREC_FP32 = 1, PREC_FP16 = 2, PREC_BF16 = 3 };

cudaError_t step_d2q9(int precision, const StepParams &p, const void *fin, void *fout, int block,
                      cudaStream_t st);
cudaError_t step_d3q19(int precision, const StepParams &p, const void *fin, void *fout, int block,
                       cudaStream_t st);
cudaError_t step_d3q27(int precision, const StepParams &p, const void *fin, void *fout, int block,
                       cudaStream_t st);

// In-place AA streaming on one lattice f: one step (loc: the local step, else
// gather-push) and the conversion of the push layout to the standard one
cudaError_t step_aa_d2q9(int precision, const StepParams &p, void *f, int block, bool loc, cudaStream_t st);
cudaError_t step_aa_d3q19(int precision, const StepParams &p, void *f, int block, bool loc, cudaStream_t st);
cudaError_t step_aa_d3q27(int precision, const StepParams &p, void *f, int block, bool loc, cudaStream_t st);
cudaError_t aa_unswap_d2q9(int precision, const StepParams &p, void *f, cudaStream_t st);
cudaError_t aa_unswap_d3q19(int precision, const StepParams &p, void *f, cudaStream_t st);
cudaError_t aa_unswap_d3q27(int precision, const StepParams &p, void *f, cudaStream_t st);

}  // namespace rr

namespace rr {

// Message returned by lbm_last_error(NULL) (for calls without a handle)
void rr_set_global_error(const char *msg);

// Vectorised kernel (no cell-type mask, nx % vec == 0).  Supported (precision,
// vec): FP64 2; FP32 2, 4; FP16 2, 4; BF16 2, 4.  sp: 0 the two-lattice pull
// (fin read, fout written), 1 / 2 the AA gather-push / local step (in place,
// fin == fout).
cudaError_t stepvec_d2q9(int precision, int vec, const StepParams &p, const void *fin, void *fout,
                         int block, cudaStream_t st, int sp = 0);
cudaError_t stepvec_d3q19(int precision, int vec, const StepParams &p, const void *fin, void *fout,
                          int block, cudaStream_t st, int sp = 0);
// D3Q27: two cells per thread (four fall back to the general kernel)
cudaError_t stepvec_d3q27(int precision, int vec, const StepParams &p, const void *fin, void *fout,
                          int block, cudaStream_t st, int sp = 0);

// Cells per thread the vectorised kernel supports for a precision (0: none)
inline bool vec_supported(int precision, int vec)
{
    switch (precision) {
    case PREC_FP64: return vec == 2;
    case PREC_FP32: return vec == 2 || vec == 4;
    case PREC_FP16:
    case PREC_BF16: return vec == 2 || vec == 4;
    }
    return false;
}
// Whether the vectorised pull takes a storage shift: two cells per thread of
// 16-bit storage, where the shift is for, and of D2Q9 FP32
constexpr bool vec_shift_supported(int q, size_t elem, int vec)
{
    return vec == 2 && (elem == 2 || (elem == 4 && q == 9));
}
// Default cells per thread, measured on GB300 (round jet 384 x 256 x 256,
// G cell updates/s, one cell per thread vs two): D3Q19 FP16 52.9 vs 63.2,
// FP64 2.05 vs 2.00, FP32 at the copy bandwidth either way; D3Q27 FP32 31.4
// vs 32.4, FP16 38.0 vs 44.5.  D2Q9, us per step of a periodic box, one vs two:
// FP32 1024^2 9.8 vs 8.1, 512^2 3.9 vs 3.5, FP16 1024^2 9.7 vs 7.0, 512^2 3.9 vs 3.0,
// 256^2 2.45 vs 2.30.
inline int vec_default(int lattice, int precision)
{
    if (precision == PREC_FP64) return 1;
    if (precision == PREC_FP32) return lattice == 1 /* D3Q19 */ ? 1 : 2;
    return 2;
}
// Small D2Q9 lattices whose in-place steps run one cell per thread by default
// when the y axis is not periodic: the two rows next to its faces take the general
// update, in the vectorised kernel V cells one after the other, and finish last.
// GB300, us per step, one cell / two (inlet, outflow on the other faces): FP32
// 128^2 4.12 / 5.57, 512^2 6.87 / 7.38, 700 x 400 7.19 / 7.69, 1024 x 512 9.95 / 9.14;
// FP16 128^2 4.23 / 5.38, 256^2 4.55 / 5.64, 512^2 7.09 / 6.77.  The lines through these
// cross at 360 000 and 210 000 cells.
inline bool aa_small_2d(int64_t ncell, size_t elem) { return ncell <= (elem == 4 ? 360000 : 210000); }
// Default threads per block.  The vectorised kernel's blocks lie along x
// rows of nx / vec threads, so the block has to divide the row's warps or the
// last block of every row holds idle warps: 64 threads where the row is a
// whole number of 64-thread blocks, one block for a row of up to three warps,
// else single warps.  Measured on GB300 (16-bit storage, two cells per
// thread), us per step at 64 / 32 / 96 threads: rows of 96 threads (192 x 128 x
// 128 jet) D3Q27 96.8 / 78.2 / 76.0, D3Q19 63.9 / 50.6 / 51.5; rows of 192 threads
// (384 x 256 x 256 jet) D3Q19 338.6 / 336.8 / 338.6.
inline int block_default(int vec, int nx)
{
    if (vec == 1) return 128;
    const int row = (nx / vec + 31) / 32 * 32;
    return row % 64 == 0 ? 64 : (row <= 96 ? row : 32);
}

// Every other step (odd) sweeps the lattice backwards (sweep_y) where a step
// moves over twice the L2's bytes.  GB300, us per pass, forwards / alternating:
// D3Q27 FP16 192 x 128 x 128 jet (340 MB a step) 5011 / 4871, D3Q19 384 x 256 x 256 jets
// FP16 (1.9 GB) 18236 / 18131, BF16 in place 21825 / 21548; below, the rows are in L2
// either way and it gained nothing (D3Q19 FP16 161 x 129 x 97, 150 MB, 4075 / 4117;
// D2Q9 FP16 1024^2 1619 / 1634).
inline bool sweep_back(int q, size_t elem, int64_t ncell, int64_t l2_bytes, bool odd)
{
    return odd && 2 * (int64_t)elem * q * ncell > 2 * l2_bytes;
}

// Row-staged kernel (bulk copies of whole rows into shared memory; FP32,
// FP16, BF16; no cell-type mask; nx * element size a multiple of 16 bytes).
struct RowsPlan {
    int R;        // rows per tile
    int RS;       // elements per direction and stage (R nx)
    int stages;   // shared-memory stages
    int block;    // threads per CTA
    int grid;     // CTAs (resident: SMs x CTAs per SM, at most the tile count)
    int per_sm;   // CTAs resident per SM
    size_t smem;  // dynamic shared memory per CTA, bytes
};
// cudaErrorNotSupported (nothing launched, no CUDA error state): not eligible
// wait_ns: limit of each wait for a tile's bulk copies (0: one non-blocking
// test, for failure-path tests)
cudaError_t rows_d2q9(int precision, const StepParams &p, const void *fin, void *fout, int block, int stages,
                      unsigned *err, uint64_t wait_ns, cudaStream_t st);
cudaError_t rows_d3q19(int precision, const StepParams &p, const void *fin, void *fout, int block, int stages,
                       unsigned *err, uint64_t wait_ns, cudaStream_t st);
cudaError_t rows_plan_d2q9(int precision, const StepParams &p, const void *fin, const void *fout, int block,
                           int stages, RowsPlan &pl);
cudaError_t rows_plan_d3q19(int precision, const StepParams &p, const void *fin, const void *fout, int block,
                            int stages, RowsPlan &pl);

}  // namespace rr
