// K1: batched banded solves t = B^{-1} f with B = diag(B_i) (Section 5.2),
// one subdomain per thread-block cluster of G CTAs, for sm_103a.
//
// Factor layout (built by host_band_factor): the Cholesky factor L_i is banded
// with half-bandwidth w; rows are grouped in planes of W rows.  For plane J
//   O_J = L_i[plane J, plane J-1]    upper triangular incl. diagonal,
//   D_J = L_i[plane J, plane J]^{-1} lower triangular incl. diagonal (inverted on the host),
//   forward  (L y = f):    t = f_J - O_J y_{J-1};          y_J = D_J t
//   backward (L^T x = y):  t = y_J - O_{J+1}^T x_{J+1};    x_J = D_J^T t
// All four products are "output row = sum over columns" of a triangular
// matrix (O_J, D_J^T upper; D_J, O_J^T lower), each stored on its own.  A plane's
// 32-row blocks are dealt to the G CTAs of a cluster (slices).  Each CTA's slice
// of a block is tiled: a row block keeps, for every four columns that meet it, one
// quad of 32 x 4 values (zero outside the triangle), a row's four together, row
// blocks one after the other, columns ascending.  A lane owns a row: a quad is one
// 16-byte shared load (two in FP64), a 16-byte broadcast load of the vector and four
// multiply-adds; the padding costs about 18 values per column (16% of a 225-wide block).
//
// A block's quads are dealt to the warps in contiguous shares; each warp streams its
// own shares through its own ring of shared slots with 1-D bulk asynchronous copies on
// its own mbarriers, so copies run ahead across planes and phases and no warp waits
// for another's slot.  A warp's partial sums of a row block form a "piece" (number
// warp + row block); a row's sum adds its few pieces in warp order after one CTA
// barrier per block.
// Each phase's input vector (t, or y/x) reaches every CTA of the cluster by
// st.async stores into distributed shared memory that complete bytes on the
// receiver's mbarrier, so a CTA waits only for the vector it reads and no
// cluster-wide barrier is taken per phase.  Every wait is a bounded spin that
// sets a device status word instead of hanging.  The shares depend on the plane width
// and the split only, not on the ring's slots or the number of right-hand sides.
#include "slr_band_kernel.cuh"

namespace slr {

template <typename T>
cudaError_t launch_band_solve(const DevOperator<T>& op, int32_t p, int32_t wmax, const T* in, int64_t ldi, T* out,
                              int64_t ldo, const T* base, int64_t ldb, int32_t nrhs, cudaStream_t st) {
    if (p == 0 || wmax == 0) return cudaSuccess;
    if constexpr (sizeof(T) == 4) {
        // blocks of right-hand sides on the tensor cores when the operator carries that factor
        if (op.band_tc && nrhs >= 8) return launch_band_solve_tc(op, p, in, ldi, out, ldo, base, ldb, nrhs, st);
    }
    // planes of at most 64 rows in one slice: four warps per subdomain (band_nt 32)
    if (op.band_nt == 32 && op.band_G == 1 && wmax <= 64)
        return launch_band_narrow(op, p, wmax, in, ldi, out, ldo, base, ldb, nrhs, st);
    for (int32_t c = 0; c < nrhs;) {
        // up to eight columns (FP64: four, which already keep its pipe busy) per launch
        // share one read of the factor, while the rings beside that many vectors hold six quads per warp
        const int32_t left = nrhs - c;
        const int nt = op.band_nt;
        int32_t nb, cq;
        auto fits = [&](int n) { return band_ring(wmax, n, sizeof(T), 0, nt, &nb, &cq) && nb * cq >= 6; };
        // FP64: three columns in a kernel of their own, since its pipe takes the absent fourth's
        // multiply-adds as well (B-solve of three columns on 3-D 60^3, 64 subdomains: 994 us by the kernel of
        // four, 1007 for four; 838 as two and one with the earlier kernels; 721 now)
        constexpr int three = sizeof(T) == 4 ? 4 : 3;
        const int nv = sizeof(T) == 4 && left > 4 && fits(8) ? 8
                       : left > 3 && fits(4)                 ? 4
                       : left > 2 && fits(three)             ? three
                       : left > 1 && fits(2)                 ? 2
                                                             : 1;
        const int nr = std::min(nv, left);
        const T* bs = base ? base + c * ldb : nullptr;
        cudaError_t e = cudaSuccess;
        const T* ic = in + c * ldi;
        T* oc = out + c * ldo;
        if (nt == 256) {
            if constexpr (sizeof(T) == 4) {
                if (nv == 8) e = band_launch_half<T, 8>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            }
            if constexpr (sizeof(T) == 8) {
                if (nv == 3) e = band_launch_half<T, 3>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            }
            if (nv == 4) e = band_launch_half<T, 4>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            else if (nv == 2) e = band_launch_half<T, 2>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            else if (nv == 1) e = band_launch_half<T, 1>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
        } else {
            if constexpr (sizeof(T) == 4) {
                if (nv == 8) e = band_launch_g<T, 8, 512>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            }
            if constexpr (sizeof(T) == 8) {
                if (nv == 3) e = band_launch_g<T, 3, 512>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            }
            if (nv == 4) e = band_launch_g<T, 4, 512>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            else if (nv == 2) e = band_launch_g<T, 2, 512>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
            else if (nv == 1) e = band_launch_g<T, 1, 512>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, nr, st);
        }
        if (e != cudaSuccess) return e;
        c += nr;
    }
    return cudaSuccess;
}

template cudaError_t launch_band_solve<double>(const DevOperator<double>&, int32_t, int32_t, const double*, int64_t,
                                               double*, int64_t, const double*, int64_t, int32_t, cudaStream_t);
template cudaError_t launch_band_solve<float>(const DevOperator<float>&, int32_t, int32_t, const float*, int64_t,
                                              float*, int64_t, const float*, int64_t, int32_t, cudaStream_t);

}  // namespace slr
