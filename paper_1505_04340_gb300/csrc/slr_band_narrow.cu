// K1 for narrow planes (W <= 64: the 2-D workloads and 3-D boxes of at most 8 x 8):
// one CTA of four warps per subdomain.
//
// With one slice per subdomain the factor layout is the one slr_band.cu describes:
// row blocks 0 and 1 (rows 32 rb .. 32 rb + 31), and per block of a plane the
// quads (32 rows x 4 columns) that meet the triangle, row
// blocks one after the other, columns ascending.  Warp w takes the quads
// w, w + 4, .. of every block (columns 4 w + 16 k + u, u < 4); a lane owns rows lane
// and 32 + lane.
//
// What bounds it is the chain of 4 c - 2 small blocks (c planes), so a block is made
// as short as the machine allows.  One CTA barrier per block:
//   before it  each warp reads its quads of the block (they landed long ago: the
//              ring holds several whole blocks) from shared memory into registers;
//   after it   the previous block's partial sums of all warps are visible, and the
//              slot that every warp has just read is refilled by a fifth warp, which
//              does nothing but issue copies.  A lane per (column, right-hand side)
//              of its warp adds the four partial sums to the input vector's entry,
//              which the warp keeps to itself, and the products follow from registers.
// Results and right-hand sides move between a lane and global memory for the same
// (column, right-hand side) in both passes, so the backward pass reads what its own
// thread wrote; right-hand sides are loaded two planes ahead.
// Measured: FV 1024^2 in 256 subdomains (W = 62, 62 planes), FP32: 131 us per B-solve, in which
// the kernel moves 0.78 GB of DRAM traffic at 6.0 TB/s (the quads' padding included); one warp per
// subdomain walking every segment in turn took 405 us.  2-D 32^2 (W = 15, FP64): 82 -> 40 us, bound
// by the latency of 58 blocks' seven dependent FP64 operations each.
//
// Up to eight right-hand sides (FP64: four) share a launch (the factor is read once).  Each sums its
// products in the same order whatever their number.  Every wait is bounded: one that
// runs out sets the status word and the CTA's abort flag; the CTA then issues no
// more copies and multiplies nothing, waits (bounded) for the copies it issued and
// returns.
#include <type_traits>

#include "slr_band_kernel.cuh"

namespace slr {
namespace {

constexpr int kNw = 4;                      // warps per subdomain
constexpr int kNc = 16;                     // columns of a plane a warp takes (64 / kNw)
constexpr int kNSlots = 8;                  // ring slots at most, each a whole block
// right-hand sides per launch at most (FP64: four keep its pipe busy; eight would spill)
template <typename T>
constexpr int kNMaxR = sizeof(T) == 4 ? 8 : 4;

// elements of a ring slot, the largest block of a plane of W rows
__host__ __device__ inline int narrow_slot(int W) { return 32 * (((W + 3) & ~3) + (W <= 32 ? 0 : 32)); }

// NV consecutive values from shared memory (16-byte aligned)
template <typename T, int NV>
__device__ __forceinline__ void ld_row(const T* p, T (&v)[NV]) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int q = 0; q < NV; q += 4) {
            const float4 a = *reinterpret_cast<const float4*>(p + q);
            v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < NV; q += 2) {
            const double2 a = *reinterpret_cast<const double2*>(p + q);
            v[q] = a.x; v[q + 1] = a.y;
        }
    }
}

template <typename T, int NR>
__global__ void __launch_bounds__(32 * (kNw + 1), 2)
k_band_narrow(const BandBlock* __restrict__ blocks, const T* __restrict__ fac, const T* in, int64_t ldi, T* out,
              int64_t ldo, const T* base, int64_t ldb, int32_t* err, int nslot, int slot, int once) {
    constexpr int NIT = (kNc * NR + 31) / 32;          // (column, right-hand side) pairs per lane
    constexpr int PB = kNw * NR * 64;                  // partial sums of a block
    extern __shared__ __align__(128) unsigned char smem[];
    const int W = blocks[blockIdx.x].w, c = blocks[blockIdx.x].c, m = blocks[blockIdx.x].m;
    if (m == 0) {
        dep_wait();
        return;
    }
    const int SU = blocks[blockIdx.x].SU, SL = blocks[blockIdx.x].SL;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint64_t* full = reinterpret_cast<uint64_t*>(smem);                      // [kNSlots]
    volatile int* abort_flag = reinterpret_cast<volatile int*>(full + kNSlots);
    T* part = reinterpret_cast<T*>(smem + 128);          // [2][kNw][NR][64] partial sums, by block parity
    T* ring = part + 2 * PB + kNw * kNc * NR;
    const int nblk = 4 * c - 2;
    if (tid == 0) {
        for (int i = 0; i < nslot; ++i) mbar_init(&full[i], 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    __syncthreads();
    if (warp == kNw) {
        // ---------------------------------------------------------------- copies
        // Block q of the stream (forward D_0, then (O_J, D_J); backward D_{c-1}^T, then
        // (O_{J+1}^T, D_J^T)) goes to slot q mod nslot, once every warp has read the
        // block before it there (the barrier of that block).
        const T* fac0 = fac + blocks[blockIdx.x].foff;
        int type = 1, plane = 0, issued = 0, sl = 0;
        const uint64_t pol = policy_stream(once != 0);
        auto issue = [&]() {
            const int64_t off = (int64_t)plane * 2 * (SU + SL) +
                                (type == 0 ? 0 : type == 1 ? SU : type == 2 ? SU + SL : SU + 2 * SL);
            const uint32_t bytes = (uint32_t)((type == 0 || type == 3 ? SU : SL) * (int)sizeof(T));
            mbar_arrive_expect_tx(&full[sl], bytes);
            bulk_g2s(ring + (size_t)sl * slot, fac0 + off, bytes, &full[sl], pol);
            next_block(c, type, plane);
            ++issued;
            if (++sl == nslot) sl = 0;
        };
        if (lane == 0)
            while (issued < nslot && issued < nblk) issue();
        for (int q = 0; q < nblk; ++q) {
            __syncthreads();
            if (lane == 0 && issued < nblk && !*abort_flag) {
                fence_proxy_async();
                issue();
            }
        }
        __syncthreads();
        // after an abort: the last copy issued into each slot has landed before the CTA leaves
        if (lane == 0 && *abort_flag) {
            for (int s = 0; s < nslot && s < issued; ++s) {
                const int last = s + ((issued - 1 - s) / nslot) * nslot;
                long long it = 0;
                while (!mbar_try_wait(&full[s], (uint32_t)((last / nslot) & 1)) && ++it <= kSpin) {
                }
            }
        }
        return;
    }
    // ------------------------------------------------------------------ products
    dep_wait();                                          // (the copy warp reads the factor only)
    const bool two = W > 32;
    T* vw = part + 2 * PB + warp * kNc * NR;             // [kNc][NR] this warp's entries of the input vector
    // the lane's pairs: column (past W: none), right-hand side; only the last plane has rows past m
    const int mlast = m - (c - 1) * W;
    bool act[NIT], last[NIT];
    int px[NIT], vx[NIT];
    const T *pi[NIT], *pb[NIT];
    T *po[NIT], *py[NIT];
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
        const int e = it * 32 + lane, i = e % kNc, j = e / kNc, cc = 4 * warp + 16 * (i / 4) + i % 4;
        act[it] = e < kNc * NR && cc < W;
        last[it] = act[it] && cc < mlast;
        px[it] = act[it] ? j * 64 + cc : 0;
        vx[it] = e < kNc * NR ? i * NR + j : -1;
        const int64_t r = blocks[blockIdx.x].row0 + cc;
        pi[it] = in + r + j * ldi;
        po[it] = out + r + j * ldo;
        py[it] = po[it];
        pb[it] = base + r + j * ldb;
    }
    const T *rd = part + PB, *wr0 = part;                // the previous block's sums, this block's
    auto psum = [&](int it) -> T {
        const T* p = rd + px[it];
        return (p[0] + p[NR * 64]) + (p[2 * NR * 64] + p[3 * NR * 64]);
    };
    int sl = 0;
    uint32_t par = 0;
    const int coff = warp * 128 + lane * 4;              // first quad, this lane's row
    // One block: vin(it) is the entry of the input vector of the lane's pair it.
    auto step = [&](auto up, auto vin) {
        constexpr bool UP = decltype(up)::value;
        constexpr int N0 = UP ? kNc : kNc / 2, S1 = UP ? kNc / 2 : 0;   // columns of row block 0; first of block 1
        {
            long long it = 0;
            while (!mbar_try_wait(&full[sl], par)) {
                if (++it > kSpin || *abort_flag) {       // the products below are then invalid, as the status says
                    atomicExch(err, 1);
                    *abort_flag = 1;
                    break;
                }
            }
        }
        const T* P = ring + (size_t)sl * slot + coff;
        // row block 1: column 0 of a lower, -32 of an upper block
        const T* P1 = P + 32 * (UP ? ((W + 3) & ~3) - 32 : 32);
        if (++sl == nslot) {
            sl = 0;
            par ^= 1;
        }
        T a0[N0], a1[kNc - S1];
#pragma unroll
        for (int g = 0; g < kNc / 4; ++g) {
            if (4 * warp + 16 * g >= W) break;           // past the plane
            if (4 * g < N0) ld_row<T, 4>(P + 128 * kNw * g, *reinterpret_cast<T(*)[4]>(&a0[4 * g < N0 ? 4 * g : 0]));
        }
        if (two) {
#pragma unroll
            for (int g = S1 / 4; g < kNc / 4; ++g) {
                if (4 * warp + 16 * g >= W) break;
                ld_row<T, 4>(P1 + 128 * kNw * g, *reinterpret_cast<T(*)[4]>(&a1[4 * g - S1]));
            }
        }
        __syncthreads();
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
            const T v = vin(it);
            if (NIT * 32 == kNc * NR || vx[it] >= 0) vw[vx[it]] = act[it] ? v : T(0);
        }
        __syncwarp();
        T acc0[NR], acc1[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) acc0[j] = acc1[j] = T(0);
#pragma unroll
        for (int g = 0; g < kNc / 4; ++g) {
            if (4 * warp + 16 * g >= W) break;
            T v[4 * NR];
            ld_row<T, 4 * NR>(vw + 4 * NR * g, v);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = 4 * g + u;
                if (i < N0) {
#pragma unroll
                    for (int j = 0; j < NR; ++j) acc0[j] = fma(a0[i < N0 ? i : 0], v[u * NR + j], acc0[j]);
                }
            }
            if (g >= S1 / 4 && two) {
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = 4 * g + u - S1;
#pragma unroll
                    for (int j = 0; j < NR; ++j) acc1[j] = fma(a1[i >= 0 ? i : 0], v[u * NR + j], acc1[j]);
                }
            }
        }
        T* p = const_cast<T*>(wr0) + warp * NR * 64 + lane;
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            p[j * 64] = acc0[j];
            if (two) p[j * 64 + 32] = acc1[j];
        }
        const T* t = rd;
        rd = wr0;
        wr0 = t;
    };
    const std::true_type upper{};
    const std::false_type lower{};

    // =================================================================== forward
    T f0[NIT] = {}, f1[NIT] = {};
    int nf = 0;                                          // the next plane to load
    auto load_f = [&](int it) -> T { return (nf < c - 1 ? act[it] : nf == c - 1 && last[it]) ? *pi[it] : T(0); };
    auto each = [&](auto f) {
#pragma unroll
        for (int it = 0; it < NIT; ++it) f(it);
    };
    auto next_f = [&](int it) -> T {                     // F of the plane; the load of the plane after next
        const T f = f0[it];
        f0[it] = f1[it];
        f1[it] = load_f(it);
        pi[it] += W;
        return f;
    };
    each([&](int it) { f0[it] = load_f(it); pi[it] += W; });
    ++nf;
    each([&](int it) { f1[it] = load_f(it); pi[it] += W; });
    ++nf;
    step(lower, next_f);                                                     // D_0 F_0
    for (int J = 1; J < c; ++J) {
        ++nf;
        step(upper, [&](int it) {                                          // O_J y_{J-1}
            const T y = psum(it);
            if (act[it]) *po[it] = y;
            po[it] += W;
            return y;
        });
        step(lower, [&](int it) { return next_f(it) - psum(it); });        // D_J t
    }
    // =================================================================== backward
    // po stands at plane c - 1; y of the planes below it was written by this thread
    T b0[NIT], b1[NIT];
    int ny = c - 2, nb = c - 1;                          // the next planes of y and of the base to load
    each([&](int it) { py[it] = po[it] - W; pb[it] += (int64_t)(c - 1) * W; });
    auto load_y = [&](int it) -> T { return (ny >= 0 && act[it]) ? *py[it] : T(0); };
    auto load_b = [&](int it) -> T {
        return (base && nb >= 0 && (nb == c - 1 ? last[it] : act[it])) ? *pb[it] : T(0);
    };
    each([&](int it) { f0[it] = load_y(it); py[it] -= W; b0[it] = load_b(it); pb[it] -= W; });
    --ny, --nb;
    each([&](int it) { f1[it] = load_y(it); py[it] -= W; b1[it] = load_b(it); pb[it] -= W; });
    --ny, --nb;
    auto put_x = [&](int it, T x, bool ok) {             // x of the plane; the load of the base two planes below
        if (ok) *po[it] = base ? b0[it] - x : x;
        po[it] -= W;
        b0[it] = b1[it];
        b1[it] = load_b(it);
        pb[it] -= W;
    };
    step(upper, [&](int it) { return psum(it); });                           // D_{c-1}^T y_{c-1}
    for (int J = c - 2; J >= 0; --J) {
        step(lower, [&](int it) {                                          // O_{J+1}^T x_{J+1}
            const T x = psum(it);
            put_x(it, x, J == c - 2 ? last[it] : act[it]);
            return x;
        });
        --nb;
        step(upper, [&](int it) {                                          // D_J^T t
            const T y = f0[it];
            f0[it] = f1[it];
            f1[it] = load_y(it);
            py[it] -= W;
            return y - psum(it);
        });
        --ny;
    }
    __syncthreads();
    each([&](int it) { put_x(it, psum(it), c == 1 ? last[it] : act[it]); });
}

template <typename T, int NR>
cudaError_t narrow_launch(const DevOperator<T>& op, int32_t p, int32_t wmax, const T* in, int64_t ldi, T* out,
                          int64_t ldo, const T* base, int64_t ldb, cudaStream_t st) {
    auto kern = k_band_narrow<T, NR>;
    constexpr size_t kCap = 200 * 1024;
    static std::mutex mu;
    static uint64_t raised = 0;                     // bit d: the limit is raised on device d
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lk(mu);
        if (!(raised >> dev & 1)) {
            e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCap);
            if (e != cudaSuccess) return e;
            raised |= 1ull << dev;
        }
    }
    // whole blocks in flight: as many as fit, 2 .. 8, in the shared memory of an SM divided
    // by the subdomains that share it (at most four)
    const size_t fixed = 128 + (size_t)(2 * kNw * 64 + kNw * kNc) * NR * sizeof(T);
    const int32_t slot = narrow_slot(wmax), sb = slot * (int32_t)sizeof(T);
    const int32_t share = std::min(4, std::max(1, (p + op.cf.nsm - 1) / op.cf.nsm));
    const size_t budget = std::min(kCap, (size_t)(224 * 1024) / share - 1024);
    const int32_t nslot =
        std::max<int32_t>(2, std::min<int32_t>(kNSlots, (int32_t)((budget - std::min(budget, fixed)) / sb)));
    if (fixed + (size_t)nslot * sb > kCap) return cudaErrorInvalidValue;
    const cudaError_t e = launch_dep(kern, p, 32 * (kNw + 1), fixed + (size_t)nslot * sb, st, op.band, op.bfac, in, ldi, out,
                                     ldo, base, ldb, op.err, nslot, slot, op.bfac_len * (int64_t)sizeof(T) > kL2Keep ? 1 : 0);
    if (e != cudaSuccess) return e;
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

// The narrow-plane band solve (planes of at most 64 rows, one slice per subdomain):
// up to eight (FP64: four) right-hand sides per launch.
template <typename T>
cudaError_t launch_band_narrow(const DevOperator<T>& op, int32_t p, int32_t wmax, const T* in, int64_t ldi, T* out,
                               int64_t ldo, const T* base, int64_t ldb, int32_t nrhs, cudaStream_t st) {
    for (int32_t c = 0; c < nrhs; c += kNMaxR<T>) {
        const T* bs = base ? base + c * ldb : nullptr;
        const T* ic = in + c * ldi;
        T* oc = out + c * ldo;
        cudaError_t e = cudaSuccess;
        const int nr = std::min(kNMaxR<T>, nrhs - c);
        if (nr == 1) e = narrow_launch<T, 1>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
        else if (nr == 2) e = narrow_launch<T, 2>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
        else if (nr == 3) e = narrow_launch<T, 3>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
        else if (nr == 4) e = narrow_launch<T, 4>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
        else if constexpr (sizeof(T) == 4) {
            if (nr == 5) e = narrow_launch<T, 5>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
            else if (nr == 6) e = narrow_launch<T, 6>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
            else if (nr == 7) e = narrow_launch<T, 7>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
            else e = narrow_launch<T, 8>(op, p, wmax, ic, ldi, oc, ldo, bs, ldb, st);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template cudaError_t launch_band_narrow<float>(const DevOperator<float>&, int32_t, int32_t, const float*, int64_t,
                                               float*, int64_t, const float*, int64_t, int32_t, cudaStream_t);
template cudaError_t launch_band_narrow<double>(const DevOperator<double>&, int32_t, int32_t, const double*, int64_t,
                                                double*, int64_t, const double*, int64_t, int32_t, cudaStream_t);

}  // namespace slr
