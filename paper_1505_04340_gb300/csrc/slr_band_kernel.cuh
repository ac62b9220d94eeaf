// The band-solve kernel K1 and its launch helpers, shared by the translation
// units that instantiate its 512- and 256-thread variants (slr_band.cu,
// slr_band_half.cu); the layout and pipeline are described in slr_band.cu.
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <mutex>
#include <type_traits>

#include "slr_device.h"

namespace cg = cooperative_groups;

namespace slr {

namespace {

constexpr int kMaxBuf = 8;         // ring slots of a warp at most
constexpr int kMinBuf = 2;         // ring slots of a warp at least
constexpr int kDefBuf = 2;         // unless the operator asks for another count
constexpr int kMaxCq = 16;         // quads per slot at most
// Shared memory a CTA may use: the opt-in maximum for 512-thread CTAs (one per
// SM); for 256-thread CTAs, half an SM's 228 KB less its per-CTA reserve, so
// two CTAs (two subdomains) share each SM.
inline size_t band_cap(int nt) { return nt == 512 ? 227 * 1024 : 112 * 1024; }
constexpr int kRB = 8;             // row blocks of 32: at most 256 rows per slice
constexpr long long kSpin = 1ll << 24;   // bounded mbarrier wait (about a second)

// ---- slice geometry (the host packer uses the same rules: band_* in slr_internal.h)
// local row block with first plane row R0: columns it meets in an upper block
// start at seg_cU0, in a lower block end before seg_cL1
__device__ __forceinline__ int seg_cU0(int W, int R0) { return min(W, R0); }
__device__ __forceinline__ int seg_cL1(int W, int R0) { return min(W, min(R0 + 31, W - 1) + 1); }

// ---- mbarrier / bulk copy PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Bulk copy to shared memory with an L2 policy.  A factor larger than kL2Keep is read once per pass and gone
// from L2 before the next one, so its lines are the first to leave and the vectors, which
// the pass reads again, stay (FV 1024^2 FP32, a 378 MB factor: an apply takes 417 us with
// the policy, 447 without); a factor that L2 can hold keeps the normal policy.
constexpr int64_t kL2Keep = 64ll << 20;
__device__ __forceinline__ uint64_t policy_stream(bool once) {
    uint64_t p;
    if (once) asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    else asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}
// Wait with acquire at cluster scope: the bytes it waits for were stored by
// peers with st.async, whose complete_tx releases at cluster scope.
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Address of the same shared-memory location in cluster CTA `rank`.
__device__ __forceinline__ uint32_t peer_addr(uint32_t a, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
// Store one value into another cluster CTA's shared memory; its bytes complete
// on that CTA's mbarrier `bar` (both addresses in the shared::cluster window, in
// the same CTA, which must not be the executing one).
__device__ __forceinline__ void st_async(uint32_t addr, float v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr),
                 "r"(__float_as_uint(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_async(uint32_t addr, double v, uint32_t bar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr),
                 "l"(__double_as_longlong(v)), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

template <int G>
__device__ __forceinline__ void cluster_barrier() {
    if constexpr (G > 1) {
        cg::this_cluster().sync();
    } else {
        __syncthreads();
    }
}

// Block types: 0 O_J (upper, fwd), 1 D_J (lower, fwd), 2 O_J^T (lower, bwd), 3 D_J^T (upper, bwd).
// Stream order: forward D_0, (O_J, D_J) J = 1..c-1; backward D_{c-1}^T, then
// (O_{J+1}^T, D_J^T) J = c-2..0 (O_{J+1}^T is stored with plane J+1).
// next_block advances (type, plane) along that order; plane < 0 ends it.
__device__ __forceinline__ void next_block(int c, int& type, int& plane) {
    switch (type) {
        case 1: if (plane + 1 < c) { type = 0; ++plane; } else { type = 3; plane = c - 1; } break;
        case 0: type = 1; break;
        case 3: if (plane > 0) type = 2; else plane = -1; break;
        default: type = 3; --plane; break;
    }
}

// bytes of the barriers and tables at the start of a CTA's shared memory
__host__ __device__ inline int band_head_bytes(int nt) {
    return (nt / 32 * kMaxBuf * 8 + 4 * 8 + kRB * 4 + 2 * kRB * 8 + 127) / 128 * 128;
}

// N consecutive values from shared memory, as wide as they allow (p aligned to
// min(16, N sizeof(T)) bytes)
template <typename T, int N>
__device__ __forceinline__ void ld_vec(const T* p, T (&v)[N]) {
    if constexpr (sizeof(T) == 4 && N % 4 == 0) {
#pragma unroll
        for (int q = 0; q < N; q += 4) {
            const float4 a = *reinterpret_cast<const float4*>(p + q);
            v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
        }
    } else if constexpr (sizeof(T) == 8 && N % 2 == 0) {
#pragma unroll
        for (int q = 0; q < N; q += 2) {
            const double2 a = *reinterpret_cast<const double2*>(p + q);
            v[q] = a.x; v[q + 1] = a.y;
        }
    } else {
#pragma unroll
        for (int q = 0; q < N; ++q) v[q] = p[q];
    }
}

}  // namespace

// NT threads per CTA: 512 (one CTA per SM, 4 warps per SM sub-partition) or 256
// (two CTAs, two subdomains, per SM).  nr <= NR right-hand sides.
//
// What bounds it is the chain of 4 c - 2 blocks (c planes); per block the slice's
// bytes, FP64's multiply-adds (its pipe takes a warp's in about 17 cycles) and
// the fixed cost of a step: products, one CTA barrier, the rows' sums, the exchange.
// So a warp's part of a block is a plain run over its quads, with a branch only where
// its row block changes.
template <typename T, int NR, int G, int NT>
__global__ void __launch_bounds__(NT, 512 / NT)
k_band_wide(const BandBlock* __restrict__ blocks, const T* __restrict__ fac, const T* in, int64_t ldi, T* out,
            int64_t ldo, const T* base, int64_t ldb, int32_t* err, int nr, int nbuf, int cq, int once) {
    constexpr int kW = NT / 32;                           // warps per CTA
    constexpr int NIT = (kRB * NR + kW - 1) / kW;         // (row block, right-hand side) pairs a warp owns
    extern __shared__ __align__(128) unsigned char smem[];
    const int sub = blockIdx.x / G;
    const int g = (G > 1) ? (int)cg::this_cluster().block_rank() : 0;
    const BandBlock& b = blocks[sub];
    const int W = b.w, c = b.c, m = b.m, WP = (W + 3) & ~3;
    if (m == 0) {                               // uniform across the cluster
        dep_wait();
        return;
    }
    const int SU = b.SU, SL = b.SL, row0 = b.row0, nrb = b.nrb[g];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // ---- shared memory carve-up: barriers, tables and vectors, then the rings
    uint64_t* full = reinterpret_cast<uint64_t*>(smem) + warp * kMaxBuf;   // [kW][kMaxBuf]
    uint64_t* vbar = reinterpret_cast<uint64_t*>(smem) + kW * kMaxBuf;      // [3] t (two buffers), y/x
    volatile int* abort_flag = reinterpret_cast<volatile int*>(vbar + 3);
    volatile unsigned* dest = reinterpret_cast<volatile unsigned*>(abort_flag + 1);   // CTAs this one sends to
    int* R0s = reinterpret_cast<int*>(vbar + 4);                            // [kRB] first row of each row block
    int2* pw = reinterpret_cast<int2*>(R0s + kRB);                          // [2][kRB] first and last warp of a row
                                                                            // block (upper, lower)
    T* vst = reinterpret_cast<T*>(smem + band_head_bytes(NT));              // [WP][NR] y_{J-1} / x_{J+1}, whole plane
    T* vt = vst + NR * WP;                          // [2][WP][NR] t, whole plane, by phase parity
    T* part = vt + 2 * NR * WP;                     // [kW + kRB][NR][32] pieces
    const int slot = cq * 128;                      // elements
    uintptr_t rp = (reinterpret_cast<uintptr_t>(part + (kW + kRB) * NR * 32) + 127) & ~uintptr_t(127);
    T* ring = reinterpret_cast<T*>(rp) + (size_t)warp * nbuf * slot;

    const int64_t PS = (int64_t)G * 2 * (SU + SL);
    const T* facg = fac + b.foff + (int64_t)g * 2 * (SU + SL);
    // Every row of a plane has one owner in the cluster.  A phase of a vector
    // barrier completes with 1 + narr arrivals (thread 0 arming it, and each warp
    // that owns rows once they are stored here) and the bytes of the other
    // slices' rows, stored by their owners with st.async.
    int my_rows = 0;
    for (int rb = 0; rb < nrb; ++rb) my_rows += min(32, W - 32 * b.rbmap[g][rb]);
    const uint32_t rbytes = (uint32_t)((W - my_rows) * nr * (int)sizeof(T));
    const int narr = min(kW, nrb * nr);

    // this warp's share of an upper (0) and a lower (1) block: first quad of the slice's
    // block, quads, and the first quad's row block and column
    int sq0[2], snq[2], srb[2], scol[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        auto quads = [&](int rb) {
            const int r0 = 32 * b.rbmap[g][rb];
            return ((t == 0 ? W - seg_cU0(W, r0) : seg_cL1(W, r0)) + 3) >> 2;
        };
        int Q = 0;
        for (int rb = 0; rb < nrb; ++rb) Q += quads(rb);
        // (with fewer quads than warps, one each: every share before the last is non-empty)
        const int ew = min(kW, Q);
        sq0[t] = warp < ew ? Q * warp / ew : Q;
        snq[t] = warp < ew ? Q * (warp + 1) / ew - sq0[t] : 0;
        srb[t] = scol[t] = 0;
        int q = 0;
        for (int rb = 0; rb < nrb; ++rb) {
            const int n = quads(rb);
            if (tid == 0) pw[t * kRB + rb] = make_int2(((q + 1) * ew - 1) / Q, ((q + n) * ew - 1) / Q);
            if (sq0[t] >= q && sq0[t] < q + n) {
                srb[t] = rb;
                scol[t] = 4 * (sq0[t] - q) + (t == 0 ? seg_cU0(W, 32 * b.rbmap[g][rb]) : 0);
            }
            q += n;
        }
    }
    if (tid < nrb) R0s[tid] = 32 * b.rbmap[g][tid];
    if (lane == 0)
        for (int i = 0; i < nbuf; ++i) mbar_init(&full[i], 1);
    if (tid == 0) {
        *abort_flag = 0;                                  // set once a bounded wait of this CTA expires
        unsigned peers = 0;                               // the others that own rows
        for (int pr = 0; pr < G; ++pr)
            if (pr != g && b.nrb[pr] > 0) peers |= 1u << pr;
        *dest = peers;
        for (int i = 0; i < 3; ++i) mbar_init(&vbar[i], 1 + narr);
        for (int i = 0; i < 3; ++i) {
            if (rbytes) mbar_arrive_expect_tx(&vbar[i], rbytes);
            else mbar_arrive(&vbar[i]);
        }
    }
    if (lane == 0) fence_mbar_init();
    // the vectors' entries past W and past nr stay zero
    for (int i = tid; i < 3 * NR * WP; i += NT) vst[i] = T(0);
    __syncthreads();

    // lane 0 of a warp issues the copies of its share in stream order, cq quads at most each
    int itype = 1, iplane = 0, iq = 0, issued = 0, islot = 0;   // next copy: block, first quad; its slot
    const uint64_t pol = policy_stream(once != 0);
    auto issue_next = [&]() {
        // (a warp may have a share of one block type only)
        while (iplane >= 0 && ((itype == 0 || itype == 3) ? snq[0] : snq[1]) == 0) next_block(c, itype, iplane);
        if (iplane < 0) return;
        const bool up = itype == 0 || itype == 3;
        const int n = min(cq, (up ? snq[0] : snq[1]) - iq);
        const int64_t off = (int64_t)iplane * PS +
                            (itype == 0 ? 0 : itype == 1 ? SU : itype == 2 ? SU + SL : SU + 2 * SL);
        const uint32_t bytes = (uint32_t)(n * 128 * (int)sizeof(T));
        mbar_arrive_expect_tx(&full[islot], bytes);
        bulk_g2s(ring + (size_t)islot * slot, facg + off + ((up ? sq0[0] : sq0[1]) + iq) * 128, bytes,
                     &full[islot], pol);
        ++issued;
        iq += n;
        if (iq == (up ? snq[0] : snq[1])) {
            iq = 0;
            next_block(c, itype, iplane);
        }
        if (++islot == nbuf) islot = 0;
    };
    // After a bounded wait expires the CTA aborts: the status word and the
    // CTA's abort flag are set, no further copy is issued, and before it exits each
    // warp waits for the copies it issued.  The CTA goes through the rest of its steps
    // with whatever its buffers hold (no wait is taken again).
    auto fail = [&]() {
        atomicExch(err, 1);
        *dest = 0;
        *abort_flag = 1;
    };
    int kslot = 0;                                        // slot and parity of the next copy to read
    uint32_t kpar = 0;
    auto wait_full = [&]() {
        long long it = 0;
        while (!mbar_try_wait(&full[kslot], kpar)) {
            if (++it > kSpin || *abort_flag) {
                fail();
                break;
            }
        }
        __syncwarp();
    };
    // the warp has read its slot: lane 0 refills it (nothing is issued after an abort: a
    // copy whose wait expired may still be in flight)
    auto next_slot = [&]() {
        __syncwarp();
        if (lane == 0 && iplane >= 0 && !*abort_flag) {
            fence_proxy_async();
            issue_next();
        }
        if (++kslot == nbuf) {
            kslot = 0;
            kpar ^= 1;
        }
    };
    // at exit after an abort: the last copy issued into each slot has landed
    auto drain = [&]() {
        if (lane != 0 || !*abort_flag) return;
        for (int sl = 0; sl < nbuf && sl < issued; ++sl) {
            const int last = sl + ((issued - 1 - sl) / nbuf) * nbuf;
            long long it = 0;
            while (!mbar_try_wait(&full[sl], (uint32_t)((last / nbuf) & 1)) && ++it <= kSpin) {
            }
        }
    };
    // The plane vector of a phase reaches every CTA of the cluster: each owner
    // stores its rows into this CTA's copy (then its warp arrives on the local
    // vector barrier) and, by st.async, into every peer's copy, where the bytes
    // complete on the peer's vector barrier, armed by the peer's thread 0 with
    // the bytes it receives.  No cluster-wide barrier is taken per phase.  A CTA re-arms a barrier for
    // its next phase as soon as it has seen the current one complete: the next
    // phase's stores into it come only after the peers have received this CTA's
    // own next rows, which it sends after consuming the current phase.  For the
    // same reason the t vector has two buffers (by phase parity): the forward
    // pass's last t and the backward pass's first t have no exchange of y
    // between them, so a fast peer can send the second before a slow CTA has
    // read the first.  y/x needs one buffer (an exchange of t always lies between
    // two of its phases).  A slice without rows (planes of fewer than G row blocks,
    // or of few more, where the assignment leaves one out) sends nothing that could hold its peers back: with their next bytes in a phase
    // it has yet to arm, the phase's count never comes to zero.  So it takes no part: its peers
    // send it nothing and it waits for nothing.  After a wait that expired the barrier
    // is left un-armed (thread 0 never arrives twice in one phase).
    auto wait_vec = [&](uint64_t* bar, uint32_t par) {
        long long it = 0;
        bool ok = true;
        while (!mbar_try_wait_cluster(bar, par)) {
            if (++it > kSpin || *abort_flag) {
                fail();
                ok = false;
                break;
            }
        }
        if (ok && tid == 0) {
            if (rbytes) mbar_arrive_expect_tx(bar, rbytes);
            else mbar_arrive(bar);
        }
        __syncwarp();
    };
    // The peers that a phase's rows go to: a word in shared memory, read once per phase (in a register
    // it cost the eight-column kernel, which spills, 4%).  An aborted CTA sends nothing more: its
    // peers' waits for its rows then expire and they abort in turn, so at most a phase or two of
    // bytes reach a barrier this CTA no longer arms.
    auto targets = [&]() -> unsigned { return G > 1 ? *dest : 0u; };
    // entry (r, j) of a phase's vector vec into every CTA that owns rows (to: targets())
    auto send = [&](T* vec, uint64_t* bar, unsigned to, int j, int r, T v) {
        vec[r * NR + j] = v;
        if constexpr (G > 1) {
            const uint32_t a = smem_u32(vec + r * NR + j), mb = smem_u32(bar);
#pragma unroll
            for (int pr = 0; pr < G; ++pr)
                if (to & (1u << pr)) st_async(peer_addr(a, pr), v, peer_addr(mb, pr));
        }
    };
    // an owner warp, once all its rows of a phase are stored here (all of its lanes)
    auto arrive_local = [&](uint64_t* bar) {
        if (warp < narr) {
            __syncwarp();
            if (lane == 0 && !*abort_flag) mbar_arrive(bar);
        }
    };

    if (lane == 0)
        while (issued < nbuf && iplane >= 0) issue_next();
    dep_wait();                                          // (the copies so far are of the factor)
    // every CTA of the cluster has armed its barriers before any st.async reaches it
    cluster_barrier<G>();
    if (G > 1 && nrb == 0) {                             // (no copy issued either: it has no quads)
        cluster_barrier<G>();
        return;
    }

    // One block: this warp's share times the vector vin (complete once phase `par` of
    // vector barrier `vb` has), its pieces to `part`.
    auto run_block = [&](auto up, const T* vin, uint64_t* vb, uint32_t par) {
        constexpr bool UP = decltype(up)::value;
        constexpr int ST = UP ? 0 : 1;
        int n = snq[ST], rb = srb[ST], col = scol[ST];
        wait_vec(vb, par);
        T acc[NR], ac2[NR];
#pragma unroll
        for (int j = 0; j < NR; ++j) acc[j] = ac2[j] = T(0);
        int left = n > 0 ? ((UP ? W : seg_cL1(W, R0s[rb])) - col + 3) >> 2 : 0;   // quads of the row block
        const T* V = vin + col * NR;
        while (n > 0) {
            wait_full();
            const T* P = ring + (size_t)kslot * slot + lane * 4;
            int nc = min(cq, n);
            n -= nc;
            while (true) {
                const int t = min(nc, left);
#pragma unroll 2
                for (int i = 0; i < t; ++i) {
                    T a[4];
                    ld_vec<T, 4>(P, a);
                    // two chains per right-hand side: even and odd columns
                    constexpr int U = NR < 4 ? 4 / NR : 1;   // columns per load of the vector
#pragma unroll
                    for (int u = 0; u < 4; u += U) {
                        T v[U * NR];
                        ld_vec<T, U * NR>(V + u * NR, v);
#pragma unroll
                        for (int w = 0; w < U; ++w)
#pragma unroll
                            for (int j = 0; j < NR; ++j)
                                if (NR <= 3 || j < nr) {
                                    T& s = ((u + w) & 1) ? ac2[j] : acc[j];
                                    s = fma(a[u + w], v[w * NR + j], s);
                                }
                    }
                    P += 128;
                    V += 4 * NR;
                }
                nc -= t;
                left -= t;
                if (left > 0) break;                       // the copy is used up
                // end of the row block: its piece
                T* pp = part + (size_t)(warp + rb) * NR * 32 + lane;
#pragma unroll
                for (int j = 0; j < NR; ++j) {
                    pp[j * 32] = acc[j] + ac2[j];
                    acc[j] = ac2[j] = T(0);
                }
                if (nc + n == 0) break;                    // end of the share
                ++rb;
                const int r0 = R0s[rb], c0 = UP ? r0 : 0;
                V = vin + c0 * NR;
                left = ((UP ? W - r0 : seg_cL1(W, r0)) + 3) >> 2;
                if (nc == 0) break;
            }
            next_slot();
        }
        if (left > 0) {                                    // the share ends inside a row block
            T* pp = part + (size_t)(warp + rb) * NR * 32 + lane;
#pragma unroll
            for (int j = 0; j < NR; ++j) pp[j * 32] = acc[j] + ac2[j];
        }
        __syncthreads();
    };
    const std::true_type upper{};
    const std::false_type lower{};

    // The warp's (row block, right-hand side) pairs: warp, warp + kW, ...; a lane owns a
    // row of each.  Its right-hand side (forward) or forward result (backward) is
    // loaded before the block product so the load is off the plane-to-plane chain.
    int orow[NIT], oj[NIT], op[NIT], on[NIT][2];         // row, column, first piece per block type, pieces
    bool own[NIT];
#pragma unroll
    for (int it = 0; it < NIT; ++it) {
        const int k = warp + kW * it;
        own[it] = k < nrb * nr;
        const int rb = own[it] ? k % nrb : 0;
        oj[it] = own[it] ? k / nrb : 0;
        orow[it] = (own[it] ? R0s[rb] : 0) + lane;
        const int2 u = own[it] ? pw[rb] : make_int2(0, 0), l = own[it] ? pw[kRB + rb] : make_int2(0, 0);
        op[it] = ((u.x + rb) << 16) | (l.x + rb);
        on[it][0] = u.y - u.x;
        on[it][1] = l.y - l.x;
        own[it] = own[it] && orow[it] < W;
    }
    // the sum of a row's pieces of an upper (t = 0) or lower (t = 1) block
    auto psum = [&](int t, int it) -> T {
        const T* p = part + ((t == 0 ? op[it] >> 16 : op[it] & 0xffff) * NR + oj[it]) * 32 + lane;
        T s = p[0];
#pragma unroll 4
        for (int w = on[it][t]; w > 0; --w) {
            p += NR * 32;
            s += *p;
        }
        return s;
    };
    int ut = 0, uy = 0;        // phases of the t vector and of the y/x vector so far
    // =================================================================== forward
    for (int J = 0; J < c; ++J) {
        T pre[NIT];
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
            const int row = J * W + orow[it];
            pre[it] = (own[it] && row < m) ? in[row0 + row + oj[it] * ldi] : T(0);
        }
        if (J > 0) run_block(upper, vst, &vbar[2], (uint32_t)(uy++ & 1));           // O_J y_{J-1}
        T* vtb = vt + (ut & 1) * NR * WP;
        unsigned to = targets();
#pragma unroll
        for (int it = 0; it < NIT; ++it)
            if (own[it]) send(vtb, &vbar[ut & 1], to, oj[it], orow[it], J > 0 ? pre[it] - psum(0, it) : pre[it]);
        arrive_local(&vbar[ut & 1]);
        run_block(lower, vtb, &vbar[ut & 1], (uint32_t)((ut >> 1) & 1));           // D_J t
        ++ut;
        to = targets();
#pragma unroll
        for (int it = 0; it < NIT; ++it)
            if (own[it]) {
                const T y = psum(1, it);
                if (J + 1 < c) send(vst, &vbar[2], to, oj[it], orow[it], y);             // read by O_{J+1}
                const int row = J * W + orow[it];
                if (row < m) out[row0 + row + oj[it] * ldo] = y;
            }
        if (J + 1 < c) arrive_local(&vbar[2]);
    }
    // =================================================================== backward
    for (int J = c - 1; J >= 0; --J) {
        T pre[NIT], bs[NIT];
#pragma unroll
        for (int it = 0; it < NIT; ++it) {
            const int row = J * W + orow[it];
            const bool has = own[it] && row < m;
            pre[it] = has ? out[row0 + row + oj[it] * ldo] : T(0);
            bs[it] = (has && base) ? base[row0 + row + oj[it] * ldb] : T(0);
        }
        if (J < c - 1) run_block(lower, vst, &vbar[2], (uint32_t)(uy++ & 1));       // O_{J+1}^T x_{J+1}
        T* vtb = vt + (ut & 1) * NR * WP;
        unsigned to = targets();
#pragma unroll
        for (int it = 0; it < NIT; ++it)
            if (own[it]) send(vtb, &vbar[ut & 1], to, oj[it], orow[it], J < c - 1 ? pre[it] - psum(1, it) : pre[it]);
        arrive_local(&vbar[ut & 1]);
        run_block(upper, vtb, &vbar[ut & 1], (uint32_t)((ut >> 1) & 1));           // D_J^T t
        ++ut;
        to = targets();
#pragma unroll
        for (int it = 0; it < NIT; ++it)
            if (own[it]) {
                const T x = psum(0, it);
                if (J > 0) send(vst, &vbar[2], to, oj[it], orow[it], x);                  // read by O_J^T
                const int row = J * W + orow[it];
                if (row < m) out[row0 + row + oj[it] * ldo] = base ? bs[it] - x : x;
            }
        if (J > 0) arrive_local(&vbar[2]);
    }
    cluster_barrier<G>();    // no CTA leaves while a peer may still store into it
    drain();                 // nor with a bulk copy still writing its shared memory
}

// Shared memory besides the rings (barriers, tables, vectors, pieces, the rings'
// alignment), for planes of at most wmax rows.
inline size_t band_fixed_bytes(int32_t wmax, int32_t nr, size_t elem, int nt) {
    const size_t wp = (size_t)(wmax + 3) / 4 * 4;
    return band_head_bytes(nt) + (3 * nr * wp + (size_t)(nt / 32 + kRB) * nr * 32) * elem + 128;
}

// The ring of a warp of a CTA of nt threads: the slot count (nbuf_req, 0 for the default,
// clamped to what fits) and the quads per slot that fill the shared memory left
// beside the tables and vectors; false if no ring fits.  Two slots: larger copies measured
// faster than more of them (16^3 boxes, one column: FP32 103 us with two, 115 with three, 127
// with four; FP64 362, 378, 375).
inline bool band_ring(int32_t wmax, int32_t nr, size_t elem, int32_t nbuf_req, int nt, int32_t* nbuf, int32_t* cq) {
    const size_t fx = band_fixed_bytes(wmax, nr, elem, nt), cap = band_cap(nt);
    const size_t qb = 128 * elem;                                  // bytes of a quad
    if (fx + (size_t)(nt / 32) * kMinBuf * qb > cap) return false;
    const int32_t avail = (int32_t)((cap - fx) / (nt / 32) / qb);  // quads a warp's ring can hold
    int32_t n = nbuf_req > 0 ? nbuf_req : kDefBuf;
    n = std::max(kMinBuf, std::min<int32_t>(n, kMaxBuf));
    n = std::min(n, avail);
    *nbuf = n;
    *cq = std::min(avail / n, kMaxCq);
    return true;
}

inline size_t band_smem_bytes(int32_t wmax, int32_t nr, size_t elem, int nt, int32_t nbuf, int32_t cq) {
    return band_fixed_bytes(wmax, nr, elem, nt) + (size_t)(nt / 32) * nbuf * cq * 128 * elem;
}

namespace {
template <typename T, int NR, int G, int NT>
cudaError_t band_launch(const DevOperator<T>& op, int32_t p, int32_t wmax, const T* in, int64_t ldi, T* out,
                        int64_t ldo, const T* base, int64_t ldb, int nr, cudaStream_t st) {
    auto kern = k_band_wide<T, NR, G, NT>;
    // The dynamic shared-memory limit of a kernel is process-wide state on its
    // device.  It is raised once, to the device's opt-in maximum, so that
    // threads launching this kernel for operators of different widths never
    // race between one thread's setting and another's launch.
    static std::mutex mu;
    static uint64_t raised = 0;                     // bit d: done on device d
    {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
        std::lock_guard<std::mutex> lk(mu);
        if (!(raised >> dev & 1)) {
            int optin = 0;
            e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
            if (e != cudaSuccess) return e;
            raised |= 1ull << dev;
        }
    }
    int32_t nbuf = 0, cq = 0;
    if (!band_ring(wmax, NR, sizeof(T), op.band_nbuf, NT, &nbuf, &cq)) return cudaErrorInvalidValue;
    const size_t smem = band_smem_bytes(wmax, NR, sizeof(T), NT, nbuf, cq);
    cudaError_t e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p * G);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    int na = G > 1 ? 1 : 0;
    if (dep_active()) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na++].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    e = cudaLaunchKernelEx(&cfg, kern, op.band, op.bfac, in, ldi, out, ldo, base, ldb, op.err, nr, (int)nbuf, (int)cq, op.bfac_len * (int64_t)sizeof(T) > kL2Keep ? 1 : 0);
    count_launches(1);
    return e;
}

template <typename T, int NR, int NT>
cudaError_t band_launch_g(const DevOperator<T>& op, int32_t p, int32_t wmax, const T* in, int64_t ldi, T* out,
                          int64_t ldo, const T* base, int64_t ldb, int nr, cudaStream_t st) {
    switch (op.band_G) {
        case 2: return band_launch<T, NR, 2, NT>(op, p, wmax, in, ldi, out, ldo, base, ldb, nr, st);
        case 4: return band_launch<T, NR, 4, NT>(op, p, wmax, in, ldi, out, ldo, base, ldb, nr, st);
        default: return band_launch<T, NR, 1, NT>(op, p, wmax, in, ldi, out, ldo, base, ldb, nr, st);
    }
}
}  // namespace

// The 256-thread variants (instantiated in their own translation unit).
template <typename T, int NR>
cudaError_t band_launch_half(const DevOperator<T>& op, int32_t p, int32_t wmax, const T* in, int64_t ldi, T* out,
                             int64_t ldo, const T* base, int64_t ldb, int nr, cudaStream_t st);


}  // namespace slr
