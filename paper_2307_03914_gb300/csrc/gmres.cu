// gmres.cu -- left-preconditioned MGS-GMRES and the refinement loop of Alg 3.1.
//
// A small system with short rows runs all its Arnoldi steps in one launch
// (k_gmres_coop).  Otherwise, per step j (the "hot loop" of the method), three
// launches run on the solve's stream, with no host synchronisation between steps:
//   w = A v_j               (u_p, SELL SpMV)                       spmv.cu
//   z = M w -> V(:, j+1)    (Alg 2.3 bucketed SpMV, stored in u_g) spmv.cu
//   k_mgs                   (cooperative, persistent)              this file
// The Krylov index j and the "done" flag live in device memory (GmresState);
// every kernel of a step reads them, so the host enqueues steps in chunks and
// only reads the flag between chunks.  Steps enqueued after convergence
// return immediately.
//
// The MGS kernels keep one contiguous range of rows per block and take the basis
// in groups of a few vectors, one grid-wide reduction per group (mgs.cuh): the
// partial sums v_t . z of a group's vectors, then z -= sum h_t v_t.  Every block
// adds the partials in the same fixed order, so all blocks hold the same h_ij
// (deterministic, no atomics).  The last pass forms ||z||_2 and normalises
// v_{j+1}; the Givens rotations (fp64) and the test |g_{j+1}| <= tau ||M r||_2
// follow.  Every wait is bounded in time (BSPAI_TIMEOUT).
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "mgs.cuh"
#include "spmv_row.cuh"
#include "tags.cuh"

namespace bspai {

__global__ void k_state_init(GmresState* st, int kmax, double tau, double target) {
    st->j = 0;
    st->done = 0;
    st->status = BSPAI_OK;
    st->kmax = kmax;
    st->beta = 0.0;
    st->tau = tau;
    st->target = target;
    st->res = 0.0;
    st->hlast = 0.0;
    st->bar.count = 0;
    st->bar.err = 0;
}

__device__ __forceinline__ void block_rows(int n, int G, int64_t& r0, int64_t& r1) {
    int64_t chunk = ceil_div(ceil_div(n, G), 32) * 32;
    r0 = (int64_t)blockIdx.x * chunk;
    r1 = r0 + chunk < n ? r0 + chunk : n;
}
__device__ __forceinline__ void block_rows(int n, int64_t& r0, int64_t& r1) { block_rows(n, (int)gridDim.x, r0, r1); }

// Sum of `v` over the whole grid, identical in every block: block sum in a
// fixed tree, partials to part[slot*G + block], barrier, then every block adds
// the G partials in the same order.  `ok` is false if the barrier failed.
template <typename T>
__device__ __forceinline__ T grid_sum(T v, T* part, int slot, GridBar* bar, unsigned long long tmo, bool& ok) {
    __shared__ T s_w[32];
    __shared__ T s_tot;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    v = warp_sum(v);
    if (lane == 0) s_w[w] = v;
    __syncthreads();
    if (w == 0) {
        T t = lane < nw ? s_w[lane] : T(0);
        t = warp_sum(t);
        if (lane == 0) part[(int64_t)slot * gridDim.x + blockIdx.x] = t;
    }
    ok = grid_sync(bar, tmo);
    if (!ok) return T(0);
    if (w == 0) {
        T t = T(0);
        for (int b = lane; b < (int)gridDim.x; b += 32)
            t = Ar<T>::add(t, *(volatile T*)&part[(int64_t)slot * gridDim.x + b]);
        t = warp_sum(t);
        if (lane == 0) s_tot = t;
    }
    __syncthreads();
    return s_tot;
}

// beta = ||s||_2 of V(:, 0) = s = M r, then v_0 = s / beta and g_0 = beta
template <typename T>
__global__ void __launch_bounds__(512) k_gmres_start(T* __restrict__ V, int n, GmresState* st, double* g, T* part,
                                                     unsigned long long tmo) {
    int64_t r0, r1;
    block_rows(n, r0, r1);
    T acc = T(0);
    for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) acc = Ar<T>::add(acc, Ar<T>::mul(V[r], V[r]));
    bool ok;
    const T tot = grid_sum(acc, part, 0, &st->bar, tmo, ok);
    if (!ok) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            st->status = BSPAI_TIMEOUT;
            st->done = 1;
        }
        return;
    }
    const T beta = Ar<T>::sqrt(tot);
    const bool fin = isfinite((double)beta);
    if (beta > T(0) && fin)
        for (int64_t r = r0 + threadIdx.x; r < r1; r += blockDim.x) V[r] = Ar<T>::div(V[r], beta);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->beta = (double)beta;
        st->res = (double)beta;
        g[0] = (double)beta;
        st->done = !(beta > T(0)) || !fin;
        if (!fin) st->status = BSPAI_NONFINITE;
    }
}

// MGS step of the orders whose rows do not fit on chip: the group's vectors and z
// are streamed from memory.  Pass g takes the previous group out of z and forms
// the products with the next group in one sweep, so a group of four costs ten
// vector streams (four of each group, z read and written) where one vector at a
// time costs sixteen.
// (fp64 keeps one block per SM: the grid, which k_gmres_start shares, fixes the
// order in which ||M r||_2 is summed.)
constexpr int kStreamGB = 4;
// One sweep of a pass over the block's rows: HAVE vectors from Vp (coefficients hp) out of z,
// then the products with CNT vectors from Vc, and for the last group (last) the Gram entries
// of its last vector; CNT = 0: ||z||^2 into a[0].  The counts are constants: no operation is
// spent on a vector that is not there, and the loads of RT rows are issued ahead of the store
// that they could not pass.  One loop for every count, a row at a time -> this, us in this
// kernel: n = 30,000 in fp64 on one SM, the first step 284 (one vector at a time: 223) -> 168;
// n = 4,000,001 in fp32, the first step 73 (49) -> 49, 30 steps 5,290 (8,254) -> 4,240.
template <typename T, int HAVE, int CNT>
__device__ __forceinline__ void stream_sweep(const T* Vp, const T* Vc, int64_t ldv, T* z, int64_t r0, int64_t r1,
                                             bool last, const T (&hp)[kStreamGB], T (&a)[kStreamGB],
                                             T (&q)[kStreamGB]) {
    constexpr int RT = HAVE + CNT <= 2 ? 4 : 2;
    const int64_t bd = blockDim.x;
    for (int64_t rb = r0 + threadIdx.x; rb < r1; rb += RT * bd) {
        T zr[RT], pv[RT][HAVE ? HAVE : 1], v[RT][CNT ? CNT : 1];
#pragma unroll
        for (int u = 0; u < RT; ++u) {
            const int64_t r = rb + u * bd;
            const bool in = r < r1;
            zr[u] = in ? z[r] : T(0);
#pragma unroll
            for (int t = 0; t < HAVE; ++t) pv[u][t] = in ? Vp[(int64_t)t * ldv + r] : T(0);
#pragma unroll
            for (int t = 0; t < CNT; ++t) v[u][t] = in ? Vc[(int64_t)t * ldv + r] : T(0);
        }
#pragma unroll
        for (int u = 0; u < RT; ++u) {
            if (rb + u * bd >= r1) break;
            if constexpr (HAVE > 0) {
#pragma unroll
                for (int t = 0; t < HAVE; ++t) zr[u] = pk_nfma(hp[t], pv[u][t], zr[u]);
                z[rb + u * bd] = zr[u];
            }
            if constexpr (CNT == 0) {
                a[0] = Ar<T>::fma(zr[u], zr[u], a[0]);
            } else {
#pragma unroll
                for (int t = 0; t < CNT; ++t) a[t] = Ar<T>::fma(v[u][t], zr[u], a[t]);
                if (last)
#pragma unroll
                    for (int t = 0; t < CNT - 1; ++t) q[t] = Ar<T>::fma(v[u][t], v[u][CNT - 1], q[t]);
            }
        }
    }
}
template <typename T>
__global__ void __launch_bounds__(512, sizeof(T) == 8 ? 1 : 2) k_mgs(T* __restrict__ V, int64_t ldv, int n, GmresState* st, double* H,
                                             double* cs, double* sn, double* g, T* part, T* tri,
                                             unsigned long long* hq, unsigned long long tmo) {
    constexpr int GB = kStreamGB;
    __shared__ int s_j, s_done, s_kmax;
    __shared__ unsigned s_seq;
    __shared__ T s_w[2 * GB][32], s_tot[2 * GB], s_h[GB], s_tri[GB][GB];
    __shared__ GivensBatch s_giv;
    if (threadIdx.x == 0) {
        s_j = st->j;
        s_done = st->done;
        s_kmax = st->kmax;
        s_seq = *(volatile unsigned*)&st->bar.seq;
    }
    __syncthreads();
    if (s_done) return;
    const int j = s_j, kmax = s_kmax;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned tag = s_seq + 1u;
    int64_t r0, r1;
    block_rows(n, r0, r1);
    T* z = V + (int64_t)(j + 1) * ldv;
    const int ng = j / GB + 1;
    T hp[GB];
#pragma unroll
    for (int t = 0; t < GB; ++t) hp[t] = T(0);
    for (int gi = 0; gi <= ng; ++gi) {  // pass ng: the last group out of z, ||z||^2
        const int i0 = gi * GB;
        const bool last = gi == ng - 1, norm = gi == ng;
        const int cnt = norm ? 0 : last ? j - i0 + 1 : GB;
        const int have = gi > 0 ? (norm ? j + 1 - (i0 - GB) : GB) : 0;  // vectors of the previous group
        T a[GB], q[GB];
#pragma unroll
        for (int t = 0; t < GB; ++t) a[t] = q[t] = T(0);
        const T *Vp = V + (int64_t)(i0 - GB) * ldv, *Vc = V + (int64_t)i0 * ldv;
        static_assert(GB == 4, "the counts below");
        if (norm) {
            if (have == 1) stream_sweep<T, 1, 0>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else if (have == 2) stream_sweep<T, 2, 0>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else if (have == 3) stream_sweep<T, 3, 0>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else stream_sweep<T, 4, 0>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
        } else if (have == 0) {
            if (cnt == 1) stream_sweep<T, 0, 1>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else if (cnt == 2) stream_sweep<T, 0, 2>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else if (cnt == 3) stream_sweep<T, 0, 3>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else stream_sweep<T, 0, 4>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
        } else {
            if (cnt == 1) stream_sweep<T, 4, 1>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else if (cnt == 2) stream_sweep<T, 4, 2>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else if (cnt == 3) stream_sweep<T, 4, 3>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
            else stream_sweep<T, 4, 4>(Vp, Vc, ldv, z, r0, r1, last, hp, a, q);
        }
        warp_multi_sum<GB>(a);
        warp_multi_sum<GB>(q);
        if ((lane & (32 / GB - 1)) == 0) {
            s_w[warp_multi_index<GB>(lane)][w] = a[0];
            s_w[GB + warp_multi_index<GB>(lane)][w] = q[0];
        }
        __syncthreads();
        if (w < 2 * GB) {
            T t = lane < (int)(blockDim.x >> 5) ? s_w[w][lane] : T(0);
            t = warp_sum(t);
            if (lane == 0) part[((int64_t)(gi & 1) * 2 * GB + w) * gridDim.x + blockIdx.x] = t;
        }
        if (!grid_sync(&st->bar, tmo)) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                st->status = BSPAI_TIMEOUT;
                st->done = 1;
            }
            return;
        }
        if (w < 2 * GB) {
            T t = T(0);
            for (int b = lane; b < (int)gridDim.x; b += 32)
                t = Ar<T>::add(t, *(volatile T*)&part[((int64_t)(gi & 1) * 2 * GB + w) * gridDim.x + b]);
            t = warp_sum(t);
            if (lane == 0) s_tot[w] = t;
        }
        __syncthreads();
        if (norm) break;
        if (w == 0) {
            T row[GB];
            group_rows<T, GB>(row, tri + (int64_t)i0 * GB, last ? cnt - 1 : cnt);
            const T h = group_coeff<T, GB>(row, s_tot, cnt, last);
            if (lane < GB) s_h[lane] = lane < cnt ? h : T(0);
            if (blockIdx.x == 0) {
                if (lane < cnt) tag_publish(h, hq + (int64_t)(i0 + lane) * TagWords<T>::W, tag);
                if (last) group_new_row<T, GB>(row, s_tot, s_tri, cnt, tri + (int64_t)j * GB);
            }
        }
        __syncthreads();
#pragma unroll
        for (int t = 0; t < GB; ++t) hp[t] = s_h[t];
    }
    const T hn = Ar<T>::sqrt(s_tot[0]);
    if (hn > T(0) && isfinite((double)hn)) {
        const Quot<T> by(hn);
        for (int64_t rb = r0 + threadIdx.x; rb < r1; rb += 4 * (int64_t)blockDim.x) {
            T x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = rb + u * blockDim.x < r1 ? z[rb + u * blockDim.x] : T(0);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (rb + u * blockDim.x < r1) z[rb + u * blockDim.x] = by(x[u]);
        }
    }
    if (blockIdx.x == 0 && w == 0) {
        if (lane == 0) {
            tag_publish(hn, hq + (int64_t)(j + 1) * TagWords<T>::W, tag);
            st->bar.seq = tag;
        }
        __syncwarp();
        if (!givens_column<T>(s_giv, j, kmax, H, cs, sn, g, st, hq, tag, tmo) && lane == 0) {
            st->status = BSPAI_TIMEOUT;
            st->done = 1;
        }
    }
}

constexpr int kMgsBlocks = 64;  // fewest blocks the on-chip MGS kernel is given
// A block's bytes of one basis vector (at the instance's capacity) from which
// an on-chip MGS instance polls its reductions by bulk copies
// (tag_poll_row_bulk) instead of loads.  Measured (fp32, 64-128 blocks,
// 64-step GMRES runs, one vector per reduction): load polling 5 % faster at
// 4 KB per block (n = 64,000), even at 7 KB; bulk polling 11 / 3 / 4 % faster at
// 16 / 32 / 64 KB (n = 262,144 / 512,000 / 2,097,152); with 9 blocks per solve
// (16 right-hand sides side by side) and 29 KB per block, slower.  Instances
// whose capacity is below the threshold are compiled without the bulk path;
// the others take it when the launch asks.
constexpr int64_t kBulkPollBytes = 16 * 1024;

// The on-chip MGS kernels: one block per SM owns a contiguous range of rows,
// holds z for them for the whole step, and reads each basis vector once
// (mgs.cuh).  With giv = 1 the last block of the launch takes no rows: its first
// warp applies the earlier rotations to column j as the coefficients arrive,
// while the other blocks run the later groups, and forms the new rotation, g and
// the tau test after the last.  With giv = 0 the first block does so at the end.
template <class I>
__device__ __forceinline__ void mgs_kernel(typename I::type* __restrict__ V, int64_t ldv, int n, GmresState* st,
                                           double* H, double* cs, double* sn, double* g, unsigned long long* tags,
                                           unsigned long long* hq, void* tri, unsigned long long tmo, int giv,
                                           int bulk) {
    typedef typename I::type T;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ MgsShared<I> sh;
    __shared__ GivensBatch s_giv;
    __shared__ unsigned s_seq;
    __shared__ int s_j, s_done, s_kmax;
    const int tid = threadIdx.x;
    if (tid == 0) {
        s_j = st->j;
        s_done = st->done;
        s_kmax = st->kmax;
        s_seq = *(volatile unsigned*)&st->bar.seq;  // reductions of this launch are s_seq + 1, s_seq + 2, ...
        mgs_shared_init<I>(sh);
    }
    __syncthreads();
    if (s_done) return;
    const int j = s_j, kmax = s_kmax;
    const unsigned seq0 = s_seq, tag = seq0 + 1u;
    const unsigned seq1 = seq0 + (unsigned)(j / I::GB) + 2u;  // the last reduction's number
    const int G = gridDim.x - giv;  // blocks that hold rows and publish partial sums
    const bool rotates = giv ? blockIdx.x == G : blockIdx.x == 0;
    if (blockIdx.x < G) {
        int64_t r0, r1;
        block_rows(n, G, r0, r1);
        MgsRows<I> R;
        R.nb = r1 > r0 ? (int)(r1 - r0) : 0;
        T* zg = V + (int64_t)(j + 1) * ldv + r0;
        typename I::P z[I::NP];
        unsigned char* zs = smraw + (size_t)I::S * I::stage_bytes;
#pragma unroll
        for (int u = 0; u < I::NU; ++u) {
            if constexpr (I::ZS) {
                typename I::P t[I::PN];
                unit_load<I>(R, zg, u, t);
#pragma unroll
                for (int k = 0; k < I::PN; ++k)
                    reinterpret_cast<typename I::P*>(zs)[(tid + u * I::BD) * I::PN + k] = t[k];
            } else {
                unit_load<I>(R, zg, u, z + u * I::PN);
            }
        }
        const MgsIo io{tags, hq, tri, &st->bar, tmo, G, bulk, blockIdx.x == 0, blockIdx.x == 0};
        unsigned seq = seq0, phase = 0, par = 0;
        T hz;
        if (!mgs_passes<I>(sh, io, R, z, smraw, zs, V + r0, ldv, j, tag, seq, phase, par, hz)) {
            if (blockIdx.x == 0 && tid == 0) {
                st->status = BSPAI_TIMEOUT;
                st->done = 1;
            }
            return;
        }
        const T hn = Ar<T>::sqrt(hz);
        const bool norm = hn > T(0) && isfinite((double)hn);
        const Quot<T> by(hn);
        const int nu = R.units();
#pragma unroll
        for (int u = 0; u < I::NU; ++u) {
            if (u >= nu) break;
            typename I::P t[I::PN];
#pragma unroll
            for (int k = 0; k < I::PN; ++k) {
                if constexpr (I::ZS) t[k] = reinterpret_cast<typename I::P*>(zs)[(tid + u * I::BD) * I::PN + k];
                else t[k] = z[u * I::PN + k];
                if (norm) t[k] = pk_quot(t[k], by);
            }
            unit_store<I>(R, zg, u, t);
        }
    }
    if (rotates && tid < 32) {
        const bool ok = givens_column<T>(s_giv, j, kmax, H, cs, sn, g, st, hq, tag, tmo);
        if (tid == 0) {
            if (ok) {
                // every block has read seq0 (the reductions are complete): advance it
                st->bar.seq = seq1;
            } else {
                st->status = BSPAI_TIMEOUT;
                st->done = 1;
            }
        }
    }
}

// rows of a thread one by one (R = 1) or in 16-byte units; fp64, and the smallest fp32 chunks
template <typename T, int R, int BD>
struct ResInst;
template <>
struct ResInst<float, 1, 1024> : MgsInst<float, 1, 1, 1024, 8, 16, false, false> {};
template <>
struct ResInst<double, 1, 1024> : MgsInst<double, 1, 1, 1024, 8, 16, false, false> {};
template <>
struct ResInst<double, 2, 1024> : MgsInst<double, 2, 1, 1024, 4, 8, true, false> {};
template <>
struct ResInst<double, 4, 1024> : MgsInst<double, 2, 2, 1024, 4, 5, true, false> {};
template <>
struct ResInst<double, 8, 1024> : MgsInst<double, 1, 8, 1024, 2, 2, true, true> {};
template <typename T, int R, int BD>
__global__ void __launch_bounds__(BD, 1) k_mgs_res(T* __restrict__ V, int64_t ldv, int n, GmresState* st, double* H,
                                                   double* cs, double* sn, double* g, unsigned long long* tags,
                                                   unsigned long long* hq, void* tri, unsigned long long tmo, int giv,
                                                   int bulk) {
    mgs_kernel<ResInst<T, R, BD>>(V, ldv, n, st, H, cs, sn, g, tags, hq, tri, tmo, giv, bulk);
}

// fp32, P pairs of adjacent rows per thread
template <int P, int BD>
struct ResInst2;
template <>
struct ResInst2<1, 1024> : MgsInst<float, 2, 1, 1024, 8, 16, false, false> {};
template <>
struct ResInst2<2, 1024> : MgsInst<float, 4, 1, 1024, 4, 8, true, false> {};
template <>
struct ResInst2<4, 1024> : MgsInst<float, 4, 2, 1024, 4, 6, true, false> {};
template <>
struct ResInst2<12, 512> : MgsInst<float, 4, 6, 512, 2, 4, true, false> {};
template <>
struct ResInst2<14, 512> : MgsInst<float, 4, 7, 512, 2, 3, true, false> {};
template <>
struct ResInst2<16, 512> : MgsInst<float, 4, 8, 512, 2, 3, true, false> {};
template <int P, int BD>
__global__ void __launch_bounds__(BD, 1) k_mgs_res2(float* __restrict__ V, int64_t ldv, int n, GmresState* st,
                                                    double* H, double* cs, double* sn, double* g,
                                                    unsigned long long* tags, unsigned long long* hq, void* tri,
                                                    unsigned long long tmo, int giv, int bulk) {
    mgs_kernel<ResInst2<P, BD>>(V, ldv, n, st, H, cs, sn, g, tags, hq, tri, tmo, giv, bulk);
}

// ------------------------------------------------------------------ one launch per run
// The whole Arnoldi loop of a small system with short rows in one cooperative launch:
// A v_j, M w and the Gram-Schmidt step of mgs.cuh with z never leaving its registers
// (fp32: two adjacent rows per thread, fp64: one).  What bounds a small system is
// latency: with three launches per step, each of a few microseconds of launch, first
// loads and drain, a step cost 35 us at n = 1,024; here it is two grid exchanges (v_j
// and w complete) and the reductions.  The row blocks exchange by tagged words;
// vectors another block writes are read from L2, after release / acquire fences around
// the exchange.  The last block applies the Givens rotations and decides the stop; the
// row blocks learn of step j - 1's decision at the end of step j, so at most one step
// is run in vain, and its column's words (two sets, by the step's parity) are not
// overwritten before they are read.
//
// A row's entries -- columns and values as the product uses them -- are kept in shared
// memory for the run (at most kCoopRow per row of each matrix, in one fp64 bucket or
// one or two narrow ones), so that a product waits for one load, x's, instead of a
// chain of three.  The others that are admitted (coop_blocks) are read from memory.
// Measured, 40 steps, us, three launches per step -> one launch per run:
//   u_g = fp32, kept:          fp32 or fp32 + fp16, 5 to 9 entries per row, n = 1,000 to
//                              32,000     1,258 to 1,372 -> 631 to 987; fp64 M 1,339 to 1,413 -> 930 to 1,240
//   u_g = fp32, from memory:   mixes with fp64, 5 entries  1,344 to 1,482 -> 932 to 1,374;
//                              fp32, 10 to 16 entries  1,281 to 1,425 -> 977 to 1,362;
//                              fp64 M, 10 to 16 entries, n = 1,000  1,388 to 1,544 -> 1,248 to 1,433,
//                              n = 8,192 and 32,000  1,363 to 1,509 -> 1,435 to 1,737
//   u_g = fp64, 5 to 9:        n = 1,000  1,775 to 1,893 -> 1,726 to 1,926; 8,192  1,741 to 1,847 -> 1,793
//                              to 1,900; 32,000  2,251 to 2,419 -> 1,951 to 2,173
//   u_g = fp64, 10 to 16:      n = 1,000  1,880 to 1,891 -> 1,912 to 2,115; 8,192  1,834 to 1,861 -> 1,959
//                              to 2,145; 32,000  2,331 to 2,390 -> 2,155 to 2,348
// The line does not look at precisions; the fp64 products of 10 to 16 entries are what it
// costs, 16 % at most.
constexpr int kCoopBD = 512;
constexpr int kCoopRow = 9;
constexpr int kCoopMax = 32;  // row blocks at most (fp64: twice as many)
constexpr int kCoopToken = kMgsMaxVals - 1;  // the slots' row of the exchanges without a value
template <typename T>
struct CoopInst : MgsInst<T, sizeof(T) == 4 ? 2 : 1, 1, kCoopBD, 8, 8, false, false> {};
// bytes of a matrix's cached entries: 4 of column and 4 or 8 of value
template <typename T>
constexpr size_t coop_cache_bytes(bool wide) {
    return (size_t)kCoopRow * kCoopBD * CoopInst<T>::VW * (wide ? 12 : 8);
}
template <typename T>
constexpr size_t coop_smem() {  // A's values are T, M's may be fp64 in either case
    return CoopInst<T>::smem + coop_cache_bytes<T>(sizeof(T) == 8) + coop_cache_bytes<T>(true);
}

// every row block's writes before it are visible to every row block's L2 reads after it
template <class I>
__device__ __forceinline__ void coop_exchange(MgsShared<I>& sh, const MgsIo& io, unsigned seq) {
    typedef typename I::type T;
    __syncthreads();
    if (io.G == 1) return;
    if (threadIdx.x < 32) {
        unsigned long long* row =
            io.tags + (int64_t)((int)(seq & 1u) * kMgsMaxVals + kCoopToken) * kTagMaxBlocks * TagWords<T>::W;
        if (threadIdx.x == 0) {
            __threadfence();
            tag_publish(T(0), row + (int64_t)blockIdx.x * TagWords<T>::W, seq);
        }
        T t;
        if (!tag_poll_row<T>(row, seq, io.G, io.bar, io.tmo, &t) && threadIdx.x == 0) *(volatile int*)&sh.ok = 0;
        __threadfence();
    }
    __syncthreads();
}

// A matrix's rows of this block in shared memory.  mode: 0 not kept, 1 one or two narrow
// buckets (fp32 values), 2 one fp64 bucket.  Slot l of row rr of thread t lies at
// (l VW + rr) kCoopBD + t, columns first, then values.
struct CoopCache {
    int mode;
    int* col;
    void* val;
};
// the entries of row r (rr of this thread) into the cache, bucket by bucket in ascending
// column order; their counts (the first bucket's in the low half); -1: too many
template <int VW>
__device__ __noinline__ int coop_cache_row(const BMDev& M, const CoopCache& c, int64_t r, int rr) {
    const int lane = (int)(r & 31);
    int at = 0, cnt = 0;
    for (int k = 0; k < M.q; ++k) {
        const BucketDev& B = M.b[k];
        const int64_t sb = B.sptr[r >> 5];
        const int w = (int)((B.sptr[(r >> 5) + 1] - sb) >> 5), first = at;
        for (int l = 0; l < w; ++l) {
            const int64_t p = sell_slot(sb, lane, l, B.packed);
            const int col = sell_col_ldg(B, p, r);
            if (col < 0) continue;
            if (at >= kCoopRow) return -1;
            const int slot = (at * VW + rr) * kCoopBD + threadIdx.x;
            c.col[slot] = col;
            if (c.mode == 2) static_cast<double*>(c.val)[slot] = __ldg(static_cast<const double*>(B.val) + p);
            else static_cast<float*>(c.val)[slot] = decode_rt(B, p, col, r);
            ++at;
        }
        cnt |= (at - first) << (16 * k);
    }
    return cnt;
}
// a row's product from its cached entries: every bucket's partial sum in ascending
// column order; the narrow buckets' sums a and b add to fl_T(fl64(a + b)), for fp32
// without fp64 arithmetic (53 >= 2 24 + 2 bits)
template <typename T, int VW>
__device__ __forceinline__ T coop_cached(const CoopCache& c, int cnt, int rr, const T* x) {
    const int n0 = cnt & 0xffff, n = n0 + (cnt >> 16);
    const int at = rr * kCoopBD + threadIdx.x;
    T xv[kCoopRow];
#pragma unroll
    for (int l = 0; l < kCoopRow; ++l) xv[l] = l < n ? __ldcg(x + c.col[l * VW * kCoopBD + at]) : T(0);
    if (c.mode == 2) {
        double a = 0.0;
#pragma unroll
        for (int l = 0; l < kCoopRow; ++l)
            if (l < n) a = __dadd_rn(a, __dmul_rn(static_cast<const double*>(c.val)[l * VW * kCoopBD + at], (double)xv[l]));
        return from_f64<T>(__dadd_rn(0.0, a));
    }
    float a = 0.0f, b = 0.0f;
#pragma unroll
    for (int l = 0; l < kCoopRow; ++l)
        if (l < n) {
            const float p = __fmul_rn(static_cast<const float*>(c.val)[l * VW * kCoopBD + at], to_f32<T>(xv[l]));
            if (l < n0) a = __fadd_rn(a, p);
            else b = __fadd_rn(b, p);
        }
    if constexpr (sizeof(T) == 4) return n > n0 ? __fadd_rn(__fadd_rn(0.0f, a), b) : __fadd_rn(0.0f, a);
    else return n > n0 ? __dadd_rn((double)a, (double)b) : __dadd_rn(0.0, (double)a);
}
// any other matrix (kept out of line, its descriptor in shared memory)
template <typename T>
__device__ __noinline__ T coop_row(const BMDev& M, int64_t r, const T* x) {
    return from_f64<T>(bucketed_row<T, true>(M, r, x));
}

template <typename T>
__global__ void __launch_bounds__(kCoopBD, 1) k_gmres_coop(const __grid_constant__ BMDev Av,
                                                           const __grid_constant__ BMDev Mv, T* V, int64_t ldv, int n,
                                                           GmresState* st, double* H, double* cs, double* sn,
                                                           double* g, unsigned long long* tags,
                                                           unsigned long long* hq, void* tri, T* W,
                                                           unsigned long long* flag, unsigned long long tmo) {
    typedef CoopInst<T> I;
    constexpr int VW = I::VW;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ MgsShared<I> sh;
    __shared__ GivensBatch s_giv;
    __shared__ unsigned s_seq;
    __shared__ int s_done, s_kmax, s_stop;
    __shared__ BMDev s_A, s_M;
    const int tid = threadIdx.x;
    if (tid == 0) {
        s_A = Av;
        s_M = Mv;
        s_done = st->done;
        s_kmax = st->kmax;
        s_seq = *(volatile unsigned*)&st->bar.seq;
        s_stop = 0;
        mgs_shared_init<I>(sh);
    }
    __syncthreads();
    if (s_done) return;
    const int kmax = s_kmax;
    const int G = gridDim.x - 1;
    const int64_t hqset = (int64_t)(kmax + 2) * TagWords<T>::W;  // one column's words
    unsigned seq = s_seq;
    auto reductions = [](int j) { return (unsigned)(j / I::GB) + 4u; };  // two exchanges, the groups, the norm
    if ((int)blockIdx.x == G) {
        if (tid >= 32) return;
        for (int j = 0; j < kmax; ++j) {
            const unsigned tag = seq + 1u;
            const bool ok = givens_column<T>(s_giv, j, kmax, H, cs, sn, g, st, hq + (j & 1) * hqset, tag, tmo);
            __syncwarp();
            seq += reductions(j);
            int done = 1;
            if (tid == 0) {
                if (ok) {
                    done = *(volatile int*)&st->done;
                    // the row blocks may run the next step in vain: its numbers are passed over too
                    if (done) st->bar.seq = seq + reductions(j + 1);
                } else {
                    st->status = BSPAI_TIMEOUT;
                    st->done = 1;
                }
                st_relaxed_u64(flag + (j & 1), ((unsigned long long)tag << 32) | (unsigned)done);
            }
            if (__shfl_sync(0xffffffffu, done, 0)) return;
        }
        return;
    }
    int64_t r0, r1;
    block_rows(n, G, r0, r1);
    MgsRows<I> R;
    R.nb = r1 > r0 ? (int)(r1 - r0) : 0;
    const int64_t r = r0 + R.row(0);
    const int rows = R.valid(0) / (int)sizeof(T);  // of this thread
    const MgsIo io{tags, hq, tri, &st->bar, tmo, G, 0, blockIdx.x == 0, blockIdx.x == 0};
    // the matrices' rows into shared memory
    CoopCache ca, cm;
    int na[VW], nm[VW];
    {
        auto mode = [](const BMDev& M) {
            if (M.q == 1 && M.b[0].prec == BSPAI_FP64) return 2;
            for (int k = 0; k < M.q; ++k)
                if (M.b[k].prec == BSPAI_FP64) return 0;
            return M.q <= 2 ? 1 : 0;
        };
        constexpr size_t slots = (size_t)kCoopRow * kCoopBD * VW;
        unsigned char* at = smraw + I::smem;
        ca.mode = mode(s_A);
        if (sizeof(T) == 4 && ca.mode == 2) ca.mode = 0;  // (A in fp64 beside fp32 vectors: no room for its values)
        ca.val = at;
        ca.col = reinterpret_cast<int*>(at + slots * sizeof(T));
        at += coop_cache_bytes<T>(sizeof(T) == 8);
        cm.mode = mode(s_M);
        cm.val = at;
        cm.col = reinterpret_cast<int*>(at + slots * 8);
        bool fa = true, fm = true;
#pragma unroll
        for (int rr = 0; rr < VW; ++rr) {
            na[rr] = nm[rr] = 0;
            if (rr < rows) {
                if (ca.mode) fa = fa && (na[rr] = coop_cache_row<VW>(s_A, ca, r + rr, rr)) >= 0;
                if (cm.mode) fm = fm && (nm[rr] = coop_cache_row<VW>(s_M, cm, r + rr, rr)) >= 0;
            }
        }
        if (!__syncthreads_and(fa)) ca.mode = 0;
        if (!__syncthreads_and(fm)) cm.mode = 0;
    }
    auto product = [&](const BMDev& M, const CoopCache& c, const int (&cnt)[VW], const T* x, T (&y)[VW]) {
#pragma unroll
        for (int rr = 0; rr < VW; ++rr)
            y[rr] = rr >= rows ? T(0) : c.mode ? coop_cached<T, VW>(c, cnt[rr], rr, x) : coop_row<T>(M, r + rr, x);
    };
    unsigned phase = 0, par = 0;
    bool good = true;
    for (int j = 0; j < kmax; ++j) {
        const unsigned tag = seq + 1u;
        T y[VW];
        typename I::P z[I::NP];
        product(s_A, ca, na, V + (int64_t)j * ldv, y);  // w = A v_j
#pragma unroll
        for (int rr = 0; rr < VW; ++rr)
            if (rr < rows) W[r + rr] = y[rr];
        coop_exchange<I>(sh, io, ++seq);
        product(s_M, cm, nm, W, y);  // z = M w
        if constexpr (VW == 2) z[0] = make_float2(y[0], y[1]);
        else z[0] = y[0];
        MgsIo ij = io;
        ij.hq = hq + (j & 1) * hqset;
        T hz;
        if (!*(volatile int*)&sh.ok ||
            !mgs_passes<I>(sh, ij, R, z, smraw, nullptr, V + r0, ldv, j, tag, seq, phase, par, hz)) {
            good = false;
            break;
        }
        const T hn = Ar<T>::sqrt(hz);
        if (hn > T(0) && isfinite((double)hn)) z[0] = pk_quot(z[0], Quot<T>(hn));
        unit_store<I>(R, V + (int64_t)(j + 1) * ldv + r0, 0, z);
        fence_proxy_async();  // later steps copy v_{j+1} by the copy engine
        // step j - 1's decision, by a warp that the exchange leaves idle
        if (j > 0 && tid == kCoopBD - 32) {
            const unsigned want = tag - reductions(j - 1);
            unsigned long long t0 = 0, f;
            while ((unsigned)((f = ld_relaxed_u64(flag + ((j - 1) & 1))) >> 32) != want) {
                const unsigned long long now = globaltimer_ns();
                if (!t0) t0 = now;
                if (now - t0 > tmo || *(volatile int*)&st->bar.err) {
                    atomicExch(&st->bar.err, 1);
                    *(volatile int*)&sh.ok = 0;
                    f = 1;
                    break;
                }
            }
            s_stop = (unsigned)f != 0u;
        }
        coop_exchange<I>(sh, ij, ++seq);
        if (!*(volatile int*)&sh.ok) {
            good = false;
            break;
        }
        if (s_stop) break;
    }
    if (!good && blockIdx.x == 0 && tid == 0) {
        st->status = BSPAI_TIMEOUT;
        st->done = 1;
    }
}

// y = R^-1 g by column-oriented back substitution (fp64): for i = k-1 .. 0,
// y_i = g_i / R_ii and g_t -= R_ti y_i for t < i (each g_t sees the same
// operations in the same order as a plain column back substitution).  When
// g and the triangle of R fit in kBackSmem bytes, the block first copies them
// into shared memory with every load in flight at once, and warp 0 then runs
// the k dependent rows from there.  Otherwise the whole block runs the rows:
// thread x holds rows x + kBackThreads c of the current column in registers
// and loads the next column's while the current row is processed, the owner
// of row i divides, and one barrier per row hands y_i to the others.
// Launch: one block of kBackThreads, kBackSmem bytes of dynamic shared memory.
constexpr int kBackThreads = 512;
constexpr size_t kBackSmem = 47 * 1024;  // with the static s_y, within the 48 KB a launch gets without opting in
constexpr int kBackC = 8;  // rows per thread in the streamed form: k <= kBackThreads * kBackC
__global__ void __launch_bounds__(kBackThreads) k_backsolve(const GmresState* st, const double* __restrict__ H,
                                                            const double* __restrict__ g, double* __restrict__ y,
                                                            int kmax) {
    extern __shared__ double sg[];
    __shared__ double s_y[2];
    const int k = st->j;
    const int tid = threadIdx.x, lane = tid & 31;
    for (int t = tid; t < k; t += blockDim.x) sg[t] = g[t];
    if ((size_t)k * (k + 3) / 2 * sizeof(double) <= kBackSmem) {
        // sg[0, k): g; then column i of R (rows 0 .. i) at sg + k + i (i + 1) / 2;
        // warp w copies columns w, w + 16, ... (integer indexing only: the fp64 pipe is narrow)
        double* R = sg + k;
        for (int i = tid >> 5; i < k; i += blockDim.x >> 5) {
            const double* hc = H + (int64_t)i * (kmax + 1);
            double* rc = R + i * (i + 1) / 2;
            for (int t = lane; t <= i; t += 32) rc[t] = hc[t];
        }
        __syncthreads();
        if (tid >= 32) return;
        for (int i = k - 1; i >= 0; --i) {
            const double* rc = R + i * (i + 1) / 2;
            const double yi = __ddiv_rn(sg[i], rc[i]);
            if (lane == 0) y[i] = yi;
            for (int t = lane; t < i; t += 32) sg[t] = __dsub_rn(sg[t], __dmul_rn(rc[t], yi));
            __syncwarp();
        }
        return;
    }
    // rows t = tid + kBackThreads c of column i (t <= i) in registers; g_t stays with its owner
    double nxt[kBackC], cur[kBackC];
    auto fetch = [&](int i) {
        const double* hc = H + (int64_t)i * (kmax + 1);
#pragma unroll
        for (int c = 0; c < kBackC; ++c) {
            const int t = tid + kBackThreads * c;
            nxt[c] = t <= i ? hc[t] : 0.0;
        }
    };
    double gt[kBackC];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kBackC; ++c) {
        const int t = tid + kBackThreads * c;
        gt[c] = t < k ? sg[t] : 0.0;
    }
    if (k > 0) fetch(k - 1);
    for (int i = k - 1; i >= 0; --i) {
#pragma unroll
        for (int c = 0; c < kBackC; ++c) cur[c] = nxt[c];
        if (i > 0) fetch(i - 1);
        if (tid == i % kBackThreads) {
            const int ci = i / kBackThreads;
            double gi = 0.0, di = 1.0;
#pragma unroll
            for (int c = 0; c < kBackC; ++c)
                if (c == ci) {
                    gi = gt[c];
                    di = cur[c];
                }
            const double yi = __ddiv_rn(gi, di);
            s_y[i & 1] = yi;
            y[i] = yi;
        }
        __syncthreads();
        const double yi = s_y[i & 1];
#pragma unroll
        for (int c = 0; c < kBackC; ++c) {
            const int t = tid + kBackThreads * c;
            if (t < i) gt[c] = __dsub_rn(gt[c], __dmul_rn(cur[c], yi));
        }
    }
}

// d = V y in u_g (y rounded to u_g, sequential over j), then x += d in fp64;
// max|d| -> norms[0], max|x| -> norms[1]
template <typename T>
__global__ void __launch_bounds__(256) k_gmres_update(const T* __restrict__ V, int64_t ldv, int n,
                                                      const GmresState* st, const double* __restrict__ y,
                                                      double* __restrict__ x, double* __restrict__ dout,
                                                      double* __restrict__ norms, int u32) {
    extern __shared__ unsigned char sraw[];
    T* sy = reinterpret_cast<T*>(sraw);
    const int k = st->j;
    for (int t = threadIdx.x; t < k; t += blockDim.x) sy[t] = Ar<T>::from(y[t]);
    __syncthreads();
    double dabs = 0.0, xabs = 0.0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        // the products added in order of j; the loads of 8 columns issued before their adds
        T acc = T(0);
        int jj = 0;
        for (; jj + 8 <= k; jj += 8) {
            T v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = V[(int64_t)(jj + u) * ldv + r];
#pragma unroll
            for (int u = 0; u < 8; ++u) acc = Ar<T>::add(acc, Ar<T>::mul(v[u], sy[jj + u]));
        }
        for (; jj < k; ++jj) acc = Ar<T>::add(acc, Ar<T>::mul(V[(int64_t)jj * ldv + r], sy[jj]));
        double d = (double)acc;
        // working precision u = fp32: d stored in u, x = fl32(x + d) (x and d
        // are fp32 values, so the fp64 sum rounds to the correctly rounded fp32 sum)
        if (u32) d = (double)__double2float_rn(d);
        if (dout) dout[r] = d;
        double xn = 0.0;
        if (x) {
            xn = __dadd_rn(x[r], d);
            if (u32) xn = (double)__double2float_rn(xn);
            x[r] = xn;
        }
        double da = fabs(d), xa = fabs(xn);
        if (!(da <= 1.7976931348623157e308)) da = __longlong_as_double(0x7ff0000000000000LL);
        if (!(xa <= 1.7976931348623157e308)) xa = __longlong_as_double(0x7ff0000000000000LL);
        dabs = fmax(dabs, da);
        xabs = fmax(xabs, xa);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dabs = fmax(dabs, __shfl_xor_sync(0xffffffffu, dabs, o));
        xabs = fmax(xabs, __shfl_xor_sync(0xffffffffu, xabs, o));
    }
    block_atomic_max_nonneg2(norms, dabs, norms + 1, xabs);
}

__global__ void k_absmax(int n, const double* __restrict__ v, double* __restrict__ out) {
    double a = 0.0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        double t = fabs(v[r]);
        if (!(t <= 1.7976931348623157e308)) t = __longlong_as_double(0x7ff0000000000000LL);
        a = fmax(a, t);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = fmax(a, __shfl_xor_sync(0xffffffffu, a, o));
    block_atomic_max_nonneg(out, a);
}

// ---------------------------------------------------------------- host side
struct HostFlags {
    int j, done, status, kmax;
};

struct GmresWork;
static int choose_mgs(GmresWork& W);

struct GmresWork {
    int n = 0, kmax = 0, G = 0, ug = BSPAI_FP32, up = BSPAI_FP32;
    int64_t ldv = 0;
    void* V = nullptr;
    void* w = nullptr;
    unsigned char* aux = nullptr;        // the reductions' buffers (carve):
    unsigned long long* tags = nullptr;  //   tagged slots: 2 parities x kMgsMaxVals x kTagMaxBlocks x 2 words
    unsigned long long* hq = nullptr;    //   tagged coefficients of the current column (two sets)
    unsigned long long* flag = nullptr;  //   tagged stopping decisions (k_gmres_coop; two sets)
    void* tri = nullptr;                 //   the groups' (I + L)^-1, up to kMgsMaxVals / 2 values per basis vector
    void* part = nullptr;                //   partial sums of the grid-barrier reductions
    GmresState* st = nullptr;
    double *H = nullptr, *cs = nullptr, *sn = nullptr, *g = nullptr, *y = nullptr, *norms = nullptr;
    HostFlags* hflags = nullptr;  // pinned
    unsigned long long tmo_ns = 2000000000ull;
    const bspai_bucketed* BA = nullptr;  // bucketed A for A v (null: A in u_p)
    int u32 = 0;                         // working precision u = fp32: d and x rounded to fp32
    void* res_fn = nullptr;  // k_mgs_res instance, or null for k_mgs
    int res_bd = 1024;       // its block size
    int res_kind = 0;        // 1: k_mgs_res, 2: k_mgs_res2 (see ResInstance)
    int res_per_thread = 0;  // its rows (k_mgs_res) or row pairs (k_mgs_res2) per thread
    int Gr = 0;              // its blocks that hold rows (at most one block per SM)
    int giv = 0;             // 1: one more block applies the Givens rotations during the passes
    int bulk = 0;            // 1: an instance able to poll by bulk copies does (see kBulkPollBytes)
    size_t res_smem = 0;
    cudaStream_t s = nullptr;

    // tags, hq and flag, which must start at zero (the sequence numbers that tag them start at one)
    size_t tagged_bytes() const {
        return sizeof(unsigned long long) *
               ((size_t)2 * kMgsMaxVals * kTagMaxBlocks * 2 + 4 * ((size_t)kmax + 2) + 2);
    }
    size_t aux_bytes() const {
        const size_t es = ug == BSPAI_FP64 ? 8 : 4;
        return tagged_bytes() + es * (kMgsMaxVals / 2) * ((size_t)kmax + 1) + es * 2 * kMgsMaxVals * (size_t)G;
    }
    // the rows past n of every basis vector: the on-chip MGS kernels copy whole 16-byte units
    int zero_pad() const {
        const size_t es = ug == BSPAI_FP64 ? 8 : 4;
        const int64_t to = ceil_div(n, 4) * 4;
        if (to == n) return BSPAI_OK;
        CUDA_TRY(cudaMemset2DAsync(static_cast<unsigned char*>(V) + es * (size_t)n, es * (size_t)ldv, 0,
                                   es * (size_t)(to - n), (size_t)kmax + 1, s));
        return BSPAI_OK;
    }
    void carve(void* base) {
        const size_t es = ug == BSPAI_FP64 ? 8 : 4;
        aux = static_cast<unsigned char*>(base);
        tags = reinterpret_cast<unsigned long long*>(aux);
        hq = tags + (size_t)2 * kMgsMaxVals * kTagMaxBlocks * 2;
        flag = hq + 4 * ((size_t)kmax + 2);
        tri = aux + tagged_bytes();
        part = static_cast<unsigned char*>(tri) + es * (kMgsMaxVals / 2) * ((size_t)kmax + 1);
    }
    int sms = 0;  // SMs the cooperative kernels may use (one block of k_mgs_res each)
    int alloc(int n_, int kmax_, int ug_, int up_, double timeout_s, int max_blocks, cudaStream_t st_) {
        sms = max_blocks > 0 && max_blocks < num_sms() ? max_blocks : num_sms();
        n = n_;
        kmax = kmax_;
        ug = ug_;
        up = up_;
        s = st_;
        tmo_ns = (unsigned long long)((timeout_s > 0 ? timeout_s : 2.0) * 1e9);
        const size_t es = ug == BSPAI_FP64 ? 8 : 4;
        ldv = ceil_div(n > 0 ? n : 1, 64) * 64;
        int occ = 0;
        cudaError_t e;
        if (ug == BSPAI_FP64) {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mgs<double>, 512, 0);
            int occ2 = 0;
            if (!e) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, k_gmres_start<double>, 512, 0);
            occ = occ < occ2 ? occ : occ2;
        } else {
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mgs<float>, 512, 0);
            int occ2 = 0;
            if (!e) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, k_gmres_start<float>, 512, 0);
            occ = occ < occ2 ? occ : occ2;
        }
        if (e) return cuda_error(e, "occupancy", __FILE__, __LINE__);
        if (occ < 1) return set_error(BSPAI_ERR_CUDA, "gmres: cooperative kernel does not fit on an SM");
        G = (occ >= 2 ? 2 : 1) * sms;
        BSPAI_TRY(dalloc(&V, es * (size_t)ldv * (size_t)(kmax + 1), s));
        BSPAI_TRY(dalloc(&w, es * (size_t)ldv, s));
        BSPAI_TRY(dalloc_t(&aux, aux_bytes(), s));
        carve(aux);
        CUDA_TRY(cudaMemsetAsync(aux, 0, tagged_bytes(), s));
        BSPAI_TRY(zero_pad());
        BSPAI_TRY(dalloc_t(&st, 1, s));
        BSPAI_TRY(dalloc_t(&H, (size_t)(kmax + 1) * kmax, s));
        BSPAI_TRY(dalloc_t(&cs, (size_t)kmax + 1, s));
        BSPAI_TRY(dalloc_t(&sn, (size_t)kmax + 1, s));
        BSPAI_TRY(dalloc_t(&g, (size_t)kmax + 2, s));
        BSPAI_TRY(dalloc_t(&y, (size_t)kmax + 1, s));
        BSPAI_TRY(dalloc_t(&norms, 4, s));
        CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(GmresState), s));
        CUDA_TRY(cudaMemsetAsync(g, 0, sizeof(double) * ((size_t)kmax + 2), s));
        // one pinned flag word per host thread, kept for the life of the process
        static thread_local HostFlags* t_flags = nullptr;
        if (!t_flags) CUDA_TRY(cudaMallocHost(&t_flags, sizeof(HostFlags)));
        hflags = t_flags;
        return choose_mgs(*this);
    }
    void release() {
        dfree(V, s); dfree(w, s); dfree(aux, s); dfree(st, s); dfree(H, s); dfree(cs, s);
        dfree(sn, s); dfree(g, s); dfree(y, s); dfree(norms, s);
        V = w = part = tri = nullptr;
        aux = nullptr;
        tags = hq = flag = nullptr;
        st = nullptr;
        H = cs = sn = g = y = norms = nullptr;
    }
};

// One k_mgs_res / k_mgs_res2 instance: its kernel, kind (1: k_mgs_res, rows of a
// thread one by one; 2: k_mgs_res2, rows in packed pairs), rows (R) or pairs (P)
// per thread, block size and dynamic shared memory.  The instance is the
// smallest that holds a block's chunk of rows: every instance listed here is
// reachable from choose_mgs for some order n (the parity tests run each one).
struct ResInstance {
    void* fn = nullptr;
    int kind = 0, per_thread = 0, bd = 0;
    size_t smem = 0;
};

template <typename T, int R, int BD>
static ResInstance res_instance() {
    return {(void*)k_mgs_res<T, R, BD>, 1, R, BD, ResInst<T, R, BD>::smem};
}
template <int P, int BD>
static ResInstance res_instance2() {
    return {(void*)k_mgs_res2<P, BD>, 2, P, BD, ResInst2<P, BD>::smem};
}

template <typename T>
static ResInstance pick_res(int64_t chunk) {
    const int R = (int)ceil_div(chunk, 1024);
    if (R <= 1) return res_instance<T, 1, 1024>();
    if constexpr (sizeof(T) == 4) {
        // fp32: rows in adjacent pairs, packed two-lane arithmetic
        if (R <= 2) return res_instance2<1, 1024>();
        if (R <= 4) return res_instance2<2, 1024>();
        if (R <= 8) return res_instance2<4, 1024>();
        // more rows per block: 512 threads with more pairs each (chunk > 8192)
        const int Rp = (int)ceil_div(chunk, 512);
        if (Rp <= 24) return res_instance2<12, 512>();
        if (Rp <= 28) return res_instance2<14, 512>();
        if (Rp <= 32) return res_instance2<16, 512>();
        return {};
    } else {
        if (R <= 2) return res_instance<T, 2, 1024>();
        if (R <= 4) return res_instance<T, 4, 1024>();
        if (R <= 8) return res_instance<T, 8, 1024>();
        return {};
    }
}

// Use the on-chip MGS kernel when one block per SM can hold its rows of z on
// chip: at most 16,384 rows of a block in fp32, 8,192 in fp64.
static int choose_mgs(GmresWork& W) {
    W.res_fn = nullptr;
    // As few blocks as hold the rows of z on chip, but not fewer than kMgsBlocks: each
    // grid reduction waits for every block, and fewer blocks shorten it (measured per
    // reduction, n = 65,536 / 262,144: 2.5 / 3.1 us at 152 blocks, 1.6 / 1.9 us at 64).
    // At 128^3 fewer blocks stopped paying: 103 blocks of 40 fp32 rows per thread solved
    // in 90.8 ms against 87.7 ms at 128 blocks of 32, and a scalar 768-thread instance
    // (22,272 rows, register spills) took 107.6 ms at 95 blocks.
    const int64_t cap = W.ug == BSPAI_FP64 ? 8192 : 16384;
    int Gr = (int)ceil_div(W.n, cap);
    if (Gr < kMgsBlocks) Gr = kMgsBlocks;
    // the Givens block wants an SM of its own (one block per SM at these sizes): the
    // rotations of a column otherwise follow its last reduction.  Not in fp64 on a few SMs,
    // where the rows' share of that SM costs more (40 steps, us, with an SM for the rotations
    // -> without: 2 SMs, 7,505 rows 8,181 -> 5,594; 6, 37,505 8,602 -> 7,877; 12, 22,005
    // 3,889 -> 3,875; 16, 30,005 3,901 -> 3,953; 38, 74,005 4,021 -> 4,113)
    if (Gr >= W.sms) {
        const int64_t share = W.sms > 1 ? ceil_div(W.n, W.sms - 1) : cap + 1;
        const bool rows_first = W.ug == BSPAI_FP64 && W.sms <= 12 && share > 1024;
        Gr = share <= cap && !rows_first ? W.sms - 1 : W.sms;
    }
    if (Gr > kTagMaxBlocks) return BSPAI_OK;
    int64_t chunk = ceil_div(ceil_div(W.n, Gr), 32) * 32;
    const size_t es = W.ug == BSPAI_FP64 ? 8 : 4;
    const ResInstance ri = es == 8 ? pick_res<double>(chunk) : pick_res<float>(chunk);
    if (!ri.fn) return BSPAI_OK;
    if (es == 8 && ri.per_thread > 1) {
        // fp64 is bound by the narrow fp64 pipe of the SMs that hold rows: spread the rows
        // over more blocks, down to just over half of the instance's capacity (per vector
        // at n = 262,144: 9.0 us before, 3.6 with groups of 4 on 127 blocks)
        const int64_t least = (int64_t)ri.per_thread * ri.bd / 2 + 32;
        const int spare = W.sms - 1 > 0 ? W.sms - 1 : 1;
        int64_t c = ceil_div(ceil_div(W.n, spare < kTagMaxBlocks ? spare : kTagMaxBlocks), 32) * 32;
        if (c < least) c = least;
        if (c < chunk) {
            chunk = c;
            Gr = (int)ceil_div(W.n, chunk);
        }
    }
    CUDA_TRY(cudaFuncSetAttribute(ri.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ri.smem));
    int occ = 0;
    CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ri.fn, ri.bd, ri.smem));
    if (occ < 1) return BSPAI_OK;
    W.res_fn = ri.fn;
    W.res_bd = ri.bd;
    W.res_kind = ri.kind;
    W.res_per_thread = ri.per_thread;
    W.Gr = Gr;
    W.giv = Gr + 1 <= W.sms ? 1 : 0;
    // bulk-copy polling where it was measured to pay: at least kMgsBlocks blocks (a solve
    // confined to a few SMs, as each of several concurrent right-hand sides is, polls few
    // slots and the copy engine's round trip loses) and kBulkPollBytes of a vector per block
    W.bulk = Gr >= kMgsBlocks && (int64_t)chunk * (int64_t)es >= kBulkPollBytes ? 1 : 0;
    W.res_smem = ri.smem;
    return BSPAI_OK;
}

// The row blocks of the whole run in one launch (k_gmres_coop), or 0: an order that few
// enough blocks cover, with a further block left for the rotations, and matrices whose
// rows are short: buckets whose widest slices add up to twice what is kept of a row, since
// packed widths are rounded up to fours (8 for a 5- or 7-point stencil's rows, in each of
// two buckets).  A longer row is read from memory; both sides measured above.  A run of one
// step in fp32 does not earn back the rows' way into shared memory (n = 1,000 and 8,192:
// 138 and 141 us in one launch, 127 and 129 in three).
static int coop_blocks(const GmresWork& W, const BMDev& A, const BMDev& M) {
    if (W.ug == BSPAI_FP32 && W.kmax < 2) return 0;
    const int per = W.ug == BSPAI_FP64 ? kCoopBD : 2 * kCoopBD;
    const int64_t G = ceil_div(W.n, per);
    if (G > (int64_t)kCoopMax * (2 * kCoopBD / per) || G >= W.sms) return 0;
    for (const BMDev* B : {&A, &M}) {
        int w = 0;
        for (int k = 0; k < B->q; ++k) {
            if (B->b[k].maxw < 0) return 0;
            w += B->b[k].maxw;
        }
        if (w > 2 * kCoopRow) return 0;
    }
    return (int)G;
}

static int coop_launch_cfg(void* fn, int G, int block, size_t smem, void** args, cudaStream_t s) {
    cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(G), dim3(block), args, smem, s);
    note_launch();
    if (e) return cuda_error(e, "cudaLaunchCooperativeKernel", __FILE__, __LINE__);
    return BSPAI_OK;
}

static int coop_launch(void* fn, int G, void** args, cudaStream_t s) {
    cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(G), dim3(512), args, 0, s);
    note_launch();
    if (e) return cuda_error(e, "cudaLaunchCooperativeKernel", __FILE__, __LINE__);
    return BSPAI_OK;
}

struct GmresResult {
    int k = 0;
    int status = BSPAI_OK;
    double beta = 0.0, res = 0.0, dmax = 0.0, xmax = 0.0;
};

// One GMRES solve of (M A) d = M r.  x != null: x += d; dout != null: d out.
template <typename T>
static int gmres_run(GmresWork& W, const bspai_matrix* A, const bspai_bucketed* BM, const double* r, double tau,
                     double* x, double* dout, GmresResult& out, double target = 0.0) {
    cudaStream_t s = W.s;
    const int n = W.n;
    const int tprec = W.ug;  // T matches u_g
    // A v: A in u_p, or A's buckets by the adaptive-precision SpMV (Alg 2.3 applied to A)
    const BMDev Aview = W.BA ? W.BA->dev() : up_view(A, W.up);
    const BMDev Mview = BM->dev();
    T* V = reinterpret_cast<T*>(W.V);
    T* w = reinterpret_cast<T*>(W.w);
    T* part = reinterpret_cast<T*>(W.part);
    {
        ProfScope ps(BSPAI_K_OTHER, s);
        k_state_init<<<1, 1, 0, s>>>(W.st, W.kmax, tau, target);
        note_launch();
        CUDA_LAUNCH_CHECK();
        CUDA_TRY(cudaMemsetAsync(W.norms, 0, 4 * sizeof(double), s));
    }
    {
        ProfScope ps(BSPAI_K_BSPMV, s);
        BSPAI_TRY(launch_bspmv(Mview, r, BSPAI_FP64, V, tprec, s));
    }
    {
        ProfScope ps(BSPAI_K_MGS, s);
        int nn = n;
        void* args[] = {&V, &nn, &W.st, &W.g, &part, &W.tmo_ns};
        BSPAI_TRY(coop_launch((void*)k_gmres_start<T>, W.G, args, s));
    }
    int launched = 0, chunk = 4;
    const int* jd = &W.st->j;
    BMDev Ac = compact_buckets(Aview), Mc = compact_buckets(Mview);
    if (const int Gc = coop_blocks(W, Ac, Mc)) {
        ProfScope ps(BSPAI_K_MGS, s);
        const void* fn = (const void*)k_gmres_coop<T>;
        CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)coop_smem<T>()));
        int nn = n;
        int64_t ld = W.ldv;
        void* args[] = {&Ac, &Mc, &V, &ld, &nn, &W.st, &W.H, &W.cs, &W.sn, &W.g, &W.tags, &W.hq, &W.tri, &w, &W.flag,
                        &W.tmo_ns};
        BSPAI_TRY(coop_launch_cfg((void*)fn, Gc + 1, kCoopBD, coop_smem<T>(), args, s));
        launched = W.kmax;
        // a solve that shares the GPU with others (max_blocks) queues nothing behind the run:
        // what waits for it would hold up the streams that share its hardware queue (eight
        // right-hand sides of n = 9,216, forward and backward: 134 ms, against 54 so)
        if (W.sms < num_sms()) CUDA_TRY(cudaStreamSynchronize(s));
    }
    while (launched < W.kmax) {
        for (int c = 0; c < chunk && launched < W.kmax; ++c, ++launched) {
            {
                ProfScope ps(BSPAI_K_SPMV_A, s);
                BSPAI_TRY(launch_bspmv_idx(Aview, V, tprec, w, tprec, jd, W.ldv, 0, 0, s));
            }
            {
                ProfScope ps(BSPAI_K_BSPMV, s);
                BSPAI_TRY(launch_bspmv_idx(Mview, w, tprec, V, tprec, jd, 0, W.ldv, 1, s));
            }
            {
                ProfScope ps(BSPAI_K_MGS, s);
                int nn = n;
                int64_t ld = W.ldv;
                if (W.res_fn) {
                    void* args[] = {&V, &ld, &nn, &W.st, &W.H, &W.cs, &W.sn, &W.g, &W.tags, &W.hq, &W.tri,
                                    &W.tmo_ns, &W.giv, &W.bulk};
                    BSPAI_TRY(coop_launch_cfg(W.res_fn, W.Gr + W.giv, W.res_bd, W.res_smem, args, s));
                } else {
                    T* tri = reinterpret_cast<T*>(W.tri);
                    void* args[] = {&V, &ld, &nn, &W.st, &W.H, &W.cs, &W.sn, &W.g, &part, &tri, &W.hq, &W.tmo_ns};
                    BSPAI_TRY(coop_launch((void*)k_mgs<T>, W.G, args, s));
                }
            }
        }
        CUDA_TRY(cudaMemcpyAsync(W.hflags, W.st, sizeof(HostFlags), cudaMemcpyDeviceToHost, s));
        CUDA_TRY(cudaStreamSynchronize(s));
        if (W.hflags->done) break;
        chunk = chunk < 32 ? chunk * 2 : 32;
    }
    {
        ProfScope ps(BSPAI_K_UPDATE, s);
        k_backsolve<<<1, kBackThreads, kBackSmem, s>>>(W.st, W.H, W.g, W.y, W.kmax);
        note_launch();
        CUDA_LAUNCH_CHECK();
        if (n > 0) {
            k_gmres_update<T><<<wave_grid(n), 256, sizeof(T) * (size_t)(W.kmax + 1), s>>>(
                V, W.ldv, n, W.st, W.y, x, dout, W.norms, W.u32);
            note_launch();
            CUDA_LAUNCH_CHECK();
        }
    }
    GmresState hs;
    double hn[2];
    CUDA_TRY(cudaMemcpyAsync(&hs, W.st, sizeof hs, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaMemcpyAsync(hn, W.norms, sizeof hn, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    BSPAI_TRY(stage_timeout_take(s));
    out.k = hs.j;
    out.status = hs.status;
    out.beta = hs.beta;
    out.res = hs.res;
    out.dmax = hn[0];
    out.xmax = hn[1];
    if (hs.status == BSPAI_TIMEOUT) {
        // the barrier state is undefined after a timeout: reset it (and the
        // tagged words, whose numbers restart with it) for reuse
        CUDA_TRY(cudaMemsetAsync(&W.st->bar, 0, sizeof(GridBar), s));
        CUDA_TRY(cudaMemsetAsync(W.aux, 0, W.tagged_bytes(), s));
        return set_error(BSPAI_TIMEOUT, "gmres: a grid barrier exceeded its time limit");
    }
    return BSPAI_OK;
}

static int check_solver_precs(int u, int u_r, int u_g, int u_p) {
    if (u != BSPAI_FP64 && u != BSPAI_FP32)
        return set_error(BSPAI_ERR_UNSUPPORTED, "working precision u must be FP64 or FP32");
    if (u_r != BSPAI_DD && u_r != BSPAI_FP64) return set_error(BSPAI_ERR_UNSUPPORTED, "u_r must be DD or FP64");
    if (u_g != BSPAI_FP32 && u_g != BSPAI_FP64) return set_error(BSPAI_ERR_UNSUPPORTED, "u_g must be FP32 or FP64");
    if (u_p != BSPAI_FP32 && u_p != BSPAI_FP64) return set_error(BSPAI_ERR_UNSUPPORTED, "u_p must be FP32 or FP64");
    return BSPAI_OK;
}

static constexpr int kKmaxLimit = 4000;  // shared-memory bound of k_backsolve / k_gmres_update

static int resolve_kmax(const bspai_opts_t* o, int n) {
    int k = o && o->kmax > 0 ? o->kmax : (n < 1000 ? n : 1000);
    if (k > n) k = n;
    if (k > kKmaxLimit) k = kKmaxLimit;
    return k < 1 ? 1 : k;
}

int launch_residual_prec(const bspai_matrix* A, const double* x, const double* b, double* r, double* norms,
                         int u_r, int u, cudaStream_t s);

__global__ void k_round_f32(int n, double* __restrict__ x) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) x[i] = (double)__double2float_rn(x[i]);
}

// d += e in fp64 (e, a restarted cycle's correction, already stored in u); first: d = 0 + e
__global__ void k_dacc_add(int n, double* __restrict__ d, const double* __restrict__ e, int first) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) d[i] = __dadd_rn(first ? 0.0 : d[i], e[i]);
}

// x = fl_u(x + fl_u(d)) for a correction summed over restarted cycles, with
// norms[0] = max |fl_u(d)|, norms[1] = max |x| (as k_gmres_update)
__global__ void __launch_bounds__(256) k_apply_d(int n, double* __restrict__ x, const double* __restrict__ d,
                                                 double* __restrict__ norms, int u32) {
    double dabs = 0.0, xabs = 0.0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
        double dv = d[r];
        if (u32) dv = (double)__double2float_rn(dv);
        double xn = __dadd_rn(x[r], dv);
        if (u32) xn = (double)__double2float_rn(xn);
        x[r] = xn;
        double da = fabs(dv), xa = fabs(xn);
        if (!(da <= 1.7976931348623157e308)) da = __longlong_as_double(0x7ff0000000000000LL);
        if (!(xa <= 1.7976931348623157e308)) xa = __longlong_as_double(0x7ff0000000000000LL);
        dabs = fmax(dabs, da);
        xabs = fmax(xabs, xa);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dabs = fmax(dabs, __shfl_xor_sync(0xffffffffu, dabs, o));
        xabs = fmax(xabs, __shfl_xor_sync(0xffffffffu, xabs, o));
    }
    block_atomic_max_nonneg2(norms, dabs, norms + 1, xabs);
}

static int ir_solve(bspai_matrix* A, const bspai_bucketed* BA, const double* b, const bspai_bucketed* BM,
                    const bspai_spai* M, int u, int u_r, int u_g, int u_p, double tol, const bspai_opts_t* opts,
                    double* x, cudaStream_t s, bspai_solve_info_t* info) {
    bspai_opts_t o;
    bspai_opts_default(&o);
    if (opts) o = *opts;
    const int n = A->n;
    const int kmax = resolve_kmax(&o, n);
    int imax = o.i_max > 0 ? o.i_max : 10;
    if (imax > 32) imax = 32;
    const double ustop = o.u_stop > 0 ? o.u_stop : (u == BSPAI_FP32 ? 0x1p-24 : 0x1p-53);
    const double stag = o.stagnation > 0 ? o.stagnation : 0.9;
    const double tau = tol > 0 ? tol : o.tau;
    bspai_solve_info_t inf;
    memset(&inf, 0, sizeof inf);
    if (BM->n != n || (M && M->n != n)) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve: size mismatch");
    if (!o.x0_given && !M) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve: need M for x0 = M b");
    if (n == 0) {
        if (info) *info = inf;
        return BSPAI_OK;
    }
    double* r = nullptr;
    double* nrm = nullptr;
    double *dacc = nullptr, *ecyc = nullptr, *rcyc = nullptr;  // restarted cycles only
    GmresWork W;
    int rc = BSPAI_OK;
    auto finish = [&](int code) {
        dfree(r, s);
        dfree(nrm, s);
        dfree(dacc, s);
        dfree(ecyc, s);
        dfree(rcyc, s);
        W.release();
        inf.status = code;
        if (info) *info = inf;
        return code;
    };
    // the Krylov basis: kmax + 1 vectors, or fewer (restarted cycles) when the caller's
    // byte cap or the device's free memory asks
    int km = kmax;
    if (o.basis_bytes_max > 0) {
        const int64_t vec = (int64_t)(u_g == BSPAI_FP64 ? 8 : 4) * (ceil_div(n, 64) * 64);
        const int64_t fit = o.basis_bytes_max / vec - 1;
        if (fit < 1)
            return finish(set_error(BSPAI_ERR_INVALID,
                                    "gmres_ir_solve: basis_bytes_max holds fewer than two Krylov vectors of order %d",
                                    n));
        if (fit < km) km = (int)fit;
    }
    if ((rc = dalloc_t(&r, (size_t)n, s))) return finish(rc);
    if ((rc = dalloc_t(&nrm, 4, s))) return finish(rc);
    rc = W.alloc(n, km, u_g, u_p, o.barrier_timeout_s, o.max_blocks, s);
    while (rc == BSPAI_ERR_NOMEM && km > 8) {
        W.release();
        (void)cudaGetLastError();  // the failed allocation's error is not the next launch's
        km = km / 2 > 8 ? km / 2 : 8;
        rc = W.alloc(n, km, u_g, u_p, o.barrier_timeout_s, o.max_blocks, s);
    }
    if (rc) return finish(rc);
    if (km < kmax) {
        if ((rc = dalloc_t(&dacc, (size_t)n, s))) return finish(rc);
        if ((rc = dalloc_t(&ecyc, (size_t)n, s))) return finish(rc);
        if ((rc = dalloc_t(&rcyc, (size_t)n, s))) return finish(rc);
    }
    inf.kmem = km;
    W.BA = BA;
    W.u32 = u == BSPAI_FP32;
    // ||A||_inf, ||b||_inf
    double anorm = 0.0, bnorm = 0.0;
    {
        ProfScope ps(BSPAI_K_OTHER, s);
        cudaError_t e0 = cudaMemsetAsync(nrm, 0, 4 * sizeof(double), s);
        if (e0) return finish(cuda_error(e0, "memset", __FILE__, __LINE__));
        k_absmax<<<wave_grid(n), 256, 0, s>>>(n, b, nrm);
        note_launch();
        if (!o.x0_given) {
            // x0 = M b with the unbucketed M in u_f (fp32 or fp16), stored in fp64
            if ((rc = launch_apply_uf(M, b, x, s))) return finish(rc);
        } else if (W.u32) {
            // a given x0 is held in u = fp32 (M b in u_f <= fp32 already is)
            k_round_f32<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(n, x);
            note_launch();
        }
    }
    cudaError_t e = cudaMemcpyAsync(&bnorm, nrm, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaMemcpyAsync(&anorm, A->norm_inf, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (e) return finish(cuda_error(e, "norms", __FILE__, __LINE__));
    double dprev = INFINITY;
    int code = BSPAI_NOT_CONVERGED;
    for (int i = 0; i < imax; ++i) {
        double hn[2] = {0, 0};
        e = cudaMemsetAsync(nrm, 0, 2 * sizeof(double), s);
        if (e) return finish(cuda_error(e, "memset", __FILE__, __LINE__));
        if ((rc = launch_residual_prec(A, x, b, r, nrm, u_r, u, s))) return finish(rc);
        e = cudaMemcpyAsync(hn, nrm, sizeof hn, cudaMemcpyDeviceToHost, s);
        if (!e) e = cudaStreamSynchronize(s);
        if (e) return finish(cuda_error(e, "residual norms", __FILE__, __LINE__));
        // a zero residual is an exact solution (b = 0, x = 0 gives 0 / 0 otherwise)
        const double nbe = hn[0] == 0.0 ? 0.0 : hn[0] / (anorm * hn[1] + bnorm);
        inf.nbe[i] = nbe;
        if (!std::isfinite(nbe)) {
            code = set_error(BSPAI_NONFINITE, "gmres_ir_solve: non-finite residual at step %d", i);
            break;
        }
        if (nbe <= ustop) {
            inf.stop_reason = 1;
            code = BSPAI_OK;
            break;
        }
        GmresResult gr;
        int cycles = 1;
        if (km >= kmax) {
            rc = u_g == BSPAI_FP64 ? gmres_run<double>(W, A, BM, r, tau, x, nullptr, gr)
                                   : gmres_run<float>(W, A, BM, r, tau, x, nullptr, gr);
            if (rc) return finish(rc);
        } else {
            // restarted cycles of km steps on the correction equation A d = r: cycle c > 0
            // starts from r - A d (u_r, stored in u) and stops at cycle 0's level tau beta_0
            int steps = 0;
            double lvl = 0.0, beta0 = 0.0;
            GmresResult gc;
            cycles = 0;
            while (steps < kmax) {
                const double* rin = r;
                if (cycles > 0) {
                    e = cudaMemsetAsync(nrm + 2, 0, 2 * sizeof(double), s);
                    if (e) return finish(cuda_error(e, "memset", __FILE__, __LINE__));
                    if ((rc = launch_residual_prec(A, dacc, r, rcyc, nrm + 2, u_r, u, s))) return finish(rc);
                    rin = rcyc;
                }
                rc = u_g == BSPAI_FP64 ? gmres_run<double>(W, A, BM, rin, tau, nullptr, ecyc, gc, lvl)
                                       : gmres_run<float>(W, A, BM, rin, tau, nullptr, ecyc, gc, lvl);
                if (rc) return finish(rc);
                if (cycles == 0) {
                    beta0 = gc.beta;
                    lvl = tau * beta0;
                }
                k_dacc_add<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(n, dacc, ecyc, cycles == 0);
                note_launch();
                steps += gc.k;
                ++cycles;
                if (gc.status == BSPAI_NONFINITE || gc.k < km || gc.res <= lvl || !(gc.beta > 0.0)) break;
            }
            {
                ProfScope ps(BSPAI_K_UPDATE, s);
                e = cudaMemsetAsync(W.norms, 0, 2 * sizeof(double), s);
                if (e) return finish(cuda_error(e, "memset", __FILE__, __LINE__));
                k_apply_d<<<wave_grid(n), 256, 0, s>>>(n, x, dacc, W.norms, W.u32);
                note_launch();
            }
            double hn2[2];
            e = cudaMemcpyAsync(hn2, W.norms, sizeof hn2, cudaMemcpyDeviceToHost, s);
            if (!e) e = cudaStreamSynchronize(s);
            if (e) return finish(cuda_error(e, "restarted GMRES update", __FILE__, __LINE__));
            gr.k = steps;
            gr.status = gc.status;
            gr.beta = beta0;
            gr.res = gc.res;
            gr.dmax = hn2[0];
            gr.xmax = hn2[1];
        }
        inf.gmres_cycles[i] = cycles;
        inf.gmres_iters[i] = gr.k;
        inf.total_iters += gr.k;
        inf.relres[i] = gr.beta > 0 ? gr.res / gr.beta : 0.0;
        inf.ir_steps = i + 1;
        inf.dx[i] = gr.xmax > 0 ? gr.dmax / gr.xmax : gr.dmax;
        if (gr.status == BSPAI_NONFINITE || !std::isfinite(gr.dmax) || !std::isfinite(gr.xmax)) {
            code = set_error(BSPAI_NONFINITE, "gmres_ir_solve: non-finite value in GMRES at step %d", i);
            break;
        }
        if (gr.dmax <= ustop * gr.xmax) {
            inf.stop_reason = 2;
            code = BSPAI_OK;
            break;
        }
        if (i > 0 && gr.dmax > stag * dprev) {
            inf.stop_reason = 3;
            code = BSPAI_OK;
            break;
        }
        dprev = gr.dmax;
    }
    if (code == BSPAI_NOT_CONVERGED) set_error(code, "gmres_ir_solve: i_max = %d steps without meeting a stopping test", imax);
    return finish(code);
}

// Failure-detection self-test: the bounded grid barrier, its arrival counter
// pre-loaded past the value at which the last arrival releases it (hold != 0),
// so that no arrival releases it and every block's wait must run out.
__global__ void k_barrier_selftest(GridBar* bar, unsigned long long tmo, int* failed) {
    const bool ok = grid_sync(bar, tmo);
    if (!ok && threadIdx.x == 0) atomicExch(failed, 1);
}

}  // namespace bspai

using namespace bspai;

extern "C" {

int bspai_barrier_selftest(int blocks, int hold, double timeout_s, bspai_stream_t st, float* waited_ms) {
    cudaStream_t s = (cudaStream_t)st;
    if (blocks < 1 || blocks > 1024 || !(timeout_s > 0) || timeout_s > 10)
        return set_error(BSPAI_ERR_INVALID, "barrier self-test: bad arguments");
    int dev = 0, coop = 0, per_sm = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_barrier_selftest, 32, 0));
    if (!coop || blocks > per_sm * num_sms())
        return set_error(BSPAI_ERR_INVALID, "barrier self-test: blocks cannot be co-resident");
    void* p = nullptr;
    int rc = dalloc(&p, sizeof(GridBar) + sizeof(int), s);
    if (rc) return rc;
    GridBar* bar = (GridBar*)p;
    int* failed = (int*)(bar + 1);
    GridBar init{hold ? (unsigned)blocks : 0u, 0u, 0, 0};  // arrivals count from here
    int h_failed = 0;
    float ms = 0;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaMemcpyAsync(bar, &init, sizeof init, cudaMemcpyHostToDevice, s);
    if (!e) e = cudaMemsetAsync(failed, 0, sizeof(int), s);
    if (!e) e = cudaEventCreate(&e0);
    if (!e) e = cudaEventCreate(&e1);
    if (!e) e = cudaEventRecord(e0, s);
    if (!e) {
        unsigned long long tmo = (unsigned long long)(timeout_s * 1e9);
        void* args[] = {&bar, &tmo, &failed};
        e = cudaLaunchCooperativeKernel((const void*)k_barrier_selftest, dim3(blocks), dim3(32), args, 0, s);
        note_launch();
    }
    if (!e) e = cudaEventRecord(e1, s);
    if (!e) e = cudaMemcpyAsync(&h_failed, failed, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (!e) e = cudaStreamSynchronize(s);
    if (!e) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    dfree(p, s);
    if (e) return cuda_error(e, "barrier self-test", __FILE__, __LINE__);
    if (waited_ms) *waited_ms = ms;
    if (h_failed) return set_error(BSPAI_TIMEOUT, "barrier self-test: the grid barrier timed out");
    return BSPAI_OK;
}

int gmres_ir_solve_h(bspai_A_h A, const double* b, bspai_BM_h BM, bspai_M_h M, bspai_prec_t u, bspai_prec_t u_r,
                     bspai_prec_t u_g, bspai_prec_t u_p, double tol, const bspai_opts_t* opts, double* x,
                     bspai_stream_t s, bspai_solve_info_t* info) {
    if (!A || A->magic != kMagicA) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve: bad A handle");
    if (!BM || BM->magic != kMagicBM) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve: bad bucketed M handle");
    if (M && M->magic != kMagicM) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve: bad M handle");
    if (A->n > 0 && (!b || !x)) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve: null vector");
    BSPAI_TRY(check_solver_precs(u, u_r, u_g, u_p));
    return ir_solve(A, nullptr, b, BM, M, u, u_r, u_g, u_p, tol, opts, x, (cudaStream_t)s, info);
}

int gmres_ir_solve_hb(bspai_A_h A, bspai_BM_h A_bucketed, const double* b, bspai_BM_h BM, bspai_M_h M,
                      bspai_prec_t u, bspai_prec_t u_r, bspai_prec_t u_g, double tol, const bspai_opts_t* opts,
                      double* x, bspai_stream_t s, bspai_solve_info_t* info) {
    if (!A || A->magic != kMagicA) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve_hb: bad A handle");
    if (!A_bucketed || A_bucketed->magic != kMagicBM || A_bucketed->n != A->n)
        return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve_hb: bad bucketed A handle");
    if (!BM || BM->magic != kMagicBM) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve_hb: bad bucketed M handle");
    if (M && M->magic != kMagicM) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve_hb: bad M handle");
    if (A->n > 0 && (!b || !x)) return set_error(BSPAI_ERR_INVALID, "gmres_ir_solve_hb: null vector");
    BSPAI_TRY(check_solver_precs(u, u_r, u_g, u_g));
    return ir_solve(A, A_bucketed, b, BM, M, u, u_r, u_g, u_g, tol, opts, x, (cudaStream_t)s, info);
}

int gmres_ir_solve(const bspai_csr_t* Acsr, const double* b, bspai_BM_h BM, bspai_M_h M, bspai_prec_t u,
                   bspai_prec_t u_r, bspai_prec_t u_g, bspai_prec_t u_p, double tol, const bspai_opts_t* opts,
                   double* x, bspai_stream_t s, bspai_solve_info_t* info) {
    BSPAI_TRY(check_solver_precs(u, u_r, u_g, u_p));
    bspai_matrix* A = nullptr;
    BSPAI_TRY(matrix_create(Acsr, (cudaStream_t)s, &A));
    int rc = gmres_ir_solve_h(A, b, BM, M, u, u_r, u_g, u_p, tol, opts, x, s, info);
    bspai_free(A);
    return rc;
}

static int gmres_one(bspai_matrix* A, const bspai_bucketed* BA, const bspai_bucketed* BM, const double* r,
                     bspai_prec_t u_g, bspai_prec_t u_p, const bspai_opts_t* opts, double* d, bspai_stream_t st,
                     bspai_solve_info_t* info) {
    cudaStream_t s = (cudaStream_t)st;
    if (!A || A->magic != kMagicA) return set_error(BSPAI_ERR_INVALID, "bspai_gmres: bad A handle");
    if (!BM || BM->magic != kMagicBM) return set_error(BSPAI_ERR_INVALID, "bspai_gmres: bad M handle");
    if (BM->n != A->n) return set_error(BSPAI_ERR_INVALID, "bspai_gmres: size mismatch");
    if (A->n > 0 && (!r || !d)) return set_error(BSPAI_ERR_INVALID, "bspai_gmres: null vector");
    BSPAI_TRY(check_solver_precs(BSPAI_FP64, BSPAI_DD, u_g, u_p));
    bspai_opts_t o;
    bspai_opts_default(&o);
    if (opts) o = *opts;
    bspai_solve_info_t inf;
    memset(&inf, 0, sizeof inf);
    if (A->n == 0) {
        if (info) *info = inf;
        return BSPAI_OK;
    }
    GmresWork W;
    int rc = W.alloc(A->n, resolve_kmax(&o, A->n), u_g, u_p, o.barrier_timeout_s, o.max_blocks, s);
    W.BA = BA;
    GmresResult gr;
    if (!rc)
        rc = u_g == BSPAI_FP64 ? gmres_run<double>(W, A, BM, r, o.tau, nullptr, d, gr)
                               : gmres_run<float>(W, A, BM, r, o.tau, nullptr, d, gr);
    W.release();
    inf.status = rc ? rc : gr.status;
    inf.ir_steps = 1;
    inf.gmres_iters[0] = gr.k;
    inf.total_iters = gr.k;
    inf.relres[0] = gr.beta > 0 ? gr.res / gr.beta : 0.0;
    if (info) *info = inf;
    if (!rc && gr.status == BSPAI_NONFINITE) return set_error(BSPAI_NONFINITE, "bspai_gmres: non-finite value");
    return rc;
}

int bspai_gmres_plan(int32_t n, bspai_prec_t u_g, int32_t max_blocks, bspai_gmres_plan_t* out) {
    if (!out) return set_error(BSPAI_ERR_INVALID, "bspai_gmres_plan: null out");
    memset(out, 0, sizeof *out);
    if (n < 1) return set_error(BSPAI_ERR_INVALID, "bspai_gmres_plan: n = %d", n);
    if (u_g != BSPAI_FP32 && u_g != BSPAI_FP64) return set_error(BSPAI_ERR_UNSUPPORTED, "u_g must be FP32 or FP64");
    GmresWork W;
    W.n = n;
    W.ug = u_g;
    W.sms = max_blocks > 0 && max_blocks < num_sms() ? max_blocks : num_sms();
    BSPAI_TRY(choose_mgs(W));
    if (W.res_fn) {
        out->kernel = W.res_kind;
        out->per_thread = W.res_per_thread;
        out->block_threads = W.res_bd;
        out->blocks = W.Gr;
        out->poll_bulk = W.bulk;
        return BSPAI_OK;
    }
    int occ = 0, occ2 = 0;
    cudaError_t e = u_g == BSPAI_FP64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mgs<double>, 512, 0)
                                      : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mgs<float>, 512, 0);
    if (!e)
        e = u_g == BSPAI_FP64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, k_gmres_start<double>, 512, 0)
                              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, k_gmres_start<float>, 512, 0);
    if (e) return cuda_error(e, "occupancy", __FILE__, __LINE__);
    occ = occ < occ2 ? occ : occ2;
    out->kernel = 0;
    out->per_thread = 0;
    out->block_threads = 512;
    out->blocks = (occ >= 2 ? 2 : 1) * W.sms;
    return BSPAI_OK;
}

int bspai_gmres(bspai_A_h A, bspai_BM_h BM, const double* r, bspai_prec_t u_g, bspai_prec_t u_p,
                const bspai_opts_t* opts, double* d, bspai_stream_t st, bspai_solve_info_t* info) {
    return gmres_one(A, nullptr, BM, r, u_g, u_p, opts, d, st, info);
}

int bspai_gmres_b(bspai_A_h A, bspai_BM_h A_bucketed, bspai_BM_h BM, const double* r, bspai_prec_t u_g,
                  const bspai_opts_t* opts, double* d, bspai_stream_t st, bspai_solve_info_t* info) {
    if (!A_bucketed || A_bucketed->magic != kMagicBM || (A && A_bucketed->n != A->n))
        return set_error(BSPAI_ERR_INVALID, "bspai_gmres_b: bad bucketed A handle");
    return gmres_one(A, A_bucketed, BM, r, u_g, u_g, opts, d, st, info);
}

}  // extern "C"

// ---------------------------------------------------------------- no-allocation GMRES
// bspai_gmres_noalloc runs exactly the kernels of bspai_gmres, but takes its
// whole workspace (Krylov basis, Hessenberg matrix, rotations, partial sums,
// solver state) from one fixed block of device memory that is part of the
// library image, so it never asks the CUDA runtime for memory.  That block is
// set aside on every GPU that loads the library and stays there until the
// process exits.
namespace bspai {

constexpr size_t kNoallocScratchBytes = 64ull << 20;  // 64 MiB: what a call's problem may take
// beside it, the reductions' buffers (GmresWork::carve) at kmax = kKmaxLimit and any grid
constexpr size_t kNoallocAuxBytes = 1ull << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes + kNoallocAuxBytes];

static std::mutex g_noalloc_mu;
// Device address of the scratch per device ordinal, with the id of the CUDA
// context it was looked up in: after a device reset the module is loaded again
// in a new context (possibly at another address), so a cached address is used
// only while the current context is the one it came from.
struct NoallocAddr {
    unsigned long long ctx_id = 0;
    void* base = nullptr;
};
static NoallocAddr g_noalloc_base[128];

// The current context's process-unique id through the driver entry points
// (the library links the CUDA runtime only); false if they are unavailable.
static bool current_context_id(unsigned long long* id) {
    typedef int (*GetCurrentFn)(void**);
    typedef int (*GetIdFn)(void*, unsigned long long*);
    static GetCurrentFn get_current = nullptr;
    static GetIdFn get_id = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_current = reinterpret_cast<GetCurrentFn>(f);
        f = nullptr;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            get_id = reinterpret_cast<GetIdFn>(f);
    });
    void* ctx = nullptr;
    if (!get_current || !get_id || get_current(&ctx) != 0 || !ctx) return false;
    return get_id(ctx, id) == 0;
}

// The host-side name of a __device__ array is only a stand-in, not a device
// address: the address is looked up with the device current, once per device
// and context (on every call if the driver cannot give the context's id).
static int noalloc_scratch_address(void** out) {
    int dev = 0;
    CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 128) return set_error(BSPAI_ERR_UNSUPPORTED, "bspai_gmres_noalloc: device ordinal %d", dev);
    unsigned long long id = 0;
    const bool have_id = current_context_id(&id);  // false too while no context is current yet
    std::lock_guard<std::mutex> g(g_noalloc_mu);
    NoallocAddr& a = g_noalloc_base[dev];
    if (!have_id || !a.base || a.ctx_id != id) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(no-allocation scratch)", __FILE__, __LINE__);
        a.base = p;
        unsigned long long id2 = 0;  // the lookup made the device's context current
        a.ctx_id = current_context_id(&id2) ? id2 : 0;
    }
    *out = a.base;
    return BSPAI_OK;
}

static size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace bspai

extern "C" {

int bspai_gmres_noalloc(bspai_A_h A, bspai_BM_h BM, const double* r, bspai_prec_t u_g, bspai_prec_t u_p,
                        const bspai_opts_t* opts, double* d, bspai_stream_t st, bspai_solve_info_t* info) {
    cudaStream_t s = (cudaStream_t)st;
    if (!A || A->magic != kMagicA) return set_error(BSPAI_ERR_INVALID, "bspai_gmres_noalloc: bad A handle");
    if (!BM || BM->magic != kMagicBM) return set_error(BSPAI_ERR_INVALID, "bspai_gmres_noalloc: bad M handle");
    if (BM->n != A->n) return set_error(BSPAI_ERR_INVALID, "bspai_gmres_noalloc: size mismatch");
    if (A->n > 0 && (!r || !d)) return set_error(BSPAI_ERR_INVALID, "bspai_gmres_noalloc: null vector");
    BSPAI_TRY(check_solver_precs(BSPAI_FP64, BSPAI_DD, u_g, u_p));
    bspai_opts_t o;
    bspai_opts_default(&o);
    if (opts) o = *opts;
    bspai_solve_info_t inf;
    memset(&inf, 0, sizeof inf);
    if (A->n == 0) {
        if (info) *info = inf;
        return BSPAI_OK;
    }
    // workspace layout inside the fixed scratch block
    GmresWork W;
    W.n = A->n;
    W.kmax = resolve_kmax(&o, A->n);
    W.ug = u_g;
    W.up = u_p;
    W.s = s;
    W.tmo_ns = (unsigned long long)((o.barrier_timeout_s > 0 ? o.barrier_timeout_s : 2.0) * 1e9);
    const size_t es = u_g == BSPAI_FP64 ? 8 : 4;
    W.ldv = ceil_div(W.n, 64) * 64;
    int occ = 0, occ2 = 0;
    cudaError_t e = u_g == BSPAI_FP64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mgs<double>, 512, 0)
                                      : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mgs<float>, 512, 0);
    if (!e)
        e = u_g == BSPAI_FP64 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, k_gmres_start<double>, 512, 0)
                              : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ2, k_gmres_start<float>, 512, 0);
    if (e) return cuda_error(e, "occupancy", __FILE__, __LINE__);
    occ = occ < occ2 ? occ : occ2;
    if (occ < 1) return set_error(BSPAI_ERR_CUDA, "bspai_gmres_noalloc: cooperative kernel does not fit on an SM");
    W.sms = o.max_blocks > 0 && o.max_blocks < num_sms() ? o.max_blocks : num_sms();
    W.G = (occ >= 2 ? 2 : 1) * W.sms;
    const size_t kx = (size_t)W.kmax;
    const size_t sz[9] = {es * (size_t)W.ldv * (kx + 1), es * (size_t)W.ldv, sizeof(GmresState),
                          sizeof(double) * (kx + 1) * kx, sizeof(double) * (kx + 1), sizeof(double) * (kx + 1),
                          sizeof(double) * (kx + 2), sizeof(double) * (kx + 1), sizeof(double) * 4};
    size_t off[10];
    off[0] = 0;
    for (int i = 0; i < 9; ++i) off[i + 1] = align256(off[i] + sz[i]);
    // partial sums and slots of one value per reduction, which had their place in the block
    // before the reductions' own buffers (carve): still counted, so that the limit is where it was
    const size_t need = off[9] + align256(es * 2 * (size_t)W.G) + align256(sizeof(unsigned long long) * 4 * kTagMaxBlocks);
    if (need > kNoallocScratchBytes)
        return set_error(BSPAI_ERR_INVALID,
                         "bspai_gmres_noalloc: n = %d with kmax = %d needs %zu bytes of scratch; the fixed block "
                         "holds %zu bytes (lower kmax or use bspai_gmres)",
                         W.n, W.kmax, need, kNoallocScratchBytes);
    unsigned char* base = nullptr;
    BSPAI_TRY(noalloc_scratch_address(reinterpret_cast<void**>(&base)));
    W.V = base + off[0];
    W.w = base + off[1];
    W.st = reinterpret_cast<GmresState*>(base + off[2]);
    W.H = reinterpret_cast<double*>(base + off[3]);
    W.cs = reinterpret_cast<double*>(base + off[4]);
    W.sn = reinterpret_cast<double*>(base + off[5]);
    W.g = reinterpret_cast<double*>(base + off[6]);
    W.y = reinterpret_cast<double*>(base + off[7]);
    W.norms = reinterpret_cast<double*>(base + off[8]);
    if (W.aux_bytes() > kNoallocAuxBytes)
        return set_error(BSPAI_ERR_INVALID, "bspai_gmres_noalloc: the reductions' buffers need %zu bytes",
                         W.aux_bytes());
    W.carve(base + kNoallocScratchBytes);
    static thread_local HostFlags t_flags;  // ordinary host memory
    W.hflags = &t_flags;
    BSPAI_TRY(choose_mgs(W));
    // the scratch keeps whatever the previous call left there: clear the parts
    // that must start at zero (solver state with its grid barrier, g, the
    // tagged slots that the barrier's sequence numbers restart with)
    CUDA_TRY(cudaMemsetAsync(W.st, 0, sizeof(GmresState), s));
    CUDA_TRY(cudaMemsetAsync(W.aux, 0, W.tagged_bytes(), s));
    BSPAI_TRY(W.zero_pad());
    CUDA_TRY(cudaMemsetAsync(W.g, 0, sizeof(double) * (kx + 2), s));
    GmresResult gr;
    int rc = u_g == BSPAI_FP64 ? gmres_run<double>(W, A, BM, r, o.tau, nullptr, d, gr)
                               : gmres_run<float>(W, A, BM, r, o.tau, nullptr, d, gr);
    inf.status = rc ? rc : gr.status;
    inf.ir_steps = 1;
    inf.gmres_iters[0] = gr.k;
    inf.total_iters = gr.k;
    inf.relres[0] = gr.beta > 0 ? gr.res / gr.beta : 0.0;
    if (info) *info = inf;
    if (!rc && gr.status == BSPAI_NONFINITE) return set_error(BSPAI_NONFINITE, "bspai_gmres_noalloc: non-finite value");
    return rc;
}

}  // extern "C"
