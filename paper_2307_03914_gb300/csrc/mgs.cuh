// mgs.cuh -- one modified Gram-Schmidt step of GMRES with the new vector on
// chip, the basis taken in groups.
//
// MGS asks for h_i = v_i . (z - sum_{s < i} h_s v_s), one vector after the
// other, which as written costs a grid-wide reduction per vector.  Taken over a
// group of GB consecutive vectors, the same coefficients follow from one
// reduction: with p_t = v_t . z (z as the group finds it) and the group's Gram
// entries L_ts = v_t . v_s (s < t),
//     h_t = p_t - sum_{s < t} L_ts h_s,     i.e.  h = (I + L)^-1 p,
// the triangular form of MGS (Bjorck, "Numerics of Gram-Schmidt
// orthogonalization", 1994; used for GMRES by Swirydowicz et al., "Low
// synchronization Gram-Schmidt and GMRES algorithms", 2021).  It differs from
// the vector-by-vector form by rounding only, and it keeps MGS's property that
// each vector is projected out of what the earlier ones left.  A step then
// needs ceil((j + 1) / GB) + 1 reductions instead of j + 2.  Groups start at
// multiples of GB, so a vector's Gram entries with its group-mates are formed
// once, in the step after the vector was made (it is then the last of the last
// group, in registers with its mates), and kept as the row of (I + L)^-1.
#pragma once

#include "common.cuh"
#include "tags.cuh"

namespace bspai {

struct GmresState {
    int j;        // completed Arnoldi steps (= k)
    int done;     // 1 once converged, broken down, failed or at kmax
    int status;   // BSPAI_OK, BSPAI_TIMEOUT, BSPAI_NONFINITE
    int kmax;
    double beta;  // ||M r||_2 (in u_g)
    double tau;
    double target;  // > 0: stop at |g| <= target instead of the tau test (restarted cycles)
    double res;   // |g_k|
    double hlast;
    GridBar bar;
};

template <typename T>
struct Ar;
template <>
struct Ar<float> {
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
    static __device__ __forceinline__ float sqrt(float a) { return __fsqrt_rn(a); }
    static __device__ __forceinline__ float from(double a) { return __double2float_rn(a); }
};
template <>
struct Ar<double> {
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
    static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
    static __device__ __forceinline__ double sqrt(double a) { return __dsqrt_rn(a); }
    static __device__ __forceinline__ double from(double a) { return a; }
};

// ------------------------------------------------------------------ units
// A thread's rows come in units of VW adjacent rows, the width of one copy
// (VW sizeof(T) = 4, 8 or 16 bytes); fp32 units of two or four rows are kept as
// packed pairs, whose fused multiply-adds are two-lane operations.
template <typename T, int VW>
struct Pack {
    typedef T P;
    static constexpr int N = VW;  // packed values per unit
    static constexpr int L = 1;   // rows per packed value
};
template <>
struct Pack<float, 2> {
    typedef float2 P;
    static constexpr int N = 1, L = 2;
};
template <>
struct Pack<float, 4> {
    typedef float2 P;
    static constexpr int N = 2, L = 2;
};
template <int BYTES>
struct UnitWord;
template <>
struct UnitWord<4> {
    typedef unsigned W;
};
template <>
struct UnitWord<8> {
    typedef uint2 W;
};
template <>
struct UnitWord<16> {
    typedef uint4 W;
};
__device__ __forceinline__ float pk_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double pk_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 pk_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// c - a b: the update of z.  fp32 in one fused operation.  fp64 with product and
// difference rounded apart, as a host code without contraction rounds them: the
// bucketed products round their fp64 operand to fp32, where a last bit that
// differs can come out as another neighbour, 2^-24 away.
__device__ __forceinline__ float pk_nfma(float a, float b, float c) { return __fmaf_rn(-a, b, c); }
__device__ __forceinline__ double pk_nfma(double a, double b, double c) { return __dsub_rn(c, __dmul_rn(a, b)); }
__device__ __forceinline__ float2 pk_nfma(float2 a, float2 b, float2 c) {
    return __ffma2_rn(make_float2(-a.x, -a.y), b, c);
}
__device__ __forceinline__ void pk_zero(float& a) { a = 0.0f; }
__device__ __forceinline__ void pk_zero(double& a) { a = 0.0; }
__device__ __forceinline__ void pk_zero(float2& a) { a = make_float2(0.0f, 0.0f); }
__device__ __forceinline__ void pk_set(float& a, float v) { a = v; }
__device__ __forceinline__ void pk_set(double& a, double v) { a = v; }
__device__ __forceinline__ void pk_set(float2& a, float v) { a = make_float2(v, v); }
__device__ __forceinline__ float pk_sum(float a) { return a; }
__device__ __forceinline__ double pk_sum(double a) { return a; }
__device__ __forceinline__ float pk_sum(float2 a) { return __fadd_rn(a.x, a.y); }
// a / h for many a and one h, from its rounded reciprocal r: the quotient a r
// corrected once by its residual (Markstein, "Computation of elementary functions
// on the IBM RISC System/6000 processor", 1990), three operations where a division
// takes a dozen on the narrow fp64 pipe.  With r = (1 + d1) / h, q = (1 + d2) a r and
// the residual rounded once (d3), all |d| <= u = 2^-24 or 2^-53, what is rounded last
// differs from a / h by (2 u) (2 u) |a / h| at most: the result is within
// 1/2 + 4 u units in the last place, where a division is within 1/2.  That takes
// reciprocal, quotient and residual inside the format's range: h and a (or a = +0)
// between the limits here; any other pair is divided.
template <typename T>
struct Quot {
    T h, r;
    bool mult;
    __device__ __forceinline__ explicit Quot(T h_) : h(h_) {
        const T big = sizeof(T) == 8 ? T(1e100) : T(1e15f);  // 2^332, 2^50
        mult = h > T(1) / big && h < big;
        r = mult ? Ar<T>::div(T(1), h) : T(0);
    }
    // 2^-76 <= |a| < 2^76 (fp64: 2^-680, 2^680), or +0 (-0 would come out +0)
    static __device__ __forceinline__ bool inside(float a) {
        const unsigned b = __float_as_uint(a), x = b << 1, lo = 51u << 24, hi = 203u << 24;
        return x - lo < hi - lo || b == 0;
    }
    static __device__ __forceinline__ bool inside(double a) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(a);
        const unsigned long long x = b << 1, lo = 343ull << 53, hi = 1703ull << 53;
        return x - lo < hi - lo || b == 0;
    }
    __device__ __forceinline__ T operator()(T a) const {
        if (!mult || !inside(a)) return Ar<T>::div(a, h);
        const T q = Ar<T>::mul(a, r);
        return Ar<T>::fma(Ar<T>::fma(-q, h, a), r, q);
    }
};
__device__ __forceinline__ float pk_quot(float a, const Quot<float>& q) { return q(a); }
__device__ __forceinline__ double pk_quot(double a, const Quot<double>& q) { return q(a); }
__device__ __forceinline__ float2 pk_quot(float2 a, const Quot<float>& q) { return make_float2(q(a.x), q(a.y)); }

__device__ __forceinline__ void bar_sync_some(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Sums of N values (a power of two, at most 8) over the lanes of a warp, by a
// butterfly that halves the values it carries: afterwards a[0] of every lane is
// the total of value warp_multi_index<N>(lane).  N = 8: 9 shuffles instead of 40.
template <int N, typename T>
__device__ __forceinline__ void warp_multi_sum(T (&a)[N]) {
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int w = N / 2; w >= 1; w /= 2, off /= 2) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int k = 0; k < w; ++k) {
            const T keep = up ? a[k + w] : a[k];
            const T send = up ? a[k] : a[k + w];
            a[k] = Ar<T>::add(keep, __shfl_xor_sync(0xffffffffu, send, off));
        }
    }
#pragma unroll
    for (; off >= 1; off /= 2) a[0] = Ar<T>::add(a[0], __shfl_xor_sync(0xffffffffu, a[0], off));
}
template <int N>
__device__ __forceinline__ int warp_multi_index(int lane) {
    int v = 0, off = 16;
#pragma unroll
    for (int w = N / 2; w >= 1; w /= 2, off /= 2)
        if (lane & off) v += w;
    return v;
}

// ------------------------------------------------------------------ a group's coefficients
// By one warp, lane t for vector t of the group.  row: its row of the group's
// (I + L)^-1 below the diagonal (zeros at and right of it), kept for the first
// `known` vectors in tri (GB values per vector; read from L2, where another block may
// have written it earlier in the launch).
template <typename T, int GB>
__device__ __forceinline__ void group_rows(T (&row)[GB], const T* tri, int known) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int s = 0; s < GB; ++s) row[s] = (lane < known && s < lane) ? __ldcg(tri + lane * GB + s) : T(0);
}
// h = (I + L)^-1 p for the cnt vectors of a group from the totals tot[t] = p_t;
// in the last group the newest vector's row is not kept yet, and its Gram
// entries q_s = tot[GB + s] give h_c = p_c - sum_s q_s h_s instead.
template <typename T, int GB>
__device__ __forceinline__ T group_coeff(const T (&row)[GB], const T* tot, int cnt, bool last) {
    const int lane = threadIdx.x & 31;
    T h = lane < cnt ? tot[lane] : T(0);
#pragma unroll
    for (int s = 0; s < GB - 1; ++s)
        if (s < lane && lane < cnt) h = Ar<T>::fma(row[s], tot[s], h);
    if (last && cnt > 1) {
        T t = lane < cnt - 1 ? Ar<T>::mul(tot[GB + lane], h) : T(0);
#pragma unroll
        for (int o = GB / 2; o > 0; o >>= 1) t = Ar<T>::add(t, __shfl_xor_sync(0xffffffffu, t, o));
        if (lane == cnt - 1) h = Ar<T>::sub(h, t);
    }
    return h;
}
// the newest vector's row of (I + L)^-1 into out: -(q_s + sum_{u > s} q_u row_u[s])
template <typename T, int GB>
__device__ __forceinline__ void group_new_row(const T (&row)[GB], const T* tot, T (*s_tri)[GB], int cnt, T* out) {
    const int lane = threadIdx.x & 31;
    if (lane < GB) {
#pragma unroll
        for (int s = 0; s < GB; ++s) s_tri[lane][s] = row[s];
    }
    __syncwarp();
    if (lane < cnt - 1) {
        T t = tot[GB + lane];
        for (int u = lane + 1; u < cnt - 1; ++u) t = Ar<T>::fma(tot[GB + u], s_tri[u][lane], t);
        out[lane] = -t;
    }
}

// ------------------------------------------------------------------ the step
constexpr int kMgsMaxVals = 16;  // rows of tagged slots: a group's p and the Gram entries of its last vector

// The bookkeeping of one GMRES run that the step reads and writes
struct MgsIo {
    unsigned long long* tags;  // 2 sets x kMgsMaxVals rows x kTagMaxBlocks slots
    unsigned long long* hq;    // tagged words of the column's coefficients h_{0..j+1,j}
    void* tri;                 // GB values per basis vector: its row of the group's (I + L)^-1, below the diagonal
    GridBar* bar;
    unsigned long long tmo;
    int G;        // blocks that hold rows
    int bulk;     // poll by bulk copies (instances that have them compiled in)
    bool tri_out; // this block writes new rows of tri
    bool hq_out;  // this block publishes the coefficients
};

template <typename T, int VW_, int NU_, int BD_, int GB_, int S_, bool BULK_, bool ZS_>
struct MgsInst {
    typedef T type;
    typedef typename Pack<T, VW_>::P P;
    static constexpr int VW = VW_;      // rows per unit
    static constexpr int NU = NU_;      // units per thread
    static constexpr int BD = BD_;      // threads
    static constexpr int GB = GB_;      // vectors per group
    static constexpr int S = S_;        // stages: vectors copied ahead or held (S >= GB)
    static constexpr bool BULK = BULK_; // able to poll by bulk copies
    static constexpr bool ZS = ZS_;     // z in shared memory (else in registers)
    static constexpr bool SKIP = sizeof(T) == 8;
    static constexpr int UB = VW_ * (int)sizeof(T);
    static constexpr int NPW = 2 * GB;   // warps that poll at most
    static constexpr size_t stage_bytes = (size_t)NU_ * BD_ * UB;
    static constexpr int AHEAD = stage_bytes >= 32768 ? 4 : 0;  // vectors asked into L2 ahead of the stages
    static constexpr int PN = Pack<T, VW_>::N;
    static constexpr int NP = NU_ * PN;  // packed values per thread
    static constexpr size_t smem = stage_bytes * (size_t)(S_ + (ZS_ ? 1 : 0));
    static_assert(S_ >= GB_ && BD_ / 32 >= 2 * GB_ && 2 * GB_ <= kMgsMaxVals, "MGS instance");
};

template <class I>
struct MgsShared {
    typedef typename I::type T;
    T w[I::NPW][32];
    T tot[I::NPW];
    T h[I::GB];
    T tri[I::GB][I::GB];
    int ok;
    alignas(16) unsigned long long slots[I::BULK ? I::NPW * kTagMaxBlocks * TagWords<T>::W : 2];
    alignas(8) uint64_t mbar[I::NPW];  // the warps' polls
    alignas(8) uint64_t full[I::S];    // the stages
};

template <class I>
__device__ __forceinline__ void mgs_shared_init(MgsShared<I>& sh) {  // one thread; a __syncthreads follows
    sh.ok = 1;
#pragma unroll
    for (int s = 0; s < I::S; ++s) mbar_init(&sh.full[s], 1);
    if constexpr (I::BULK) {
#pragma unroll
        for (int w = 0; w < I::NPW; ++w) mbar_init(&sh.mbar[w], 1);
    }
    mbar_init_fence();
}
template <class I>
struct MgsRows {  // the rows of one thread of one block
    int nb;       // rows of the block
    // units of this warp that hold rows; all of them but in fp64, whose pipe is the bound
    __device__ __forceinline__ int units() const {
        if (!I::SKIP) return I::NU;
        const int left = nb - ((int)threadIdx.x & ~31) * I::VW;
        return left <= 0 ? 0 : (left + I::BD * I::VW - 1) / (I::BD * I::VW);
    }
    __device__ __forceinline__ int row(int u) const { return ((int)threadIdx.x + u * I::BD) * I::VW; }
    __device__ __forceinline__ int valid(int u) const {  // bytes of unit u that are rows of the block
        const int left = nb - row(u);
        return (left <= 0 ? 0 : left >= I::VW ? I::VW : left) * (int)sizeof(typename I::type);
    }
};

// unit u of this thread between global memory (the block's first row at p) and registers
template <class I>
__device__ __forceinline__ void unit_load(const MgsRows<I>& R, const typename I::type* p, int u,
                                          typename I::P* out) {
    typedef typename UnitWord<I::UB>::W W;
    const int lr = R.row(u), ok = R.valid(u);
    union {
        W w;
        typename I::type x[I::VW];
        typename I::P p[I::PN];
    } t;
#pragma unroll
    for (int k = 0; k < I::VW; ++k) t.x[k] = 0;
    if (ok == I::UB) {
        t.w = *reinterpret_cast<const W*>(p + lr);
    } else if (ok > 0) {
#pragma unroll
        for (int k = 0; k < I::VW; ++k)
            if (lr + k < R.nb) t.x[k] = p[lr + k];
    }
#pragma unroll
    for (int k = 0; k < I::PN; ++k) out[k] = t.p[k];
}
template <class I>
__device__ __forceinline__ void unit_store(const MgsRows<I>& R, typename I::type* p, int u,
                                           const typename I::P* in) {
    typedef typename UnitWord<I::UB>::W W;
    const int lr = R.row(u), ok = R.valid(u);
    union {
        W w;
        typename I::type x[I::VW];
        typename I::P p[I::PN];
    } t;
#pragma unroll
    for (int k = 0; k < I::PN; ++k) t.p[k] = in[k];
    if (ok == I::UB) {
        *reinterpret_cast<W*>(p + lr) = t.w;
    } else if (ok > 0) {
#pragma unroll
        for (int k = 0; k < I::VW; ++k)
            if (lr + k < R.nb) p[lr + k] = t.x[k];
    }
}

// The block's part of reduction `seq`: this thread's values a[0..N) summed over
// the warp into rows v0 .. v0 + N of sh.w (mgs_arrive finishes them); any = false:
// the warp has no rows and its values are zero
template <class I, int N>
__device__ __forceinline__ void mgs_warp_rows(MgsShared<I>& sh, int v0, typename I::type (&a)[N], bool any) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (any) warp_multi_sum<N>(a);
    if ((lane & (32 / N - 1)) == 0) sh.w[v0 + warp_multi_index<N>(lane)][w] = a[0];
}

// After every warp has left its sums: warp `val` (one that `mine` selects) adds
// its row over the block's warps and publishes it in the grid's slots.  A grid
// of one block has its totals at once.
template <class I>
__device__ __forceinline__ void mgs_arrive(MgsShared<I>& sh, const MgsIo& io, unsigned seq, bool mine) {
    typedef typename I::type T;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __syncthreads();
    if (mine) {
        T t = lane < I::BD / 32 ? sh.w[w][lane] : T(0);
        t = warp_sum(t);
        if (lane == 0) {
            if (io.G == 1) sh.tot[w] = t;
            else
                tag_publish(t, io.tags + ((int64_t)((int)(seq & 1u) * kMgsMaxVals + w) * kTagMaxBlocks + blockIdx.x) *
                                             TagWords<T>::W, seq);
        }
    }
}

// The grid's totals of the rows that `mine` selects, into sh.tot by the warps
// that own them; sh.ok = 0 after a timeout.
template <class I>
__device__ __forceinline__ void mgs_poll(MgsShared<I>& sh, const MgsIo& io, unsigned seq, bool mine,
                                         unsigned& phase) {
    typedef typename I::type T;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (!mine || io.G == 1) return;
    const unsigned long long* row =
        io.tags + (int64_t)((int)(seq & 1u) * kMgsMaxVals + w) * kTagMaxBlocks * TagWords<T>::W;
    T t;
    bool ok;
    if constexpr (I::BULK) {
        ok = io.bulk ? tag_poll_row_bulk<T>(row, seq, io.G, io.bar, io.tmo, &t,
                                            sh.slots + (size_t)w * kTagMaxBlocks * TagWords<T>::W, &sh.mbar[w], phase)
                     : tag_poll_row<T>(row, seq, io.G, io.bar, io.tmo, &t);
    } else {
        ok = tag_poll_row<T>(row, seq, io.G, io.bar, io.tmo, &t);
    }
    if (lane == 0) {
        sh.tot[w] = t;
        if (!ok) *(volatile int*)&sh.ok = 0;
    }
}

// The Gram-Schmidt passes of step j on z (this thread's rows; in registers, or
// for ZS at zs in shared memory) against V's columns 0 .. j, whose rows of this
// block start at Vb.  seq: the reductions done so far; hz: ||z||^2 at the end.
// stage: I::S buffers of I::stage_bytes.  Every thread of every row block calls
// it; false after a timeout (no copy is then in flight).
//
// What bounds it: the basis is read once per step, (j + 1) n values, so the
// bytes bound large n; the reductions' round trip (1.4 us over 64 blocks, about 2
// over 128, more while the memory system is busy) bounds small n.  The copy
// engine brings the next vectors into S stages while the block waits, and the
// group's own vectors stay in registers from the dot products to the update.
// The sweep over a thread's units takes the previous group out of z and forms
// the next group's products together, so the stages' reads overlap the
// arithmetic.  Large chunks hold few stages: there the vectors after them are
// asked into L2 early, and one copy of each refill waits until the reduction
// is over, since copies in flight hold its words up.  Measured per basis
// vector (fits of fixed-step runs, us, one vector per reduction before):
// n = 2,097,152 (128 blocks, groups of 2) 2.66 -> 1.65, 857,375 (64, 2)
// 2.32 -> 1.22, 262,144 (64, 4) 1.37 -> 0.78, 64,000 (64, 8) 1.36 -> 0.37; the
// HBM time of a vector at 2,097,152 is 1.24.  Copies by the threads themselves
// (cp.async) 1.99 at 2,097,152: they queue in front of the reduction's words.
template <class I>
__device__ __forceinline__ bool mgs_passes(MgsShared<I>& sh, const MgsIo& io, const MgsRows<I>& R,
                                           typename I::P* z, unsigned char* stage, unsigned char* zs,
                                           const typename I::type* Vb, int64_t ldv, int j, unsigned hq_tag,
                                           unsigned& seq, unsigned& phase, unsigned& par,
                                           typename I::type& hz) {
    typedef typename I::type T;
    typedef typename I::P P;
    typedef typename UnitWord<I::UB>::W W;
    constexpr int GB = I::GB, S = I::S, NU = I::NU, PN = I::PN, NP = I::NP;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int ng = j / GB + 1;
    const int nu = R.units();
    auto zget = [&](int p) -> P {
        if constexpr (I::ZS) return reinterpret_cast<const P*>(zs)[(tid + (p / PN) * I::BD) * PN + p % PN];
        else return z[p];
    };
    auto zput = [&](int p, P v) {
        if constexpr (I::ZS) reinterpret_cast<P*>(zs)[(tid + (p / PN) * I::BD) * PN + p % PN] = v;
        else z[p] = v;
    };
    // vector i into its stage by the copy engine, and the wait for it
    const unsigned bytes = (unsigned)((R.nb * (int)sizeof(T) + 15) & ~15);
    auto fetch = [&](int i) {
        if (i <= j && bytes && tid == I::BD - 32) {
            mbar_arrive_expect(&sh.full[i % S], bytes);
            bulk_g2s(stage + (size_t)(i % S) * I::stage_bytes, Vb + (int64_t)i * ldv, bytes, &sh.full[i % S]);
        }
    };
    auto ahead = [&](int i) {
        if (i <= j && bytes && tid == I::BD - 32) bulk_prefetch_l2(Vb + (int64_t)i * ldv, bytes);
    };
    auto arrived = [&](int i) {
        if (i <= j && bytes) {
            if (!mbar_wait_bounded(&sh.full[i % S], (par >> (i % S)) & 1u, io.tmo)) *(volatile int*)&sh.ok = 0;
            par ^= 1u << (i % S);
        }
    };
    auto take = [&](const unsigned char* src, int u, P* out) {
        union {
            W w;
            P p[PN];
        } x;
        x.w = *reinterpret_cast<const W*>(src + (size_t)(tid + u * I::BD) * I::UB);
#pragma unroll
        for (int k = 0; k < PN; ++k) out[k] = x.p[k];
    };
#pragma unroll
    for (int i = 0; i < S; ++i) fetch(i);
    // units past the block's rows are never copied: zero in every stage
#pragma unroll
    for (int u = 0; u < NU; ++u)
        if (R.row(u) >= R.nb)
#pragma unroll
            for (int i = 0; i < S; ++i)
                *reinterpret_cast<W*>(stage + (size_t)i * I::stage_bytes + (size_t)(tid + u * I::BD) * I::UB) = W{};
    P v[GB][NP];
    P hm[GB];
#pragma unroll
    for (int t = 0; t < GB; ++t) pk_zero(hm[t]);
    // one sweep over the thread's units per group: the previous group's update of z, the
    // group's vectors into the registers the previous ones leave, and p_t = v_t . z
    for (int g = 0; g < ng; ++g) {
        const int i0 = g * GB;
        const bool last = g == ng - 1;
        const int cnt = last ? j - i0 + 1 : GB;
#pragma unroll
        for (int t = 0; t < GB; ++t) arrived(i0 + t);
        {
            P acc[GB];
            const unsigned char* src[GB];
#pragma unroll
            for (int t = 0; t < GB; ++t) {
                pk_zero(acc[t]);
                src[t] = stage + (size_t)((i0 + t) % S) * I::stage_bytes;
            }
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                if (u < nu) {
                    if (g > 0) {
#pragma unroll
                        for (int k = 0; k < PN; ++k) {
                            P zp = zget(u * PN + k);
#pragma unroll
                            for (int t = 0; t < GB; ++t) zp = pk_nfma(hm[t], v[t][u * PN + k], zp);
                            zput(u * PN + k, zp);
                        }
                    }
#pragma unroll
                    for (int t = 0; t < GB; ++t) {
                        if (I::SKIP && t >= cnt) break;
                        take(src[t], u, &v[t][u * PN]);
#pragma unroll
                        for (int k = 0; k < PN; ++k) {
                            if (t >= cnt) pk_zero(v[t][u * PN + k]);
                            acc[t] = pk_fma(v[t][u * PN + k], zget(u * PN + k), acc[t]);
                        }
                    }
                }
            }
            T a[GB];
#pragma unroll
            for (int t = 0; t < GB; ++t) a[t] = pk_sum(acc[t]);
            mgs_warp_rows<I, GB>(sh, 0, a, nu > 0);
        }
        // the last group (its stages are not refilled): v_j's Gram entries with its mates
        if (last && cnt > 1) {
            P acc[GB];
#pragma unroll
            for (int t = 0; t < GB; ++t) pk_zero(acc[t]);
            const unsigned char* src = stage + (size_t)(j % S) * I::stage_bytes;
#pragma unroll
            for (int u = 0; u < NU; ++u) {
                if (u < nu) {
                    P vj[PN];
                    take(src, u, vj);
#pragma unroll
                    for (int k = 0; k < PN; ++k)
#pragma unroll
                        for (int t = 0; t < GB - 1; ++t)
                            if (!I::SKIP || t < cnt - 1) acc[t] = pk_fma(v[t][u * PN + k], vj[k], acc[t]);
                }
            }
            T a[GB];
#pragma unroll
            for (int t = 0; t < GB; ++t) a[t] = pk_sum(acc[t]);
            mgs_warp_rows<I, GB>(sh, GB, a, nu > 0);
        }
        ++seq;
        const bool mine = w < cnt || (last && w >= GB && w < GB + cnt - 1);
        mgs_arrive<I>(sh, io, seq, mine);
        // every thread has read the group's stages: refill them, in large chunks the last one
        // after the reduction only (a full refill in flight holds the reduction's words up)
        constexpr int late = I::AHEAD ? 1 : 0;
#pragma unroll
        for (int t = 0; t < GB - late; ++t) fetch(i0 + S + t);
        if constexpr (I::AHEAD > 0) {
            if (g == 0) {
#pragma unroll
                for (int t = 0; t < I::AHEAD; ++t) ahead(S + GB - late + t);
            } else {
#pragma unroll
                for (int t = 0; t < GB; ++t) ahead(i0 + S - late + I::AHEAD + t);
            }
        }
        const int npw = last ? I::NPW : GB;
        T rowt[GB];
        if (w == 0)
            group_rows<T, GB>(rowt, reinterpret_cast<const T*>(io.tri) + (int64_t)i0 * GB, last ? cnt - 1 : cnt);
        mgs_poll<I>(sh, io, seq, mine, phase);
        if (w < npw) bar_sync_some(1, npw * 32);
        if (w == 0) {
            const T h = group_coeff<T, GB>(rowt, sh.tot, cnt, last);
            if (lane < GB) sh.h[lane] = lane < cnt ? h : T(0);
            if (lane < cnt && io.hq_out) tag_publish(h, io.hq + (int64_t)(i0 + lane) * TagWords<T>::W, hq_tag);
        }
        __syncthreads();
        if (!*(volatile int*)&sh.ok) {
            // not before the copies in flight have ended
            for (int i = i0 + GB; i < i0 + GB + S - (I::AHEAD ? 1 : 0); ++i) arrived(i);
            __syncthreads();
            return false;
        }
#pragma unroll
        for (int t = 0; t < GB; ++t) pk_set(hm[t], sh.h[t]);
        if constexpr (I::AHEAD > 0) fetch(i0 + S + GB - 1);
        if (last && w == 0 && io.tri_out)
            group_new_row<T, GB>(rowt, sh.tot, sh.tri, cnt, reinterpret_cast<T*>(io.tri) + (int64_t)j * GB);
    }
    // the last group's update, and ||z||^2
    {
        P acc;
        pk_zero(acc);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (p / PN < nu) {
                P zp = zget(p);
#pragma unroll
                for (int t = 0; t < GB; ++t)
                    if (!I::SKIP || t <= j % GB) zp = pk_nfma(hm[t], v[t][p], zp);
                zput(p, zp);
                acc = pk_fma(zp, zp, acc);
            }
        }
        T a[1] = {pk_sum(acc)};
        mgs_warp_rows<I, 1>(sh, 0, a, nu > 0);
        ++seq;
        mgs_arrive<I>(sh, io, seq, w == 0);
        mgs_poll<I>(sh, io, seq, w == 0, phase);
        if (w == 0 && lane == 0 && io.hq_out)
            tag_publish(Ar<T>::sqrt(sh.tot[0]), io.hq + (int64_t)(j + 1) * TagWords<T>::W, hq_tag);
        __syncthreads();
    }
    if (!*(volatile int*)&sh.ok) return false;
    hz = sh.tot[0];
    return true;
}

// ------------------------------------------------------------------ Givens
// The new rotation of step j from the swept column (carry, the entry the
// earlier rotations handed on, and hn = h_{j+1,j}), the update of g and the
// tau test (fp64)
__device__ __forceinline__ void givens_finish(int j, int kmax, double hn, double carry, double* __restrict__ hc,
                                              double* cs, double* sn, double* g, GmresState* st) {
    const double a = carry, b = hn;
    const double rr = __dsqrt_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)));
    double c = 1.0, s = 0.0;
    if (rr != 0.0) {
        c = __ddiv_rn(a, rr);
        s = __ddiv_rn(b, rr);
    }
    cs[j] = c;
    sn[j] = s;
    hc[j] = rr;
    hc[j + 1] = 0.0;
    const double gj = g[j];
    g[j + 1] = __dmul_rn(-s, gj);
    g[j] = __dmul_rn(c, gj);
    const double res = fabs(__dmul_rn(-s, gj));
    const int k = j + 1;
    const bool fin = isfinite(res) && isfinite(hn) && isfinite(rr);
    st->res = res;
    st->hlast = hn;
    st->j = k;
    if (!fin) st->status = BSPAI_NONFINITE;
    const double lvl = st->target > 0.0 ? st->target : __dmul_rn(st->tau, st->beta);
    st->done = (res <= lvl) || hn == 0.0 || k >= kmax || !fin;
}

// The earlier rotations applied by one warp to up to 32 entries of a column (lane t:
// entry h of the column and the rotation c, s that takes it in), carry the entry
// handed on from the ones before.  Only the carry is a chain, -s carry + c h, two
// dependent operations of 64 cycles each on GB300's narrow fp64 pipe; the products
// c h and the rotated entries c carry + s h are formed 32 at a time around it (per
// rotation 175 cycles, against 364 with both rows of a rotation inside the chain).
struct GivensBatch {
    double s[32], m[32];
};
// entries [from, to) of the batch, whose lanes hold c, s, h; lane t keeps the carry its rotation met
__device__ __forceinline__ void givens_chain(GivensBatch& gb, int from, int to, double c, double s, double h,
                                             double& carry, double& met) {
    const int lane = threadIdx.x & 31;
    if (lane >= from && lane < to) {
        gb.s[lane] = -s;
        gb.m[lane] = __dmul_rn(c, h);
    }
    __syncwarp();
#pragma unroll 4
    for (int t = from; t < to; ++t) {
        const double ms = gb.s[t], m = gb.m[t];
        if (lane == t) met = carry;
        carry = __dadd_rn(__dmul_rn(ms, carry), m);
    }
    __syncwarp();
}
__device__ __forceinline__ double givens_entry(double c, double s, double h, double met) {
    return __dadd_rn(__dmul_rn(c, met), __dmul_rn(s, h));
}

// The earlier rotations applied to column j of H by one warp, entry by entry as
// the coefficients arrive in hq (tag: this step's; the words are not overwritten
// within a step, so a warp that starts late misses nothing), then the new
// rotation, g and the tau test.  False after a timeout.
template <typename T>
__device__ bool givens_column(GivensBatch& gb, int j, int kmax, double* __restrict__ H, double* cs, double* sn,
                              double* g, GmresState* st, const unsigned long long* hq, unsigned tag,
                              unsigned long long tmo) {
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    double* __restrict__ hc = H + (int64_t)j * (kmax + 1);
    double carry = 0.0, hn = 0.0;
    for (int base = 0; base <= j + 1; base += 32) {
        const int i = base + lane;
        const int nin = j + 2 - base < 32 ? j + 2 - base : 32;
        // rotation i - 1 takes entry i in
        const bool rot = i >= 1 && i <= j;
        const double ci = rot ? cs[i - 1] : 1.0, si = rot ? sn[i - 1] : 0.0;
        T hv = T(0);
        bool have = lane >= nin;
        int taken = 0;
        double met = 0.0;
        unsigned long long t0 = 0;
        for (int it = 0; taken < nin; ++it) {
            if (!have) have = tag_read(hq + (int64_t)i * TagWords<T>::W, tag, &hv);
            const unsigned pend = ~__ballot_sync(full, have);
            const int upto = pend ? __ffs((int)pend) - 1 : nin;  // entries base .. base + upto are here
            if (upto == taken) {
                int stop = 0;
                if (lane == 0) {
                    const unsigned long long now = globaltimer_ns();
                    if (!t0) t0 = now;
                    if (now - t0 > tmo) {
                        atomicExch(&st->bar.err, 1);
                        stop = 1;
                    } else if ((it & 63) == 63 && *(volatile int*)&st->bar.err) {
                        stop = 1;
                    }
                }
                if (__shfl_sync(full, stop, 0)) return false;
                continue;
            }
            t0 = 0;
            const double hd = (double)hv;
            int to = upto;
            if (base + to == j + 2) {  // the last word is h_{j+1,j}
                --to;
                hn = __shfl_sync(full, hd, to);
            }
            if (base == 0 && taken == 0) {
                carry = __shfl_sync(full, hd, 0);
                taken = 1;
            }
            givens_chain(gb, taken, to, ci, si, hd, carry, met);
            taken = upto;
        }
        if (rot) hc[i - 1] = givens_entry(ci, si, (double)hv, met);
    }
    if (lane == 0) givens_finish(j, kmax, hn, carry, hc, cs, sn, g, st);
    return true;
}

}  // namespace bspai
