// spai_team.cuh -- the fixed-pattern SPAI's least-squares solves (u_f = fp32) with
// Abar in registers, a team of TS threads per column k.
//
// Thread t of the team holds rows t, t + TS, ... of Abar = B(I_k, J_k) (NR rows,
// NC columns) and of ebar.  Householder step c forms x . x, x . a_cc and x . ebar
// of the column x = Abar(c:, c) in one reduction: with v = x + s ||x|| e_c
// (s the sign of x_c) the products the reflector needs are v . a = x . a +
// s ||x|| a_c, so the norm and the products do not wait for one another, and a
// column costs |J| reductions instead of |J|^2 / 2.
//   TS = 8, four columns per warp: stencils (|J| <= 12, |I| <= 32).  What bounds
//     these solves is instruction issue; eight lanes with four rows each waste no
//     lanes on |I| = 25 rows and reduce over three levels, not five.
//   TS = 128, one column per block: wide blocks (|J| <= 24, |I| <= 512), whose
//     shared-memory form ran one warp's dependent loads per (column, target) pair.
// A column whose shadow does not fit its instance is listed and left to k_spai.
// Measured (u_f = fp32, kernel time): 7-point 128^3 6.0 -> 2.26 ms, 5-point 1000^2
// 2.1 -> 0.83, random n = 65,536 (|J| = 24, shadows of about 400 rows) 29.6 -> 4.7;
// blocks per SM (launch bounds): narrow 3 (2: 2.83 ms), wide 4 (3: 6.2, 5: 5.8).
#pragma once

#include <climits>
#include <type_traits>
#include <utility>

#include "common.cuh"

namespace bspai {

struct SpaiCounters {
    int n_conv;
    int n_rankdef;
    float max_resid;
    int n_nonfinite;  // entries of M outside the range of u_f (fp16: |m| >= 65520 rounds to Inf)
    int n_left;       // columns left to k_spai
};

template <int TS>
struct SpaiTeam {
    static constexpr int WARPS = TS > 32 ? TS / 32 : 1;  // warps of a team
    static constexpr int LANES = TS < 32 ? TS : 32;      // its lanes in a warp
};

template <class F, int... Cs>
__device__ __forceinline__ void for_each_const(F& f, std::integer_sequence<int, Cs...>) {
    (f(std::integral_constant<int, Cs>{}), ...);
}

// key of the sorted sequence after a compare with the partner's: the smaller or the larger
__device__ __forceinline__ int cmp_pick(int a, int b, bool low) { return low ? min(a, b) : max(a, b); }

// TS: threads of a team; E: candidates per thread (a power of two: TS E slots are sorted);
// NR rows and NC columns of Abar at most TS NR x NC; BD: threads of a block
template <int TS, int E, int NR, int NC, int BD>
struct SpaiShape {
    static constexpr int COLS = BD / TS;       // columns per block
    static constexpr int SLOTS = TS * E;       // candidates
    static constexpr int ROWS = TS * NR;       // rows
    // shared memory of a team: J, dJ, row starts and entry offsets, the distinct rows, Abar
    static constexpr int LD = ROWS + (TS < 32 ? 1 : 0);  // leading dimension of Abar
    static constexpr size_t team_bytes =
        ((size_t)NC * 8 + (size_t)NC * 4 * 2 + (size_t)(NC + 1) * 4 + (size_t)ROWS * 4 + (size_t)LD * NC * 4 + 15) & ~(size_t)15;
    static constexpr size_t smem = team_bytes * COLS;
};

template <int TS, int E, int NR, int NC, int BD, int MINB>
__global__ void __launch_bounds__(BD, MINB) k_spai_team(
    int n, const int32_t* __restrict__ arp, const int32_t* __restrict__ acol, const double* __restrict__ aval,
    const double* __restrict__ d, const int64_t* __restrict__ msptr, const int32_t* __restrict__ mcol,
    const int32_t* __restrict__ mrowlen, float* __restrict__ mval, float* __restrict__ resid, float spai_eps,
    float u_f, SpaiCounters* __restrict__ cnt, int* __restrict__ left) {
    typedef SpaiShape<TS, E, NR, NC, BD> Sh;
    constexpr unsigned full = 0xffffffffu;
    constexpr bool wide = TS > 32;
    constexpr int NW = SpaiTeam<TS>::WARPS, TL = SpaiTeam<TS>::LANES;
    constexpr int NV = NC + 2;  // values of one reduction
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int s_cross[wide ? Sh::SLOTS : 1];               // cross-warp stages of the sort
    __shared__ __align__(16) float s_red[2][wide ? NV : 1][4];  // cross-warp sums, by parity
    __shared__ float s_piv[2][wide ? NV : 1];                   // row c of Abar and ebar
    __shared__ float s_R[wide ? NC : 1][wide ? NC + 1 : 1];
    __shared__ int s_scan[5];
    __shared__ float s_m[wide ? NC : 1];
    __shared__ int s_stat[3];  // this block's converged, rank deficient, non-finite
    __shared__ float s_max;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int t = tid & (TS - 1), tl = lane & (TL - 1);  // thread of the team, its lane in the warp
    const int64_t k = (int64_t)blockIdx.x * Sh::COLS + tid / TS;
    if (tid == 0) {
        s_stat[0] = s_stat[1] = s_stat[2] = 0;
        s_max = 0.0f;
    }
    __syncthreads();  // a narrow team's own barriers join a warp only, and its counts may come at any time
    auto team_sync = [&]() {
        if constexpr (wide) __syncthreads();
        else __syncwarp();
    };
    unsigned char* base = smem + Sh::team_bytes * (tid / TS);
    double* dJ = reinterpret_cast<double*>(base);
    int* J = reinterpret_cast<int*>(dJ + NC);
    int* rbeg = J + NC;
    int* eoff = rbeg + NC;
    int* I = eoff + NC + 1;
    float* Ab = reinterpret_cast<float*>(I + Sh::ROWS);
    auto team_shfl = [&](float v, int src) { return __shfl_sync(full, v, src, TL); };

    // J, d_J and the bounds of rows J of A
    const int nJ = k < n ? mrowlen[k] : 0;
    const int64_t mbase = k < n ? msptr[k >> 5] + (k & 31) : 0;
    bool fits = nJ <= NC;
    int L = 0;
    {
        // NC <= TL (wide) or two rounds of TS lanes (narrow)
        constexpr int RND = wide ? 1 : (NC + TS - 1) / TS;
        int carry = 0;
#pragma unroll
        for (int h = 0; h < RND; ++h) {
            const int q = tl + h * TL;
            int len = 0;
            if ((!wide || w == 0) && q < nJ && q < NC) {
                const int j = mcol[mbase + (int64_t)q * kSlice];
                J[q] = j;
                dJ[q] = d[j];
                const int rb = arp[j];
                rbeg[q] = rb;
                len = arp[j + 1] - rb;
            }
            int inc = len;  // inclusive prefix over the team's lanes
#pragma unroll
            for (int o = 1; o < TL; o <<= 1) {
                const int v = __shfl_up_sync(full, inc, o, TL);
                if (tl >= o) inc += v;
            }
            if ((!wide || w == 0) && q < NC) eoff[q + 1] = carry + inc;
            carry += __shfl_sync(full, inc, TL - 1, TL);
        }
        if ((!wide || w == 0) && tl == 0) eoff[0] = 0;
        team_sync();
        L = nJ > 0 ? eoff[nJ < NC ? nJ : NC] : 0;
    }
    fits = fits && L <= Sh::SLOTS;
    if (!fits) L = 0;
    // the entries of rows J of A: columns, values scaled by d_j (rounded once to u_f), their q;
    // entry e of thread t is number t + TS e
    int ec[E], eq[E];
    float ev[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int idx = t + TS * e;
        ec[e] = INT_MAX;
        eq[e] = 0;
        ev[e] = 0.0f;
        if (idx < L) {
            int lo = 0, hi = nJ;  // the q with eoff[q] <= idx < eoff[q + 1]
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (eoff[mid] <= idx) lo = mid;
                else hi = mid;
            }
            const int p = rbeg[lo] + (idx - eoff[lo]);
            ec[e] = acol[p];
            eq[e] = lo;
            ev[e] = __double2float_rn(__dmul_rn(aval[p], dJ[lo]));
        }
    }
    // bitonic sort of the candidates in registers: thread t holds positions E t .. E t + E - 1
    // (any assignment of the candidates to positions does)
    int key[E];
#pragma unroll
    for (int e = 0; e < E; ++e) key[e] = ec[e];
#pragma unroll
    for (int size = 2; size <= Sh::SLOTS; size <<= 1) {
#pragma unroll
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            if (stride < E) {  // both elements in this thread
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    if (e & stride) continue;
                    const bool up = ((E * t + e) & size) == 0;
                    const int a = key[e], b = key[e | stride];
                    key[e] = cmp_pick(a, b, up);
                    key[e | stride] = cmp_pick(a, b, !up);
                }
            } else if (stride < E * TL) {  // in another lane of the warp
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int b = __shfl_xor_sync(full, key[e], stride / E);
                    const bool up = ((E * t + e) & size) == 0;
                    key[e] = cmp_pick(key[e], b, up == ((E * t & stride) == 0));
                }
            } else {  // in another warp of the team
                __syncthreads();
#pragma unroll
                for (int e = 0; e < E; ++e) s_cross[e * TS + t] = key[e];
                __syncthreads();
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int b = s_cross[e * TS + (t ^ (stride / E))];
                    const bool up = ((E * t + e) & size) == 0;
                    key[e] = cmp_pick(key[e], b, up == ((E * t & stride) == 0));
                }
            }
        }
    }
    // distinct values -> I (ascending)
    int nI;
    {
        int prev = __shfl_up_sync(full, key[E - 1], 1, TL);
        if constexpr (wide) {
            __syncthreads();
            if (lane == 31) s_cross[w] = key[E - 1];
            __syncthreads();
            if (lane == 0 && w > 0) prev = s_cross[w - 1];
        }
        if (t == 0) prev = -1;
        int mine = 0;
        bool fl[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
            const int before = e ? key[e ? e - 1 : 0] : prev;
            fl[e] = key[e] != INT_MAX && key[e] != before;
            mine += fl[e];
        }
        int inc = mine;
#pragma unroll
        for (int o = 1; o < TL; o <<= 1) {
            const int v = __shfl_up_sync(full, inc, o, TL);
            if (tl >= o) inc += v;
        }
        int off = inc - mine;
        nI = __shfl_sync(full, inc, TL - 1, TL);
        if constexpr (wide) {
            if (lane == 31) s_scan[w] = inc;
            __syncthreads();
            int tot = 0;
#pragma unroll
            for (int v = 0; v < NW; ++v) {
                if (v < w) off += s_scan[v];
                tot += s_scan[v];
            }
            nI = tot;
        }
#pragma unroll
        for (int e = 0; e < E; ++e)
            if (fl[e]) {
                if (off < Sh::ROWS) I[off] = key[e];
                ++off;
            }
    }
    fits = fits && nI <= Sh::ROWS;
    const bool work = fits && nJ > 0;
    bool rankdef = work && nI < nJ;
    // Abar in shared memory (its original, for the residual), then this thread's rows
    for (int q = 0; q < NC; ++q)
#pragma unroll
        for (int r = 0; r < NR; ++r) Ab[q * Sh::LD + t + TS * r] = 0.0f;
    team_sync();
    const int nIc = nI < Sh::ROWS ? nI : Sh::ROWS;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        if (t + TS * e < L) {
            int lo = 0, hi = nIc;
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (I[mid] < ec[e]) lo = mid + 1;
                else hi = mid;
            }
            if (lo < Sh::ROWS) Ab[eq[e] * Sh::LD + lo] = ev[e];
        }
    }
    team_sync();
    float a[NR][NC], y[NR];
    float fro = 0.0f;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int row = t + TS * r;
        y[r] = row < nIc && I[row] == (int)k ? 1.0f : 0.0f;
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            a[r][q] = Ab[q * Sh::LD + row];
            fro = __fmaf_rn(a[r][q], a[r][q], fro);
        }
    }
    // Sums over the team.  Narrow: in every thread, by butterflies over its lanes.  Wide:
    // eight values at a time over a warp (9 shuffles), the four warps' sums into
    // s_red[par]; after the barrier that follows, wide_sum(i) is value i in every thread.
    int par = 0;
    auto lane_sum = [&](float v) {
#pragma unroll
        for (int o = TL / 2; o > 0; o >>= 1) v = __fadd_rn(v, __shfl_xor_sync(full, v, o));
        return v;
    };
    auto warp_sums8 = [&](float (&x)[8], int b, int cntv) {
        int off = 16;
#pragma unroll
        for (int h = 4; h >= 1; h >>= 1, off >>= 1) {
            const bool up = (lane & off) != 0;
#pragma unroll
            for (int i = 0; i < h; ++i) {
                const float keep = up ? x[i + h] : x[i], send = up ? x[i] : x[i + h];
                x[i] = __fadd_rn(keep, __shfl_xor_sync(full, send, off));
            }
        }
        x[0] = __fadd_rn(x[0], __shfl_xor_sync(full, x[0], 2));
        x[0] = __fadd_rn(x[0], __shfl_xor_sync(full, x[0], 1));
        const int vi = b + ((lane & 16) ? 4 : 0) + ((lane & 8) ? 2 : 0) + ((lane & 4) ? 1 : 0);
        if ((lane & 3) == 0 && vi < cntv) s_red[par][vi][w] = x[0];
    };
    auto wide_sum = [&](int i) {
        const float4 f = *reinterpret_cast<const float4*>(s_red[par][i]);
        return __fadd_rn(__fadd_rn(f.x, f.y), __fadd_rn(f.z, f.w));
    };
    auto one_sum = [&](float v) {
        v = lane_sum(v);
        if constexpr (wide) {
            if (lane == 0) s_red[par][0][w] = v;
            __syncthreads();
            v = wide_sum(0);
            par ^= 1;
        }
        return v;
    };
    fro = __fsqrt_rn(one_sum(fro));
    float rd[NC];
    const int nS = work ? nJ : 0;  // steps of this column (none: left to k_spai)
    auto step = [&](auto C) {
        constexpr int c = decltype(C)::value;
        constexpr int pr = c / TS, pl = c % TS;  // the thread and register of row c
        rd[c] = 1.0f;
        if constexpr (wide) {
            if (c >= nS) return;  // (the whole block)
        } else {
            if (__all_sync(full, c >= nS)) return;
        }
        const bool act = c < nS && !rankdef;
        float x[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) x[r] = (TS * (r + 1) <= c || (TS * r < c && t + TS * r < c)) ? 0.0f : a[r][c];
        constexpr int m = NC - c;  // values x . a_cc, cc = c .. NC - 1, then x . ebar
        auto target = [&](int r, int i) -> float& { return i < m ? a[r][i < m ? c + i : c] : y[r]; };
        auto partial = [&](int i) {
            float p = 0.0f;
#pragma unroll
            for (int r = 0; r < NR; ++r) p = __fmaf_rn(x[r], target(r, i), p);
            return p;
        };
        float v[wide ? 1 : m + 1];
        float s2, x0;
        if constexpr (wide) {
            if (t == pl) {
#pragma unroll
                for (int i = 0; i <= m; ++i) s_piv[par][i] = target(pr, i);
            }
#pragma unroll
            for (int b = 0; b <= m; b += 8) {
                float p[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) p[i] = b + i <= m ? partial(b + i) : 0.0f;
                warp_sums8(p, b, m + 1);
            }
            __syncthreads();
            s2 = wide_sum(0);
            x0 = s_piv[par][0];
        } else {
#pragma unroll
            for (int i = 0; i <= m; ++i) v[i] = lane_sum(partial(i));
            s2 = v[0];
            x0 = team_shfl(a[pr][c], pl);
        }
        const float sig = __fsqrt_rn(s2);
        const bool ok = act && sig > 0.0f;
        if (act && !(sig > 0.0f)) rankdef = true;
        const float ss = x0 >= 0.0f ? sig : -sig;  // s ||x||
        const float v0 = __fadd_rn(x0, ss);
        const float vtv = __fmul_rn(__fmul_rn(2.0f, sig), __fadd_rn(sig, fabsf(x0)));
        const float twoinv = ok ? __fdiv_rn(2.0f, vtv) : 0.0f;
        if (t == pl) x[pr] = v0;
#pragma unroll
        for (int i = 1; i <= m; ++i) {
            float dot, pv;
            if constexpr (wide) {
                dot = wide_sum(i);
                pv = s_piv[par][i];
            } else {
                dot = v[i];
                pv = team_shfl(target(pr, i), pl);
            }
            const float tau = __fmul_rn(__fmaf_rn(ss, pv, dot), twoinv);
#pragma unroll
            for (int r = 0; r < NR; ++r) {
                if (TS * (r + 1) <= c) continue;  // rows above c
                target(r, i) = __fmaf_rn(-tau, x[r], target(r, i));
            }
        }
        par ^= 1;
        if (ok) rd[c] = -ss;
        if (ok && !(sig > (float)nI * u_f * fro)) rankdef = true;
        if constexpr (wide) {
            if (t == pl) {
#pragma unroll
                for (int i = 1; i < m; ++i) s_R[c][c + i] = a[pr][c + i];
                s_R[c][NC] = y[pr];
            }
        }
    };
    for_each_const(step, std::make_integer_sequence<int, NC>{});
    // back substitution R mbar = (Q^T ebar)(1:|J|)
    float mq[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) mq[q] = 0.0f;
    if constexpr (wide) {
        __syncthreads();
        if (w == 0) {
            // lane i: row i; column by column
            float z = lane < nJ && lane < NC ? s_R[lane][NC] : 0.0f;
            float own = 1.0f;
#pragma unroll
            for (int q = 0; q < NC; ++q)
                if (lane == q) own = rd[q];
#pragma unroll
            for (int c = NC - 1; c >= 0; --c) {
                if (c >= nJ) continue;
                const float mc = __shfl_sync(full, __fdiv_rn(z, own), c);
                if (lane < c) z = __fmaf_rn(-s_R[lane][c], mc, z);
                if (lane == c) s_m[c] = mc;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NC; ++q) mq[q] = q < nJ ? s_m[q] : 0.0f;
    } else {
#pragma unroll
        for (int c = NC - 1; c >= 0; --c) {
            const int pr = c / TS, pl = c % TS;
            float sum = y[pr];
#pragma unroll
            for (int cc = c + 1; cc < NC; ++cc) sum = __fmaf_rn(-a[pr][cc], mq[cc], sum);
            const float mc = team_shfl(__fdiv_rn(sum, rd[c]), pl);
            mq[c] = c < nJ && !rankdef ? mc : 0.0f;
        }
    }
    // sbar = Abar mbar - ebar from the original rows
    float r2 = 0.0f;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int row = t + TS * r;
        float s = row < nIc && I[row] == (int)k ? -1.0f : 0.0f;
#pragma unroll
        for (int q = 0; q < NC; ++q) s = __fmaf_rn(Ab[q * Sh::LD + row], mq[q], s);
        r2 = __fmaf_rn(s, s, r2);
    }
    r2 = one_sum(r2);
    const float res_norm = (work && !rankdef) ? __fsqrt_rn(r2) : 1.0f;
    if (k < n && fits) {
        // M[k, J[q]] = mbar_q d_J[q]  (M = M'^T D)
#pragma unroll
        for (int q = 0; q < NC; ++q) {
            if (q < nJ && t == q % TS) {
                const float mv = rankdef ? 0.0f : __double2float_rn(__dmul_rn((double)mq[q], dJ[q]));
                if (!isfinite(mv)) atomicAdd(&s_stat[2], 1);
                mval[mbase + (int64_t)q * kSlice] = mv;
            }
        }
    }
    if (wide) __syncthreads();
    if (k < n && t == 0) {
        if (fits) {
            resid[k] = res_norm;
            if (res_norm <= spai_eps) atomicAdd(&s_stat[0], 1);
            if (rankdef) atomicAdd(&s_stat[1], 1);
            atomic_max_nonneg(&s_max, res_norm);
        } else {
            left[atomicAdd(&cnt->n_left, 1)] = (int)k;
        }
    }
    // one update per block (one per column on four addresses held the solves up)
    __syncthreads();
    if (tid == 0) {
        if (s_stat[0]) atomicAdd(&cnt->n_conv, s_stat[0]);
        if (s_stat[1]) atomicAdd(&cnt->n_rankdef, s_stat[1]);
        if (s_stat[2]) atomicAdd(&cnt->n_nonfinite, s_stat[2]);
        atomic_max_nonneg(&cnt->max_resid, s_max);
    }
}

}  // namespace bspai
