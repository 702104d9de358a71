// Restarted GMRES with the basis, the gathered vectors and (as far as they fit)
// the matrix values on the chip: one cooperative launch per solve in place of
// three or four kernels per Arnoldi step and one per preconditioner sweep.  The steps are
// those of krylov_kernels.cuh: CGS2 on unnormalised columns with sigma_k =
// 1 / ||.||, Givens rotations, true residual at every restart, right
// preconditioning by damped Jacobi sweeps or the Chebyshev recurrence.
//
// A block owns a range of slices (matrices in slot form with common offsets).
// Waits per step: three reductions (h1, h2, ||w||^2) and one plain barrier per
// sweep; the Hessenberg column and its rotations are formed by every block from
// the same totals, so no block waits for another's serial part.
//
// What bounds it (10,000 rows, us per step, FP32 and FP64): the three reductions
// 8.4 and 12, the Hessenberg step 4.5 (one FP64 chain), the passes 3.6 and 9
// (FP64: the adds that reduce 16 to 32 columns over a warp), the product 0.6 and
// 1.4; a sweep costs 2.8 us.
#pragma once

#include <type_traits>

#include "krylov_kernels.cuh"
#include "resident.cuh"

namespace sa {

constexpr int kResRestart = 32;                // longest restart

template <typename T> struct GmresShape;
template <> struct GmresShape<float> { static constexpr int threads = 512; };
// FP64: eight warps fill the FP64 pipe, and the widest pass needs 255 registers.
template <> struct GmresShape<double> { static constexpr int threads = 256; };

// Sizes of the shared arrays (elements unless noted).
struct GmresLayout {
    int per, pad;
    int nval;                  // slices whose matrix values lie in shared memory
};

__host__ __device__ inline size_t gmres_bytes(const GmresLayout& l, int W, int R, int sweeps, size_t el) {
    const size_t rows = 32 * (size_t)l.per, ext = rows + 2 * (size_t)l.pad;
    return el * (ext * (sweeps > 0 ? 3 : 1) + rows * (R + 2) + (size_t)l.nval * 32 * W);
}

inline bool gmres_layout(int n, int W, int reach, int nblk, int R, int sweeps, size_t el,
                         size_t budget, GmresLayout* l) {
    const int ns = (n + 31) / 32;
    l->per = (ns + nblk - 1) / nblk;
    l->pad = (reach + 31) & ~31;
    l->nval = 0;
    if (gmres_bytes(*l, W, R, sweeps, el) > budget) return false;
    const size_t fit = (budget - gmres_bytes(*l, W, R, sweeps, el)) / (el * 32 * W);
    l->nval = (int)(fit < (size_t)l->per ? fit : (size_t)l->per);
    return true;
}

// Rows of one pass over the basis (K <= KM columns, VW rows per thread):
// MODE 0: part_k = sum v_k w.  MODE 1: w -= sum c_k v_k, part_k = sum v_k w.
// MODE 2: v_{j+1} = w - sum c_k v_k, part_0 = its sum of squares.  The warp's
// sums go to wsum[warp * 32 + k].
template <typename T, int KM, int VW, int MODE>
__device__ __forceinline__ void gmres_rows(const T* __restrict__ V, size_t ldv, T* w, T* vout,
                                        T* edge_out, int reach, const T* cf, int K, int rows,
                                        T* wsum) {
    constexpr int KP = KM <= 8 ? 8 : KM <= 16 ? 16 : 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, bd = blockDim.x;
    if (warp * 32 * VW >= rows && warp * 32 >= rows % VW) {   // no row here: no FP64 adds either
        wsum[warp * 32 + lane] = 0;
        return;
    }
    T part[KP];
#pragma unroll
    for (int k = 0; k < KP; ++k) part[k] = 0;
    auto body = [&](int i, auto width) {
        constexpr int N = decltype(width)::value;
        T v[KM][N], r[N];
#pragma unroll
        for (int k = 0; k < KM; ++k)
            if (k < K) {
                const T* at = V + (size_t)k * ldv + i;
                if constexpr (N == 4) {
                    const float4 t = *reinterpret_cast<const float4*>(at);
                    v[k][0] = t.x; v[k][1] = t.y; v[k][2] = t.z; v[k][3] = t.w;
                } else if constexpr (N == 2 && sizeof(T) == 4) {
                    const float2 t = *reinterpret_cast<const float2*>(at);
                    v[k][0] = t.x; v[k][1] = t.y;
                } else {
                    v[k][0] = *at;
                }
            }
#pragma unroll
        for (int e = 0; e < N; ++e) r[e] = w[i + e];
        if constexpr (MODE != 0) {
#pragma unroll
            for (int k = 0; k < KM; ++k)
                if (k < K) {
                    const T c = cf[k];
#pragma unroll
                    for (int e = 0; e < N; ++e) r[e] = fma(-v[k][e], c, r[e]);
                }
            T* out = MODE == 1 ? w : vout;
#pragma unroll
            for (int e = 0; e < N; ++e) {
                out[i + e] = r[e];
                if (MODE == 2 && (i + e < reach || i + e >= rows - reach)) edge_out[i + e] = r[e];
            }
        }
        if constexpr (MODE == 2) {
#pragma unroll
            for (int e = 0; e < N; ++e) part[0] = fma(r[e], r[e], part[0]);
        } else {
#pragma unroll
            for (int k = 0; k < KM; ++k)
                if (k < K)
#pragma unroll
                    for (int e = 0; e < N; ++e) part[k] = fma(v[k][e], r[e], part[k]);
        }
    };
    const int full = rows / VW * VW;
    for (int i = threadIdx.x * VW; i < full; i += bd * VW) body(i, std::integral_constant<int, VW>{});
    for (int i = full + threadIdx.x; i < rows; i += bd) body(i, std::integral_constant<int, 1>{});
    if constexpr (MODE == 2) {
        const T t = warp_total1(part[0]);
        if (lane == 0) wsum[warp * 32] = t;
    } else {
        const T t = warp_reduce_scatter<T, KP>(part);
        if (lane < KP) wsum[warp * 32 + lane] = t;
    }
}

template <typename T, int MODE>
__device__ __forceinline__ void gmres_pass(const T* V, size_t ldv, T* w, T* vout, T* edge_out,
                                           int reach, const T* cf, int K, int rows, T* wsum) {
    constexpr bool F = sizeof(T) == 4;
    if (K <= 8) gmres_rows<T, 8, F ? 4 : 1, MODE>(V, ldv, w, vout, edge_out, reach, cf, K, rows, wsum);
    else if (K <= 16) gmres_rows<T, 16, F ? 2 : 1, MODE>(V, ldv, w, vout, edge_out, reach, cf, K, rows, wsum);
    else if (K <= 24) gmres_rows<T, 24, F ? 2 : 1, MODE>(V, ldv, w, vout, edge_out, reach, cf, K, rows, wsum);
    else gmres_rows<T, 32, 1, MODE>(V, ldv, w, vout, edge_out, reach, cf, K, rows, wsum);
}

// What one solve needs beyond DevArgs.
template <typename T>
struct GmresArgs {
    T* V;                  // (R + 1) columns of ldv (edges only where the basis is on the chip)
    size_t ldv;
    int R;
    T* kpart;              // 2 x 32 x gridDim.x partial sums
    TeamSlot* team;        // counter of the grid team (behind the slots)
    int sweeps, cheb;
    double omega;
    const T* dinv;
    T *za, *zb, *t;
    const double* tab;
};

// Totals of K values per block (bs[k], shared) over the grid into tot[k]
// (shared, FP64); a barrier for the whole team.  K = 0: the barrier alone.
template <typename T>
struct GmresTeam {
    unsigned* count;
    int* bad;
    unsigned epoch = 0;
    __device__ bool late() const { return *bad != 0; }
    __device__ void wait() {
        ++epoch;
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(count) : "memory");
            const unsigned want = epoch * gridDim.x;
            unsigned seen = want - 1;
            for (int left = *bad ? 0 : kTeamPolls; left > 0; --left) {
                asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
                if (team_arrived(seen, want)) break;
            }
            if (!team_arrived(seen, want)) *bad = 1;
            team_fence();
        }
        __syncthreads();
    }
    // wsum: the warps' sums (32 per warp).
    __device__ void totals(int K, const T* wsum, T* kpart, double* tot) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const int nb = gridDim.x;
        T* at = kpart + (size_t)((epoch + 1) & 1) * 32 * nb;
        __syncthreads();
        for (int k = threadIdx.x; k < K; k += blockDim.x) {
            T s = wsum[k];
            for (int v = 1; v < nw; ++v) s += wsum[v * 32 + k];
            at[(size_t)k * nb + blockIdx.x] = s;
        }
        wait();
        constexpr int kMany = 4;             // values whose loads are in flight together
        for (int k0 = warp; k0 < K; k0 += kMany * nw) {
            T u[kMany][kTeamMax / 32];
#pragma unroll
            for (int f = 0; f < kMany; ++f)
#pragma unroll
                for (int q = 0; q < kTeamMax / 32; ++q)
                    u[f][q] = k0 + f * nw < K && lane + 32 * q < nb
                                  ? __ldcg(at + (size_t)(k0 + f * nw) * nb + lane + 32 * q) : (T)0;
#pragma unroll
            for (int f = 0; f < kMany; ++f) {
                if (k0 + f * nw >= K) break;
                const T t = warp_total(u[f]);
                if (lane == 0) tot[k0 + f * nw] = (double)t;
            }
        }
        __syncthreads();
    }
};

template <class Sys, int WM>
__global__ void __launch_bounds__(GmresShape<typename Sys::T>::threads, 1)
resident_gmres_kernel(const DevArgs* __restrict__ a, KState* ks,
                      const GmresArgs<typename Sys::T> A, const GmresLayout L) {
    using T = typename Sys::T;
    constexpr int kMaxK = kResRestart;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ T wsum[(GmresShape<T>::threads / 32) * 32];
    __shared__ T cf[kMaxK];
    __shared__ double tot[kMaxK];
    __shared__ double sig[kMaxK + 1], h[kMaxK + 1], cs[kMaxK], sn[kMaxK], g[kMaxK + 1];
    __shared__ double H[kMaxK * (kMaxK + 1)], rdiag[kMaxK];
    __shared__ double s_hh, s_hn, s_hinv, s_beta, s_bnorm, s_target, s_first;
    __shared__ int s_end, s_status, s_finished, s_iters, s_bad;
    const int tid = threadIdx.x, bd = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = bd >> 5;
    const int n = a->n, W = a->slot_w, ns = (n + 31) >> 5, reach = a->slot_reach, pad = L.pad;
    const int s_lo = min(ns, (int)blockIdx.x * L.per), s_hi = min(ns, s_lo + L.per), nsl = s_hi - s_lo;
    const int lo = s_lo * 32, rows = nsl > 0 ? min(n, s_hi * 32) - lo : 0;
    const int below = nsl > 0 ? lo - max(0, lo - reach) : 0;
    const int halo = nsl > 0 ? below + min(n, lo + rows + reach) - (lo + rows) : 0;
    const int cap = 32 * L.per, ext = cap + 2 * pad;
    T* const x = Sys::x(a);
    const T* const rhs = Sys::rhs(a);
    T* cur = reinterpret_cast<T*>(dsm);
    T* next = cur + ext;
    T* oth = next;                                  // second sweep buffer
    T* const dinv = next + ext;                     // with the neighbours' rows
    if (A.sweeps > 0) next += 2 * (size_t)ext;
    T* const w = next;                              // also the Chebyshev vector during the sweeps
    next += cap;
    T* const Vs = next;
    next += (size_t)cap * (A.R + 1);
    T* const sval = next;
    const T* const gval = reinterpret_cast<const T*>(a->sell_val) + (size_t)s_lo * W * 32;
    const int nval = min(L.nval, nsl);
    GmresTeam<T> tm;
    tm.count = reinterpret_cast<unsigned*>(A.team + 2 * kTeamMax);
    tm.bad = &s_bad;
    if (tid == 0) {
        s_bad = s_finished = s_iters = 0;
        s_status = ST_OK;
    }
    auto halo_at = [&](int j) { return j < below ? j - below : rows + j - below; };
    for (int i = tid; i < ext; i += bd) {
        cur[i] = 0;
        if (A.sweeps > 0) {
            oth[i] = 0;
            dinv[i] = 0;
        }
    }
    for (int i = tid; i < nval * W * 32; i += bd) sval[i] = __ldg(gval + i);
    __syncthreads();
    if (A.sweeps > 0) {
        for (int i = tid; i < rows; i += bd) dinv[pad + i] = A.dinv[lo + i];
        for (int j = tid; j < halo; j += bd) dinv[pad + halo_at(j)] = A.dinv[lo + halo_at(j)];
    }
    int off[WM];
#pragma unroll
    for (int k = 0; k < WM; ++k) off[k] = k < W ? a->slot_off.off[k] : 0;
    // epi(row, (A v)_row) over the own rows, v in the buffer at `from`.
    auto some = [&](const T* v, const T* from, int s, auto count, const auto& epi) {
        constexpr int G = decltype(count)::value;
        T m[G][WM], b[G][WM];
#pragma unroll
        for (int q = 0; q < G; ++q)
#pragma unroll
            for (int k = 0; k < WM; ++k)
                m[q][k] = k < W ? v[((s + q * nw) * W + k) * 32 + lane] : (T)0;
#pragma unroll
        for (int q = 0; q < G; ++q)
#pragma unroll
            for (int k = 0; k < WM; ++k)
                b[q][k] = k < W ? from[pad + (s + q * nw) * 32 + lane + off[k]] : (T)0;
#pragma unroll
        for (int q = 0; q < G; ++q) {
            T ax = 0;
#pragma unroll
            for (int k = 0; k < WM; ++k)
                if (k < W) ax = fma(m[q][k], b[q][k], ax);
            const int i = (s + q * nw) * 32 + lane;
            if (i < rows) epi(i, ax);
        }
    };
    auto product = [&](const T* from, const auto& epi) {
        constexpr int G = sizeof(T) == 4 && WM <= 5 ? 2 : 1;
        int s = warp;
        for (; s + (G - 1) * nw < nval; s += G * nw) some(sval, from, s, std::integral_constant<int, G>{}, epi);
        for (; s < nval; s += nw) some(sval, from, s, std::integral_constant<int, 1>{}, epi);
        for (; s + (G - 1) * nw < nsl; s += G * nw) some(gval, from, s, std::integral_constant<int, G>{}, epi);
        for (; s < nsl; s += nw) some(gval, from, s, std::integral_constant<int, 1>{}, epi);
    };
    auto fetch = [&](T* to, const T* from) {           // neighbours' rows of a global vector
        for (int j = tid; j < halo; j += bd) to[pad + halo_at(j)] = __ldcg(from + lo + halo_at(j));
    };
    auto column = [&](int j) { return Vs + (size_t)j * cap; };
    // cur = M^{-1} (s u) with its halo, u the own rows of the global vector ug
    // (own rows read at u).
    auto precondition = [&](const T* u, const T* ug, T s) {
        const T om = A.cheb ? (T)A.tab[1] : (T)A.omega;
        for (int i = tid; i < rows; i += bd) {
            const T z = (om * dinv[pad + i]) * (s * u[i]);
            cur[pad + i] = z;
            if (A.cheb) w[i] = z;
        }
        for (int j = tid; j < halo; j += bd) {
            const int i = pad + halo_at(j);
            cur[i] = (om * dinv[i]) * (s * __ldcg(ug + lo + halo_at(j)));
        }
        for (int sw = 1; sw < A.sweeps; ++sw) {
            __syncthreads();
            T* const out = (sw & 1) ? A.za : A.zb;
            T* const to = oth;
            const T* const from = cur;
            auto put = [&](int i, T z) {
                to[pad + i] = z;
                if (i < reach || i >= rows - reach) out[lo + i] = z;
            };
            if (A.cheb) {
                const T c1 = (T)A.tab[2 * sw], c2 = (T)A.tab[2 * sw + 1];
                product(from, [&](int i, T ax) {
                    const T dn = c1 * w[i] + c2 * (dinv[pad + i] * (s * u[i] - ax));
                    w[i] = dn;
                    put(i, from[pad + i] + dn);
                });
            } else {
                product(from, [&](int i, T ax) {
                    put(i, from[pad + i] + (om * dinv[pad + i]) * (s * u[i] - ax));
                });
            }
            tm.wait();
            fetch(to, out);
            oth = cur;
            cur = to;
        }
        __syncthreads();
    };
    // Residual of the iterate into column 0, its norm, and whether the solve is over.
    auto start = [&](bool first) {
        const bool zero_x = first && sizeof(T) == 4;
        T* const v0 = column(0);
        T* const v0g = A.V + lo;
        T acc[2] = {0, 0};
        auto take = [&](int i, T ax) {
            const T bi = rhs[lo + i], r = bi - ax;
            v0[i] = r;
            if (i < reach || i >= rows - reach) v0g[i] = r;
            if (zero_x) x[lo + i] = 0;
            acc[0] = fma(r, r, acc[0]);
            acc[1] = fma(bi, bi, acc[1]);
        };
        if (zero_x) {
            for (int i = tid; i < rows; i += bd) take(i, (T)0);
        } else {
            __syncthreads();
            for (int i = tid; i < rows; i += bd) cur[pad + i] = x[lo + i];
            fetch(cur, x);
            __syncthreads();
            product(cur, take);
        }
        const T t0 = warp_total1(acc[0]), t1 = warp_total1(acc[1]);
        if (lane == 0) {
            wsum[warp * 32] = t0;
            wsum[warp * 32 + 1] = t1;
        }
        tm.totals(2, wsum, A.kpart, tot);
        if (tid == 0) {
            const double beta = sqrt(tot[0]);
            if (first) {
                s_bnorm = sqrt(tot[1]);
                s_target = a->tol * s_bnorm;
                s_first = rel_residual(beta, s_bnorm);
            }
            s_beta = beta;
            g[0] = beta;
            sig[0] = beta > 0.0 ? 1.0 / beta : 0.0;
            if (!isfinite(beta)) {
                s_status = ST_NONFINITE;
                s_finished = 1;
            } else if (beta <= s_target) {
                s_status = ST_OK;
                s_finished = 1;
            } else if (s_iters >= a->max_iters) {
                s_status = ST_NOT_CONVERGED;
                s_finished = 1;
            }
        }
        __syncthreads();
    };
    __syncthreads();
    start(true);
    while (!s_finished && !tm.late()) {
        int K = 0;                                     // steps of this cycle
        for (int j = 0; j < A.R; ++j) {
            const T* const u = column(j);
            const T* const ug = A.V + (size_t)j * A.ldv;
            T scale = (T)sig[j];
            if (A.sweeps > 0) {
                precondition(u, ug, scale);
                scale = (T)1;
            } else if (j == 0) {
                for (int i = tid; i < rows; i += bd) cur[pad + i] = u[i];
                fetch(cur, ug);
                __syncthreads();
            }
            product(cur, [&](int i, T ax) { w[i] = ax * scale; });
            __syncthreads();
            K = j + 1;
            const T* const V = column(0);
            const size_t ldv = cap;
            gmres_pass<T, 0>(V, ldv, w, nullptr, nullptr, reach, cf, K, rows, wsum);
            tm.totals(K, wsum, A.kpart, tot);
            if (tid < K) {
                const double hk = sig[tid] * tot[tid];
                h[tid] = hk;
                cf[tid] = (T)(sig[tid] * hk);
            }
            __syncthreads();
            gmres_pass<T, 1>(V, ldv, w, nullptr, nullptr, reach, cf, K, rows, wsum);
            tm.totals(K, wsum, A.kpart, tot);
            if (tid < K) {
                const double hk = sig[tid] * tot[tid];
                h[tid] += hk;
                cf[tid] = (T)(sig[tid] * hk);
            }
            __syncthreads();
            gmres_pass<T, 2>(V, ldv, w, column(K), A.V + (size_t)K * A.ldv + lo, reach, cf, K,
                                  rows, wsum);
            tm.totals(1, wsum, A.kpart, tot);
            if (tm.late()) break;
            // Hessenberg column, rotations and the end of the cycle, as in
            // arnoldi_finish: ||h||^2 and the rotation chain in warp 0, ||w|| in
            // warp 1.
            if (warp == 0) {
                double v = lane < K ? h[lane] * h[lane] : 0.0;
                v = warp_total1(v);
                if (lane == 0) {
                    s_hh = v;
                    double carry = h[0];
                    for (int i = 0; i < j; ++i) {
                        const double hi1 = h[i + 1];
                        h[i] = cs[i] * carry + sn[i] * hi1;
                        carry = -sn[i] * carry + cs[i] * hi1;
                    }
                    h[j] = carry;
                }
            } else if (warp == 1) {
                if (lane == 0) {
                    const double hn = sqrt(tot[0]);
                    s_hn = hn;
                    s_hinv = hn > 0.0 ? 1.0 / hn : 0.0;
                }
            } else if (A.sweeps == 0 && K < A.R) {
                // The other warps fetch the next column meanwhile.
                const T* const v = column(K);
                const T* const vg = A.V + (size_t)K * A.ldv + lo;
                for (int i = tid - 64; i < rows; i += bd - 64) cur[pad + i] = v[i];
                for (int q = tid - 64; q < halo; q += bd - 64) cur[pad + halo_at(q)] = __ldcg(vg + halo_at(q));
            }
            __syncthreads();
            if (tid == 0) {
                // hypot without its scaling where the squares are in range (its
                // FP64 instructions took longer than the step's reductions).
                const double hn = s_hn, av = h[j], sq = fma(av, av, hn * hn);
                const double rr = sq > 1e-200 && sq < 1e200 ? sqrt(sq) : hypot(av, hn);
                double c = 1.0, sv = 0.0;
                if (rr != 0.0) {
                    const double rinv = 1.0 / rr;
                    c = av * rinv;
                    sv = hn * rinv;
                }
                cs[j] = c;
                sn[j] = sv;
                h[j] = rr;
                const double gj = g[j], gj1 = -sv * gj;
                g[j + 1] = gj1;
                g[j] = c * gj;
                s_iters += 1;
                sig[j + 1] = s_hinv;
                const bool nonfinite = !isfinite(hn) || !isfinite(gj1);
                const bool happy = hn * hn <= 1e-28 * (s_hh + hn * hn);
                s_end = nonfinite || happy || fabs(gj1) <= s_target || s_iters >= a->max_iters ||
                        j == A.R - 1;
                if (nonfinite) {
                    s_status = ST_NONFINITE;
                    s_finished = 1;
                }
            }
            __syncthreads();
            for (int i = tid; i <= j; i += bd) H[j * (kMaxK + 1) + i] = h[i];
            __syncthreads();
            if (s_end) break;
        }
        if (s_finished || tm.late()) break;
        // R y = g by warp 0 (lane l owns row l), sigma_k y_k into cf.
        if (warp == 0) {
            const bool sing = lane < K && H[lane * (kMaxK + 1) + lane] == 0.0;
            if (__any_sync(0xffffffffu, sing)) {
                if (lane == 0) {
                    s_status = ST_BREAKDOWN;
                    s_finished = 1;
                }
            } else {
                if (lane < K) rdiag[lane] = 1.0 / H[lane * (kMaxK + 1) + lane];
                __syncwarp();
                double acc = lane < K ? g[lane] : 0.0, y = 0.0;
                for (int i = K - 1; i >= 0; --i) {
                    const double yi = __shfl_sync(0xffffffffu, acc, i) * rdiag[i];
                    if (lane == i) y = yi;
                    if (lane < i) acc -= H[i * (kMaxK + 1) + lane] * yi;
                }
                if (lane < K) cf[lane] = (T)(sig[lane] * y);
            }
        }
        __syncthreads();
        if (s_finished) break;
        // x += V y, or x += M^{-1} (V y).
        auto combine = [&](int i) {
            T acc = 0;
            const T* const V = column(0) + i;
            for (int l = 0; l < K; ++l) acc = fma(V[(size_t)l * cap], cf[l], acc);
            return acc;
        };
        if (A.sweeps > 0) {
            for (int i = tid; i < rows; i += bd) A.t[lo + i] = combine(i);
            tm.wait();
            precondition(A.t + lo, A.t, (T)1);
            for (int i = tid; i < rows; i += bd) x[lo + i] += cur[pad + i];
        } else {
            for (int i = tid; i < rows; i += bd) x[lo + i] += combine(i);
        }
        tm.wait();                                     // x complete before it is gathered
        if (tm.late()) break;
        start(false);
    }
    if (blockIdx.x == 0 && tid == 0) {
        ks->iters = s_iters;
        ks->status = tm.late() ? ST_TIMEOUT : s_status;
        ks->beta = s_beta;
        ks->bnorm = s_bnorm;
        ks->target = s_target;
        ks->first_relres = s_first;
        ks->finished = 1;
        ks->cycle_over = 1;
    }
}

// Whether the streaming kernels are faster although the size fits.  Every block
// fetches the neighbours' rows of every product's vector, 2 reach of them and one
// product per sweep and one for the step: 1.4 to 2 us for 1,000 rows of reach.
// What a step has to spend on that: in FP64 9 us where a block has at most eight
// slices (one pass of its warps), 3 us up to sixteen (1.6 with more than
// five offsets), above that nothing once there are sweeps; in FP32 1.5 us.  Per step of full cycles, streaming and
// resident, us (five offsets): FP64 10,000 rows, reach 4,000, 35.5 and 33.8;
// 56,000 rows, reach 1,500, 37.6 and 35.6; 85,184 rows, reach 1,936 (44^3), 40.4
// and 45.5; four sweeps 22,500 rows, reach 1,500, 48.4 and 47.4, reach 3,000 48.4
// and 58.7; eight sweeps 10,000 rows, reach 1,000, 61.1 and 60.3, reach 2,000 61.2
// and 76.3; 77,000 rows, reach 277, 69.2 and 72.4; 56,000 rows, reach 236, nine
// offsets, 65.6 and 74.9; 92,000 rows, reach 303, 73.3 and 84.9.  FP32 22,500 rows, reach 1,500, 20.1 and 21.5, reach 3,000 20.2 and
// 25.1; eight sweeps 36,864 rows, reach 192, 39.5 and 42.2, reach 1,000 39.8 and
// 52.3, 10,000 rows, reach 4,000, 39.3 and 98.8.  A cycle that ends early costs the
// streaming kernels the launches of the rest: eight iterations with eight sweeps,
// 56,000 rows, reach 236, FP64 860 and 613, FP32 703 and 525, so a step may cost up
// to a twentieth more.
inline bool long_fetch(int W, int reach, int sweeps, int per, size_t el) {
    const long long rows = (sweeps + 1LL) * reach;
    if (el == 4) return rows > (sweeps > 0 ? 2500 : 1800);
    return rows > (per <= 8 ? 9000 : per <= 16 ? (W <= 5 ? 3000 : 1600) : sweeps <= 1 ? 1000 : 0);
}

// Launch of a whole GMRES solve by a resident grid; false when the size does not
// fit or the driver refuses the launch (the caller takes the cycle graph).
template <class Sys>
static bool launch_resident_gmres(const DevArgs* a, KState* ks, const GmresArgs<typename Sys::T>& A,
                                  int n, const SlotPlan& plan, cudaStream_t st) {
    using T = typename Sys::T;
    if (plan.list.count == 0 || plan.W > 9 || A.R > kResRestart) return false;
    int dev = 0, sms = 0, optin = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop) return false;
    if (sms > kTeamMax) sms = kTeamMax;
    const int ns = (n + 31) / 32;
    int nblk = (ns + 3) / 4;
    if (nblk > sms) nblk = sms;
    GmresLayout L;
    const size_t budget = (size_t)optin - 20480;   // less the static arrays; also the kernel's limit
    if (!gmres_layout(n, plan.W, plan.reach, nblk, A.R, A.sweeps, sizeof(T), budget, &L)) return false;
    if (n > (sizeof(T) == 8 ? kResGmresRows64 : A.sweeps > 0 ? kResGmresRows32Pre : kResGmresRows32) ||
        long_fetch(plan.W, plan.reach, A.sweeps, L.per, sizeof(T)))
        return false;
    nblk = (ns + L.per - 1) / L.per;
    int threads = 32 * L.per;
    threads = threads < 256 ? 256 : (threads > GmresShape<T>::threads ? GmresShape<T>::threads : threads);
    using Kern = void (*)(const DevArgs*, KState*, const GmresArgs<T>, const GmresLayout);
    const Kern k = plan.W <= 5 ? resident_gmres_kernel<Sys, 5> : resident_gmres_kernel<Sys, 9>;
    const size_t bytes = gmres_bytes(L, plan.W, A.R, A.sweeps, sizeof(T));
    int per_sm = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, bytes) != cudaSuccess ||
        per_sm * sms < nblk) {
        cudaGetLastError();
        return false;
    }
    cudaMemsetAsync(A.team, 0, kTeamSlotBytes, st);
    GmresArgs<T> args_copy = A;
    void* args[] = {(void*)&a, (void*)&ks, (void*)&args_copy, (void*)&L};
    if (cudaLaunchCooperativeKernel((const void*)k, dim3(nblk), dim3(threads), args, bytes, st) !=
        cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

}  // namespace sa
