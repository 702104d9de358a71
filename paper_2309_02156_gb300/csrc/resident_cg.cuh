// Conjugate gradients with the iteration's vectors on the chip (matrices in
// slot form; see resident.cuh): one launch per solve, two team reductions per
// iteration.  An iteration is one product; when the recursive residual passes
// the test the true residual b - A x is formed and the solve either ends or
// restarts from it; p^T A p <= 0 is a breakdown.
//
// What bounds it: at small sizes the two reductions (0.9 us each in a cluster
// of 16, 2.1 in a grid of 152, plus their FP64 sums), above about 200,000 rows
// in FP64 the FP64 pipe (ten multiply-adds per row, 0.53 T/s: 5 us of the 12 us
// per iteration at 262,144 rows).  Per iteration, before (one block below
// 65,536 rows, three graph kernels above) and now: FP64 4,096 rows 42 -> 5.2 us,
// 262,144 rows 22.4 -> 12.0 us; FP32 32,761 rows 58 -> 3.6 us.
#pragma once

#include "krylov_kernels.cuh"
#include "resident.cuh"

namespace sa {

constexpr int kResThreads = 512;

// r, q and x of rows that do not fit in shared memory lie in rg, qg and xg,
// vectors of the context: the iteration reads and writes 16 bytes at a time, and
// the caller's x is aligned to its element only.
template <class Sys, class Team>
__device__ __forceinline__ void resident_cg(const DevArgs* __restrict__ a, KState* ks,
                                            typename Sys::T* rg, typename Sys::T* qg,
                                            typename Sys::T* xg, Team& tm, const ResLayout& L) {
    using T = typename Sys::T;
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ T scratch[33];
    __shared__ T s_alpha, s_beta, s_rr;
    __shared__ int s_go;
    __shared__ double s_target, s_bnorm, s_first;
    const int n = a->n, W = a->slot_w, ns = (n + 31) >> 5;
    const int tid = threadIdx.x, bd = blockDim.x;
    const int s_lo = min(ns, tm.rank() * L.per), s_hi = min(ns, s_lo + L.per);
    T* x = Sys::x(a);
    const T* b = Sys::rhs(a);
    const bool zero_x = sizeof(T) == 4;        // the FP32 inner solve starts from d = 0
    __shared__ ResBlock<T> B;
    T* const p = reinterpret_cast<T*>(dsm);
    B.setup(p, L, n, s_lo, s_hi, W, a->slot_reach, a->slot_off, a->slot,
            reinterpret_cast<const T*>(a->sell_val), rg, qg, xg);
    const int rows = B.rows, r_lo = B.lo;
    // r = b - A x over the global iterate (p = r on the own rows), |r|^2; all
    // own rows are published.  ldcg: other blocks wrote their rows of x during
    // this launch.
    auto residual = [&](bool start) {
        T acc = 0;
        auto take = [&](int i, T ax) {
            const T ri = b[r_lo + i] - ax;
            B.r[i] = ri;
            if (B.publish) rg[r_lo + i] = ri;
            p[B.pad + i] = ri;
            acc = fma(ri, ri, acc);
        };
        if (start && zero_x) {
            for (int i = tid; i < rows; i += bd) take(i, (T)0);
        } else {
            const int lane = tid & 31, warp = tid >> 5, nw = bd >> 5;
            for (int s = warp; s < B.nsl; s += nw) {
                const int i = s * 32 + lane;
                T ax = 0;
                for (int k = 0; k < W; ++k) {
                    const int2 m = B.slots(p)[s * W + k];
                    if ((m.y >> lane) & 1)
                        ax = fma(B.gval[((size_t)s * W + k) * 32 + lane],
                                 __ldcg(x + r_lo + i + m.x), ax);
                }
                if (i < rows) take(i, ax);
            }
        }
        return acc;
    };
    int it = 0, status = ST_OK;
    T bb = 0;
    for (int i = tid; i < rows; i += bd) {
        const T bi = b[r_lo + i];
        bb = fma(bi, bi, bb);
        B.x[i] = zero_x ? (T)0 : x[r_lo + i];
    }
    tm.total(bb, scratch, [&](T t) {
        s_bnorm = sqrt((double)t);
        s_target = a->tol * s_bnorm;
    });
    tm.total(residual(true), scratch, [&](T t) {
        const double rn = sqrt((double)t);
        s_rr = t;
        s_first = rel_residual(rn, s_bnorm);
        s_go = isfinite((double)t) && isfinite(s_bnorm) ? (rn <= s_target ? 0 : 1) : ST_NONFINITE;
    });
    const double target = s_target, t2 = target * target * (1.0 + 1e-12);
    T rr = s_rr;
    bool known = false;                            // rr is the true residual of the final x
    if (s_go == ST_NONFINITE) status = ST_NONFINITE;
    known = s_go == 0;
    if (s_go == 1 && !tm.late) {
        const int cap_it = a->max_iters;
        B.halo_fresh(p);
        for (;;) {
            if (it >= cap_it) {
                status = ST_NOT_CONVERGED;
                break;
            }
            __syncthreads();
            tm.total(B.template product<sizeof(T) == 4 ? 4 : 2>(p), scratch, [&](T pq) {
                s_alpha = rr / pq;
                s_go = pq > 0 ? 1 : (isfinite((double)pq) ? ST_BREAKDOWN : ST_NONFINITE);
            });
            if (tm.late) break;
            if (s_go != 1) {
                status = s_go;
                break;
            }
            const T alpha = s_alpha;
            tm.total(B.update_r(alpha), scratch, [&](T t) {
                s_beta = t / rr;
                s_rr = t;
                s_go = !isfinite((double)t) ? ST_NONFINITE
                       : ((double)t <= t2 && sqrt((double)t) <= target) ? 0 : 1;
            }, [&](int w0, int step) {             // while the total is on its way
                B.update_x(p, alpha, w0, step);
            });
            if (tm.late) break;
            ++it;
            if (s_go == ST_NONFINITE) {
                status = ST_NONFINITE;
                break;
            }
            if (s_go == 0) {                       // the true residual decides
                for (int i = tid; i < rows; i += bd) x[r_lo + i] = B.x[i];
                tm.total((T)0, scratch, [&](T) {});
                if (tm.late) break;
                tm.total(residual(false), scratch, [&](T t) {
                    s_rr = t;
                    s_go = sqrt((double)t) <= target ? 0 : 1;
                });
                if (tm.late) break;
                rr = s_rr;
                if (s_go == 0) {
                    known = true;
                    break;
                }
                B.halo_fresh(p);
                continue;
            }
            rr = s_rr;
            B.direction(p, s_beta);
        }
    }
    // The final iterate and its true residual (reported, and used by the
    // refinement loop).
    __syncthreads();
    for (int i = tid; i < rows; i += bd) x[r_lo + i] = B.x[i];
    if (!known && !tm.late) {
        tm.total((T)0, scratch, [&](T) {});
        if (!tm.late) tm.total(residual(false), scratch, [&](T t) { s_rr = t; });
        rr = s_rr;
    }
    if (tm.rank() == 0 && tid == 0) {
        ks->iters = it;
        ks->status = tm.late ? ST_TIMEOUT : status;
        ks->bnorm = s_bnorm;
        ks->target = target;
        ks->first_relres = s_first;
        ks->beta = sqrt((double)rr);
        ks->finished = 1;
        ks->cycle_over = 1;
    }
}

template <class Sys>
__global__ void __launch_bounds__(kResThreads, 1)
resident_cg_grid_kernel(const DevArgs* __restrict__ a, KState* ks, typename Sys::T* r,
                        typename Sys::T* q, typename Sys::T* x, TeamSlot* slots, const ResLayout L) {
    __shared__ int bad;
    if (threadIdx.x == 0) bad = 0;
    __syncthreads();
    GridTeam<typename Sys::T> tm;
    tm.slots = slots;
    tm.count = reinterpret_cast<unsigned*>(slots + 2 * kTeamMax);
    tm.bad = &bad;
    resident_cg<Sys>(a, ks, r, q, x, tm, L);
}

template <class Sys>
__global__ void __launch_bounds__(kResThreads, 1)
resident_cg_cluster_kernel(const DevArgs* __restrict__ a, KState* ks, typename Sys::T* r,
                           typename Sys::T* q, typename Sys::T* x, const ResLayout L) {
    __shared__ typename Sys::T box[32];
    ClusterTeam<typename Sys::T> tm;
    tm.box = box;
    tm.sync();                                     // every block has started before a remote store
    resident_cg<Sys>(a, ks, r, q, x, tm, L);
    tm.sync();                                     // no block leaves while another may store to it
}

// What the current device gives a resident team: blocks of a grid, bytes of
// shared memory of a block.  The bytes leave out the kernel's static shared
// memory; they are also its limit, which belongs to the process and is set by
// other threads too: always to the same value, not to a launch's size.
struct TeamRoom {
    int sms;
    size_t budget;
};
static TeamRoom team_room() {
    int dev = 0, sms = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return {sms < kTeamMax ? sms : kTeamMax, (size_t)optin - 2048};
}

// Rows up to which the team is a cluster; the layout of the grid's blocks, at
// least four slices in each: the reductions cost more than rows save.
inline int cluster_rows(size_t el) { return el == 8 ? kClusterCgRows64 : kClusterCgRows32; }
inline bool grid_layout(int n, int W, int reach, size_t el, const TeamRoom& room, ResLayout* L) {
    const int nblk = ((n + 31) / 32 + 3) / 4;
    return res_layout(n, W, reach, nblk < room.sms ? nblk : room.sms, el, room.budget, L);
}

// Whether the streaming kernels are faster although the grid has room.  A block
// forms the direction on the rows within reach too, at 1.0 ns per iteration for
// each of those 2 reach rows in FP64 (256 threads); without them the grid is
// 8.5 us + n / 128 ns ahead of the streaming kernels.  FP64, us per iteration,
// streaming and resident: 262,144 rows, reach 512, 23.3 and 12.1, reach 4,096
// (64^3) 25.0 and 20.5; 360,000 rows, reach 6,000, 26.5 and 26.0; 512,000 rows,
// reach 6,400 (80^3), 31.9 and 32.5; 200,000 rows, reach 10,000, 21.8 and 31.4;
// 1,000,000 rows, reach 1,000, 42.0 and 26.3, reach 8,000, 41.8 and 42.0, reach
// 10,000 (100^3), 57.6 and 65.4; 3,240,000 rows, reach 1,800, 150 and 124.  In
// FP32 the grid is ahead wherever it has room (1,000,000 rows, reach 10,000: 30.2
// and 18.2), as it is of the one-block form that serves fewer rows.
inline bool long_halo(int n, int reach, size_t el) {
    return el == 8 && n >= kGridCgMinRows && 2LL * reach > 8500 + n / 128;
}

// Whether a resident team takes the solve.
inline bool resident_cg_takes(int n, int W, int reach, size_t el, const TeamRoom& room) {
    ResLayout L;
    return (n <= cluster_rows(el) && res_layout(n, W, reach, 16, el, room.budget, &L)) ||
           (!long_halo(n, reach, el) && grid_layout(n, W, reach, el, room, &L));
}

// Launch of one CG solve by a resident team; false when none takes it or the driver
// refuses the launch (the caller takes the streaming kernels).
template <class Sys>
static bool launch_resident_cg(const DevArgs* a, KState* ks, typename Sys::T* r, typename Sys::T* q,
                               typename Sys::T* x, TeamSlot* slots, int n, int W, int reach,
                               cudaStream_t st) {
    using T = typename Sys::T;
    const TeamRoom room = team_room();
    const int ns = (n + 31) / 32;
    // A warp per slice; in FP64 eight warps fill the FP64 pipe and more only
    // add to the reductions.
    auto threads = [](int per) {
        const int t = 32 * per, most = sizeof(T) == 8 ? kResThreads / 2 : kResThreads;
        return t < 128 ? 128 : (t > most ? most : t);
    };
    ResLayout L;
    if (n <= cluster_rows(sizeof(T))) {
        for (int c = 16; c >= 8; c >>= 1) {
            if (!res_layout(n, W, reach, c, sizeof(T), room.budget, &L)) continue;
            auto k = resident_cg_cluster_kernel<Sys>;
            const size_t bytes = res_bytes(L, W, sizeof(T));
            if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room.budget) != cudaSuccess ||
                (c > 8 && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
                cudaGetLastError();
                continue;
            }
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = c;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3(c);
            cfg.blockDim = dim3(threads(L.per));
            cfg.dynamicSmemBytes = bytes;
            cfg.stream = st;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int fit = 0;
            if (cudaOccupancyMaxActiveClusters(&fit, (const void*)k, &cfg) != cudaSuccess || fit < 1) {
                cudaGetLastError();
                continue;
            }
            if (cudaLaunchKernelEx(&cfg, k, a, ks, r, q, x, (const ResLayout)L) == cudaSuccess) return true;
            cudaGetLastError();
        }
    }
    if (long_halo(n, reach, sizeof(T)) || !grid_layout(n, W, reach, sizeof(T), room, &L)) return false;
    const int nblk = (ns + L.per - 1) / L.per;
    auto k = resident_cg_grid_kernel<Sys>;
    const size_t bytes = res_bytes(L, W, sizeof(T));
    int dev = 0, per_sm = 0, coop = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (!coop ||
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)room.budget) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads(L.per), bytes) != cudaSuccess ||
        per_sm * room.sms < nblk) {
        cudaGetLastError();
        return false;
    }
    cudaMemsetAsync(slots, 0, kTeamSlotBytes, st);
    void* args[] = {(void*)&a, (void*)&ks, (void*)&r, (void*)&q, (void*)&x, (void*)&slots, (void*)&L};
    if (cudaLaunchCooperativeKernel((const void*)k, dim3(nblk), dim3(threads(L.per)), args, bytes, st) !=
        cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

}  // namespace sa
