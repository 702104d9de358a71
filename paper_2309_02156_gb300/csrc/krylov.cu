// Krylov solvers on the FP64 system, the mixed-precision outer loop and the
// single-block CG.  The kernel templates live in krylov_kernels.cuh.
#include <math.h>

#include <algorithm>

#include "krylov_kernels.cuh"
#include "cg_kernels.cuh"
#include "resident_cg.cuh"
#include "resident_gmres.cuh"

namespace sa {

int stream_grid(int n) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms > kTeamBlocks) sms = kTeamBlocks;      // what pass_coefficients adds up
    const int need = (n + kStreamBlock - 1) / kStreamBlock;
    return need < sms ? (need > 0 ? need : 1) : sms;
}

// ---------------------------------------------------------------------------
// FP64 residuals from the CSR arrays (outside a solve there is no copy of the
// matrix, and a mixed solve's copy is FP32): pipelined warp tiles on 24 warps per
// SM with one multiply-add per entry; 12 warps, separate multiplications and
// additions and no pipelining before.  1,048,576 rows: 72 -> 44 us.
//
// ||b - A x|| and ||b||; x_override replaces a->x when not NULL; r64 (may be
// NULL) receives the residual.
template <bool REFINE>
__global__ void __launch_bounds__(kSpmvBlock, 1)
residual_kernel(const DevArgs* __restrict__ a, KState* ks, double* r64, double* partial,
                const double* x_override) {
    extern __shared__ unsigned char dsm[];
    __shared__ double scratch[kSpmvWarps * 2];
    __shared__ double red[2];
    const double* x = x_override ? x_override : a->x;
    const double* b = a->b;
    int lo, hi;
    block_rows(a->n, gridDim.x, blockIdx.x, lo, hi);
    double acc[2] = {0.0, 0.0};
    csr_tile_rows<double>(a, a->val64, x, lo, hi, kSpmvWarps, reinterpret_cast<double*>(dsm),
                          &ks->bad_index, [&](int row, double ax) {
                              const double bi = b[row], r = bi - ax;
                              if (REFINE) r64[row] = r;
                              acc[0] = fma(r, r, acc[0]);
                              acc[1] = fma(bi, bi, acc[1]);
                          });
    block_sum<double, 2>(acc, 2, red, scratch);
    if (threadIdx.x < 2) partial[blockIdx.x * 2 + threadIdx.x] = red[threadIdx.x];
    const int which = REFINE ? CNT_REFINE : CNT_RES;
    if (last_block_arrive(&ks->counter[which])) {
        __shared__ double tot[2];
        reduce_blocks(partial, gridDim.x, 2, 2, tot);
        if (threadIdx.x == 0) {
            ks->beta = sqrt(tot[0]);
            ks->bnorm = sqrt(tot[1]);
            if (REFINE) ks->target = a->tol * ks->bnorm;
            else ks->first_relres = rel_residual(ks->beta, ks->bnorm);
            ks->counter[which] = 0;
        }
    }
}

template <bool REFINE>
static void launch_residual(const DevArgs* a, KState* ks, double* r64, double* partial, int nblk,
                            const double* x_override, cudaStream_t st) {
    const size_t smem = sizeof(double) * (size_t)kSpmvWarps * kTile;
    cudaFuncSetAttribute(residual_kernel<REFINE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    residual_kernel<REFINE><<<nblk, kSpmvBlock, smem, st>>>(a, ks, r64, partial, x_override);
}

void launch_residual_norm(const DevArgs* a, KState* ks, double* partial, int nblk,
                          const double* x_override, cudaStream_t st) {
    launch_residual<false>(a, ks, nullptr, partial, nblk, x_override, st);
}

// Mixed precision: r = b - A64 x in FP64 (into r64), beta = ||r||, ||b||.
void launch_refine_residual(const DevArgs* a, KState* ks, double* r64, double* partial, int nblk,
                            cudaStream_t st) {
    launch_residual<true>(a, ks, r64, partial, nblk, nullptr, st);
}

void launch_gmres_start_f64(const DevArgs* a, KState* ks, double* V, size_t, double* partial,
                            int nblk, int first, cudaStream_t st) {
    launch_start<SysF64>(a, ks, V, partial, nblk, first, st);
}
void launch_gmres_cycle_f64(const DevArgs* a, KState* ks, double* V, size_t ldv, double* w,
                            double* partial, int nblk, int R, cudaStream_t st, int* launches,
                            cudaEvent_t* ev, int sweeps, double omega, const double* dinv,
                            double* za, double* zb, double* t, const ChebConfig* cheb, double* dvec) {
    PrecondArgs<double> pc;
    pc.sweeps = sweeps;
    pc.omega = omega;
    pc.dinv = dinv;
    pc.za = za;
    pc.zb = zb;
    pc.t = t;
    if (cheb && cheb->on) {
        pc.cheb = 1;
        pc.tab = cheb->tab;
        pc.dvec = dvec;
    }
    launch_cycle<SysF64>(a, ks, V, ldv, w, partial, nblk, R, st, launches, ev, pc);
}
void launch_cheb_table(double* tab, double lfix, double ratio, int sweeps, cudaStream_t st) {
    cheb_table_kernel<<<1, 32, 0, st>>>(tab, lfix, ratio, sweeps);
}
void launch_diag_inv_f64(const DevArgs* a, double* dinv, int n, cudaStream_t st,
                         unsigned long long* bound) {
    int b = (n + 255) / 256;
    if (b > 152 * 8) b = 152 * 8;
    diag_inv_kernel<SysF64><<<b > 0 ? b : 1, 256, 0, st>>>(a, dinv, bound);
}
// ---------------------------------------------------------------------------
// CSR -> SELL-32 conversion (once per solve; the GMRES cycles then run ~10^3
// products on the same matrix).  Slice s holds rows 32 s .. 32 s + 31; its
// width is its longest row; entry k of row 32 s + l sits at
// off[s] + 32 k + l.  Padding entries have column -1 and value 0.
//
// Slot form: where the rows of a slice share their column offsets (stencils,
// bands), the slice is stored by offset instead: slot k holds one offset and
// the mask of the rows that have an entry at it, values at (W s + k) 32 + l, W
// slots in every slice.  It needs every row's columns to ascend strictly and
// lie in [0, n) (a row's entries then meet their slots in CSR order).  Where the
// whole matrix has few distinct offsets (stencils), all slices use the same
// ascending list, and products need not read the slot words at all.

// The next slot of a slice: the smallest offset column - row that a lane has
// not passed yet (kNoSlot: none), called by all lanes; e is advanced in the
// lanes that have an entry there.  *ok: the lane's columns ascend in range.
constexpr int kNoSlot = 0x7fffffff;
__device__ __forceinline__ int next_slot(const int* __restrict__ colind, int row, int n, int re,
                                         int& e, int& prev, bool& mine, bool& ok) {
    int off = kNoSlot;
    if (e < re) {
        const int c = colind[e];
        ok = ok && c > prev && c < n;
        off = c - row;
        prev = c;
    }
    const int o = __reduce_min_sync(0xffffffffu, ok ? off : -kNoSlot);
    mine = off == o && o != kNoSlot;
    if (mine) ++e;
    else if (off != kNoSlot) prev = -1;
    return o;
}

// Per slice its width (longest row) into width[s]; over the matrix: stats[0]
// the SELL entries (32 x the widths), [1] the widest slice, [2] the most slots
// of a slice (kMaxSlots + 1: no slot form), [3] the largest |offset|; table:
// the distinct offsets of the matrix in any order (kNoSlot: free; the last
// word stays free unless there are more than kMaxSlots).
__device__ __forceinline__ void note_offset(int* table, int o) {
    for (int j = 0; j <= kMaxSlots; ++j) {
        const int v = *(volatile int*)(table + j);
        if (v == o) return;
        if (v == kNoSlot) {
            const int old = atomicCAS(table + j, kNoSlot, o);
            if (old == kNoSlot || old == o) return;
        }
    }
}

__global__ void slot_clear_kernel(unsigned long long* stats, int* table) {
    if (threadIdx.x < 4) stats[threadIdx.x] = 0;
    if (threadIdx.x <= kMaxSlots) table[threadIdx.x] = kNoSlot;
}

__global__ void __launch_bounds__(256)
slot_stats_kernel(const int* __restrict__ rowptr, const int* __restrict__ colind, int n, int nnz,
                  int* width, unsigned long long* stats, int* table) {
    __shared__ int seen[kMaxSlots + 1];
    __shared__ unsigned long long tot[8];
    __shared__ int wmax[8], smax[8], reach[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s = blockIdx.x * 8 + warp, ns = (n + 31) >> 5;
    int len = 0, slots = 0, far = 0;
    if (threadIdx.x <= kMaxSlots) seen[threadIdx.x] = kNoSlot;
    __syncthreads();
    if (s < ns) {
        const int row = s * 32 + lane;
        int rs = 0, re = 0;
        if (row < n) {
            rs = max(0, min(rowptr[row], nnz));
            re = max(rs, min(rowptr[row + 1], nnz));
        }
        len = __reduce_max_sync(0xffffffffu, re - rs);
        int e = rs, prev = -1;
        bool ok = true, mine;
        while (slots <= kMaxSlots) {
            const int o = next_slot(colind, row, n, re, e, prev, mine, ok);
            if (o == kNoSlot) break;
            if (o == -kNoSlot) {
                slots = kMaxSlots + 1;
                break;
            }
            ++slots;
            far = max(far, abs(o));
            if (lane == 0) note_offset(seen, o);
        }
        if (lane == 0) width[s] = len;
    }
    if (lane == 0) {
        tot[warp] = 32ull * len;
        wmax[warp] = len;
        smax[warp] = slots;
        reach[warp] = far;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) {
            tot[0] += tot[w];
            wmax[0] = max(wmax[0], wmax[w]);
            smax[0] = max(smax[0], smax[w]);
            reach[0] = max(reach[0], reach[w]);
        }
        atomicAdd(stats, tot[0]);
        atomicMax(stats + 1, (unsigned long long)wmax[0]);
        atomicMax(stats + 2, (unsigned long long)smax[0]);
        atomicMax(stats + 3, (unsigned long long)reach[0]);
    }
    if (threadIdx.x <= kMaxSlots && seen[threadIdx.x] != kNoSlot) note_offset(table, seen[threadIdx.x]);
}

// Slots by the slice's own offsets in ascending order, or (list.count > 0) by
// the matrix's: slot k of every slice then has offset list.off[k].
template <typename VT>
__global__ void __launch_bounds__(256)
slot_fill_kernel(const int* __restrict__ rowptr, const int* __restrict__ colind,
                 const VT* __restrict__ val, int n, int nnz, int W, const OffsetList list,
                 int2* slot, VT* __restrict__ val_out) {
    const int lane = threadIdx.x & 31;
    const int s = blockIdx.x * 8 + (threadIdx.x >> 5), ns = (n + 31) >> 5;
    if (s >= ns) return;
    const int row = s * 32 + lane;
    int rs = 0, re = 0;
    if (row < n) {
        rs = max(0, min(rowptr[row], nnz));
        re = max(rs, min(rowptr[row + 1], nnz));
    }
    int e = rs, prev = -1;
    bool ok = true, mine;
    for (int k = 0; k < W; ++k) {
        const int at = e;
        int o;
        if (list.count) {
            o = list.off[k];
            mine = e < re && colind[e] - row == o;
            if (mine) ++e;
        } else {
            o = next_slot(colind, row, n, re, e, prev, mine, ok);
        }
        const unsigned mask = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) slot[s * W + k] = mask ? make_int2(o, (int)mask) : make_int2(0, 0);
        val_out[(s * W + k) * 32 + lane] = mine ? val[at] : (VT)0;
    }
}

// Exclusive scan of 32 * width over the slices by one block (off[ns] = total,
// off[ns + 1] = the widest slice).
__global__ void sell_scan_kernel(const int* __restrict__ width, int ns, int* off) {
    __shared__ long long wsum[32];
    __shared__ long long carry;
    __shared__ int wmax;
    if (threadIdx.x == 0) {
        carry = 0;
        wmax = 0;
    }
    __syncthreads();
    for (int s = threadIdx.x; s < ns; s += blockDim.x) atomicMax(&wmax, width[s]);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int base = 0; base < ns; base += blockDim.x) {
        const int s = base + threadIdx.x;
        long long v = s < ns ? 32LL * width[s] : 0;
        long long incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        long long before = 0;
        for (int w = 0; w < warp; ++w) before += wsum[w];
        const long long excl = carry + before + incl - v;
        if (s < ns) off[s] = (int)min(excl, (long long)0x7fffffff);
        __syncthreads();
        if (threadIdx.x == 0) {
            long long tot = 0;
            for (int w = 0; w < nw; ++w) tot += wsum[w];
            carry += tot;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        off[ns] = (int)min(carry, (long long)0x7fffffff);
        off[ns + 1] = wmax;
    }
}

// Every slice padded to width w: off[s] = 32 w s for s <= ns.
__global__ void sell_uniform_kernel(int ns, int w, int* off) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s <= ns; s += gridDim.x * blockDim.x)
        off[s] = 32 * w * s;
}

template <typename VT>
__global__ void sell_fill_kernel(const int* __restrict__ rowptr, const int* __restrict__ colind,
                                 const VT* __restrict__ val, int n, int nnz,
                                 const int* __restrict__ off, int* col_out, VT* val_out) {
    const int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    const int ns = (n + 31) >> 5;
    if (s >= ns) return;
    const int o = off[s], w = (off[s + 1] - o) >> 5;
    const int row = s * 32 + lane;
    int rs = 0, re = 0;
    if (row < n) {
        rs = max(0, min(rowptr[row], nnz));
        re = max(rs, min(rowptr[row + 1], nnz));
    }
    for (int k = 0; k < w; ++k) {
        const int e = rs + k;
        const bool ok = e < re;
        col_out[o + k * 32 + lane] = ok ? colind[e] : -1;
        val_out[o + k * 32 + lane] = ok ? val[e] : (VT)0;
    }
}

void launch_slot_stats(const int* rowptr, const int* colind, int n, int nnz, int* width,
                       SlotStats* out, cudaStream_t st) {
    slot_clear_kernel<<<1, 64, 0, st>>>(out->total, out->table);
    slot_stats_kernel<<<((n + 31) / 32 + 7) / 8, 256, 0, st>>>(rowptr, colind, n, nnz, width,
                                                               out->total, out->table);
}

SlotPlan plan_slots(const SlotStats& st, int n) {
    SlotPlan p = {};
    const long long ns = (n + 31) / 32, total = (long long)st.total[0];
    auto fits = [&](long long w) {
        return w > 0 && w <= kMaxSlots && 32 * ns * w <= total + total / 4 &&
               32 * ns * w < 0x7fffffffLL;
    };
    if (!fits((long long)st.total[2])) return p;
    p.W = (int)st.total[2];
    p.reach = (int)st.total[3];
    int count = 0;
    while (count <= kMaxSlots && st.table[count] != kNoSlot) ++count;
    if (fits(count)) {
        p.W = p.list.count = count;
        for (int k = 0; k < count; ++k) p.list.off[k] = st.table[k];
        std::sort(p.list.off, p.list.off + count);
    }
    return p;
}

void launch_slot_fill_f64(const int* rowptr, const int* colind, const double* val, int n, int nnz,
                          const SlotPlan& p, int2* slot, double* v, cudaStream_t st) {
    slot_fill_kernel<double><<<((n + 31) / 32 + 7) / 8, 256, 0, st>>>(rowptr, colind, val, n, nnz,
                                                                     p.W, p.list, slot, v);
}

void launch_slot_fill_f32(const int* rowptr, const int* colind, const float* val, int n, int nnz,
                          const SlotPlan& p, int2* slot, float* v, cudaStream_t st) {
    slot_fill_kernel<float><<<((n + 31) / 32 + 7) / 8, 256, 0, st>>>(rowptr, colind, val, n, nnz,
                                                                    p.W, p.list, slot, v);
}

void launch_sell_scan(const int* width, int n, int* off, cudaStream_t st) {
    sell_scan_kernel<<<1, 1024, 0, st>>>(width, (n + 31) / 32, off);
}

void launch_sell_uniform(int n, int w, int* off, cudaStream_t st) {
    const int ns = (n + 31) / 32;
    sell_uniform_kernel<<<(ns + 256) / 256, 256, 0, st>>>(ns, w, off);
}

void launch_sell_fill_f64(const int* rowptr, const int* colind, const double* val, int n, int nnz,
                          const int* off, int* col, double* v, cudaStream_t st) {
    const int ns = (n + 31) / 32;
    sell_fill_kernel<double><<<(ns + 7) / 8, 256, 0, st>>>(rowptr, colind, val, n, nnz, off, col, v);
}

void launch_sell_fill_f32(const int* rowptr, const int* colind, const float* val, int n, int nnz,
                          const int* off, int* col, float* v, cudaStream_t st) {
    const int ns = (n + 31) / 32;
    sell_fill_kernel<float><<<(ns + 7) / 8, 256, 0, st>>>(rowptr, colind, val, n, nnz, off, col, v);
}

// rhs32 = r / ||r|| in FP32: the inner equation is A d = r / ||r|| and the
// correction ||r|| d, the same solve in exact arithmetic (the inner tolerance
// is relative), with the FP32 right-hand side and its dot products in range
// whatever the scale of b.
__global__ void refine_scale_kernel(const double* __restrict__ r64, const KState* __restrict__ ks,
                                    float* __restrict__ rhs32, int n) {
    const double inv = 1.0 / ks->beta;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        rhs32[i] = (float)(r64[i] * inv);
}

void launch_refine_scale(const double* r64, const KState* ks, float* rhs32, int n, cudaStream_t st) {
    int b = (n + 255) / 256;
    if (b > 152 * 8) b = 152 * 8;
    refine_scale_kernel<<<b > 0 ? b : 1, 256, 0, st>>>(r64, ks, rhs32, n);
}

// x += ||r|| d (FP64 += the FP32 correction of the inner solve on r / ||r||;
// ||r|| = outer->beta, the residual norm the right-hand side was scaled by).
__global__ void refine_update_kernel(const DevArgs* __restrict__ a, const KState* __restrict__ outer) {
    const int n = a->n;
    const float* d = reinterpret_cast<const float*>(a->d);
    const double beta = outer->beta;
    double* x = a->x;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        x[i] = fma(beta, (double)d[i], x[i]);
}

void launch_refine_update(const DevArgs* a, const KState* outer, cudaStream_t st) {
    refine_update_kernel<<<152 * 8, 256, 0, st>>>(a, outer);
}

__global__ void round_f32_kernel(const double* __restrict__ src, float* __restrict__ dst, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        dst[i] = (float)src[i];
}

void launch_round_f32(const double* src, float* dst, int n, cudaStream_t st) {
    int b = (n + 255) / 256;
    if (b > 152 * 8) b = 152 * 8;
    if (b < 1) b = 1;
    round_f32_kernel<<<b, 256, 0, st>>>(src, dst, n);
}

// ---------------------------------------------------------------------------
// CG in one thread block: the whole iteration runs on the device with block
// barriers only (no launches, no host round trips).  Meant for small and
// medium systems; the batched form runs one such solve per sequence.
template <class Sys>
__device__ __forceinline__ typename Sys::T csr_row(const DevArgs* a, const typename Sys::T* x,
                                                   int i, int n, int nnz, int& bad) {
    using T = typename Sys::T;
    const T* val = Sys::val(a);
    int rs = max(0, min(a->rowptr[i], nnz));
    int re = max(rs, min(a->rowptr[i + 1], nnz));
    T acc = 0;
    for (int e = rs; e < re; ++e) {
        const int c = a->colind[e];
        if ((unsigned)c < (unsigned)n)
            acc += val[e] * x[c];
        else
            bad = 1;
    }
    return acc;
}

template <typename T>
__device__ __forceinline__ T block_total(T v, T* sred) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    v = warp_sum(v);
    __syncthreads();
    if (lane == 0) sred[warp] = v;
    __syncthreads();
    T t = 0;
    for (int w = 0; w < nw; ++w) t += sred[w];
    return t;
}

template <class Sys>
__global__ void __launch_bounds__(1024)
cg_block_kernel(const DevArgs* __restrict__ a, KState* ks, typename Sys::T* r, typename Sys::T* p,
                typename Sys::T* q) {
    using T = typename Sys::T;
    __shared__ T sred[32];
    const int n = a->n, nnz = a->nnz, tid = threadIdx.x, bd = blockDim.x;
    T* x = Sys::x(a);
    const T* b = Sys::rhs(a);
    int bad = 0;
    const bool zero_x = sizeof(T) == 4;      // the FP32 inner solve starts from d = 0
    if (zero_x)
        for (int i = tid; i < n; i += bd) x[i] = 0;
    __syncthreads();
    T rr_l = 0, bb_l = 0;
    for (int i = tid; i < n; i += bd) {
        const T ri = b[i] - (zero_x ? (T)0 : csr_row<Sys>(a, x, i, n, nnz, bad));
        r[i] = ri;
        p[i] = ri;
        rr_l += ri * ri;
        bb_l += b[i] * b[i];
    }
    T rr = block_total(rr_l, sred);
    const T bb = block_total(bb_l, sred);
    const double bnorm = sqrt((double)bb);
    const double target = a->tol * bnorm;
    const double first = rel_residual(sqrt((double)rr), bnorm);
    int it = 0, status = ST_OK;
    if (!isfinite((double)rr) || !isfinite(bnorm)) {
        status = ST_NONFINITE;
    } else if (sqrt((double)rr) > target) {
        for (;;) {
            if (it >= a->max_iters) {
                status = ST_NOT_CONVERGED;
                break;
            }
            __syncthreads();
            T pq_l = 0;
            for (int i = tid; i < n; i += bd) {
                const T qi = csr_row<Sys>(a, p, i, n, nnz, bad);
                q[i] = qi;
                pq_l += p[i] * qi;
            }
            const T pq = block_total(pq_l, sred);
            if (!(pq > 0)) {
                status = isfinite((double)pq) ? ST_BREAKDOWN : ST_NONFINITE;
                break;
            }
            const T alpha = rr / pq;
            T rn_l = 0;
            for (int i = tid; i < n; i += bd) {
                x[i] += alpha * p[i];
                const T ri = r[i] - alpha * q[i];
                r[i] = ri;
                rn_l += ri * ri;
            }
            const T rr_new = block_total(rn_l, sred);
            ++it;
            if (!isfinite((double)rr_new)) {
                status = ST_NONFINITE;
                break;
            }
            if (sqrt((double)rr_new) <= target) {
                __syncthreads();
                T t_l = 0;
                for (int i = tid; i < n; i += bd) {
                    const T ri = b[i] - csr_row<Sys>(a, x, i, n, nnz, bad);
                    r[i] = ri;
                    t_l += ri * ri;
                }
                rr = block_total(t_l, sred);
                if (sqrt((double)rr) <= target) break;
                for (int i = tid; i < n; i += bd) p[i] = r[i];
                continue;
            }
            const T beta = rr_new / rr;
            rr = rr_new;
            for (int i = tid; i < n; i += bd) p[i] = r[i] + beta * p[i];
        }
    }
    if (bad) atomicOr(&ks->bad_index, 1);
    __syncthreads();
    // Final true residual (reported, and used by the refinement loop).
    T f_l = 0;
    for (int i = tid; i < n; i += bd) {
        const T ri = b[i] - csr_row<Sys>(a, x, i, n, nnz, bad);
        f_l += ri * ri;
    }
    const T ff = block_total(f_l, sred);
    if (tid == 0) {
        ks->iters = it;
        ks->status = status;
        ks->bnorm = bnorm;
        ks->target = target;
        ks->first_relres = first;
        ks->beta = sqrt((double)ff);
        ks->finished = 1;
        ks->cycle_over = 1;
    }
}

void launch_cg_block_f64(const DevArgs* a, KState* ks, double* r, double* p, double* q,
                         cudaStream_t st) {
    cg_block_kernel<SysF64><<<1, 1024, 0, st>>>(a, ks, r, p, q);
}
void launch_cg_block_f32(const DevArgs* a, KState* ks, float* r, float* p, float* q,
                         cudaStream_t st) {
    cg_block_kernel<SysF32><<<1, 1024, 0, st>>>(a, ks, r, p, q);
}

bool resident_cg_takes_here(int n, int W, int reach, size_t el) {
    return resident_cg_takes(n, W, reach, el, team_room());
}

bool launch_resident_cg_f64(const DevArgs* a, KState* ks, double* r, double* q, double* x, TeamSlot* slots,
                            int n, int W, int reach, cudaStream_t st) {
    return launch_resident_cg<SysF64>(a, ks, r, q, x, slots, n, W, reach, st);
}
bool launch_resident_cg_f32(const DevArgs* a, KState* ks, float* r, float* q, float* x, TeamSlot* slots,
                            int n, int W, int reach, cudaStream_t st) {
    return launch_resident_cg<SysF32>(a, ks, r, q, x, slots, n, W, reach, st);
}

bool launch_resident_gmres_f64(const DevArgs* a, KState* ks, double* V, size_t ldv, int R,
                               double* kpart, TeamSlot* team, int sweeps, double omega,
                               const double* dinv, double* za, double* zb, double* t,
                               const ChebConfig* cheb, int n, const SlotPlan& plan,
                               cudaStream_t st) {
    const GmresArgs<double> A = {V, ldv, R, kpart, team, sweeps, cheb && cheb->on, omega, dinv, za, zb, t,
                                cheb ? cheb->tab : nullptr};
    return launch_resident_gmres<SysF64>(a, ks, A, n, plan, st);
}

void launch_cgg_start_f64(const DevArgs* a, KState* ks, double* r, double* p, double* partial,
                          int nblk, cudaStream_t st) {
    cgg_start_kernel<SysF64><<<nblk, kStreamBlock, 0, st>>>(a, ks, r, p, partial, 0);
}
void launch_cgg_start_f32(const DevArgs* a, KState* ks, float* r, float* p, float* partial,
                          int nblk, cudaStream_t st) {
    cgg_start_kernel<SysF32><<<nblk, kStreamBlock, 0, st>>>(a, ks, r, p, partial, 1);
}
void launch_cgg_iterations_f64(const DevArgs* a, KState* ks, double* r, double* p, double* q,
                               double* partial, int nblk, int iters, cudaStream_t st) {
    launch_cg_iterations<SysF64>(a, ks, r, p, q, partial, nblk, iters, st);
}
void launch_cgg_iterations_f32(const DevArgs* a, KState* ks, float* r, float* p, float* q,
                               float* partial, int nblk, int iters, cudaStream_t st) {
    launch_cg_iterations<SysF32>(a, ks, r, p, q, partial, nblk, iters, st);
}
void launch_cgg_true_residual_f64(const DevArgs* a, KState* ks, double* r, double* p,
                                  double* partial, int nblk, int check, cudaStream_t st) {
    cgg_true_residual_kernel<SysF64><<<nblk, kStreamBlock, 0, st>>>(a, ks, r, p, partial, check);
}
void launch_cgg_true_residual_f32(const DevArgs* a, KState* ks, float* r, float* p,
                                  float* partial, int nblk, int check, cudaStream_t st) {
    cgg_true_residual_kernel<SysF32><<<nblk, kStreamBlock, 0, st>>>(a, ks, r, p, partial, check);
}

}  // namespace sa
