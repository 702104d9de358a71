// Thread-block teams that keep an iteration's vectors on the chip.
//
// A team is a cooperative grid of up to one block per SM, or one thread-block
// cluster.  Block k owns a contiguous range of 32-row slices; the vector that
// products gather lies in its shared memory with the rows within the matrix's
// reach (the largest |column - row|) on both sides, and other blocks' rows
// reach it through global memory at the team's reductions.  A reduction is
// also the team's barrier: every block posts its partial sum and waits for
// all of them, so all blocks hold bitwise the same total (blocks in order) and
// take the same branches.
#pragma once

#include "common.cuh"
#include "internal.h"

namespace sa {

constexpr int kTeamMax = kTeamBlocks;      // blocks of a grid team
constexpr int kTeamPolls = 1 << 21;        // bound of a wait (each poll is an L2 round trip)

// One posted partial: the value's bits and the reduction's number.
struct __align__(16) TeamSlot {
    unsigned long long bits, epoch;
};

__device__ __forceinline__ void team_post(TeamSlot* s, unsigned long long bits,
                                          unsigned long long epoch) {
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\t"
                 "st.relaxed.gpu.global.b128 [%0], t;\n\t}"
                 :: "l"(s), "l"(bits), "l"(epoch) : "memory");
}
__device__ __forceinline__ void team_peek(const TeamSlot* s, unsigned long long& bits,
                                          unsigned long long& epoch) {
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\t"
                 "mov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(bits), "=l"(epoch) : "l"(s) : "memory");
}

// Whether a counter that reads `seen` has reached `want`.  Both count modulo 2^32
// (a long solve passes it) and lie less than 2^31 apart: no block is more than
// one wait ahead of another.
__host__ __device__ inline bool team_arrived(unsigned seen, unsigned want) {
    return (int)(seen - want) >= 0;
}

__device__ __forceinline__ unsigned long long to_bits(double v) {
    return (unsigned long long)__double_as_longlong(v);
}
__device__ __forceinline__ unsigned long long to_bits(float v) { return __float_as_uint(v); }
__device__ __forceinline__ void from_bits(unsigned long long b, double& v) {
    v = __longlong_as_double((long long)b);
}
__device__ __forceinline__ void from_bits(unsigned long long b, float& v) {
    v = __uint_as_float((unsigned)b);
}

__device__ __forceinline__ void team_fence() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Sum of N values per lane over the warp.  FP64: on this GPU a warp-wide FP64
// add holds a sub-partition's FP64 pipe for 64 cycles, so a butterfly of five
// costs more than the rest of a reduction.  The values are added as integers
// instead, aligned to the largest exponent with kHead bits of headroom (exact
// addition; each value is rounded once, at 2^(kHead - 63) of the largest), and
// the sum is rounded to FP64 once.  Infinities and NaN take the butterfly.
template <int N>
__device__ __forceinline__ double warp_total(const double (&v)[N]) {
    constexpr int kHead = 5 + (N > 4 ? 3 : N > 2 ? 2 : N > 1 ? 1 : 0) + 1;   // with the sign
    constexpr int kUp = 63 - 53 - kHead + 1;          // mantissas move up by this
    int ex[N], top = 0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        ex[q] = (__double2hiint(v[q]) >> 20) & 0x7ff;
        top = max(top, ex[q]);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (top == 0x7ff) {
        double t = v[0];
#pragma unroll
        for (int q = 1; q < N; ++q) t += v[q];
        return warp_sum(t);
    }
    top = max(top, 1);
    long long sum = 0;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const long long bits = __double_as_longlong(v[q]);
        long long m = (bits & 0xfffffffffffffll) | (ex[q] ? 0x10000000000000ll : 0ll);
        const int d = top - max(ex[q], 1);
        m <<= kUp;
        m = d < 62 ? (m + ((1ll << d) >> 1)) >> d : 0ll;
        sum += bits < 0 ? -m : m;
    }
    const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)sum & 0x3ffffffu);
    const unsigned mi = __reduce_add_sync(0xffffffffu, (unsigned)(sum >> 26) & 0x3ffffffu);
    const int hi = __reduce_add_sync(0xffffffffu, (int)(sum >> 52));
    sum = (long long)lo + ((long long)mi << 26) + ((long long)hi << 52);
    if (sum == 0) return 0.0;
    // sum x 2^(top - 1075 - kUp) rounded to nearest (halves up in magnitude).
    unsigned long long u = sum < 0 ? (unsigned long long)(-sum) : (unsigned long long)sum;
    const int lz = __clzll((long long)u);
    u <<= lz;
    unsigned long long f = (u >> 11) + ((u >> 10) & 1);    // 2^52 <= f <= 2^53
    int e = top - kUp + 11 - lz;                           // exponent field of f's leading bit
    if (f >> 53) {
        f >>= 1;
        ++e;
    }
    if (e >= 0x7ff || e < 1)                               // out of the normal range
        return ldexp((double)sum, top - 1075 - kUp);
    const unsigned long long r =
        (f & 0xfffffffffffffull) | ((unsigned long long)e << 52) | (sum < 0 ? 1ull << 63 : 0ull);
    return __longlong_as_double((long long)r);
}
template <int N>
__device__ __forceinline__ float warp_total(const float (&v)[N]) {
    float t = v[0];
#pragma unroll
    for (int q = 1; q < N; ++q) t += v[q];
    return warp_sum(t);
}
template <typename T>
__device__ __forceinline__ T warp_total1(T v) {
    const T a[1] = {v};
    return warp_total(a);
}

// Grid team: a counter and slots (2 x gridDim.x) in global memory, zeroed
// before the launch.  One lane per block polls the counter and the slots are
// read once it is full: polling the slots themselves saves an L2 read but
// loads them with 152 x 5 requests per round (measured per reduction on 152
// blocks, FP32: 2.1 us with the counter, 2.4 to 4.9 polling the slots).
template <typename T>
struct GridTeam {
    TeamSlot* slots;
    unsigned* count;
    int* bad;                              // shared, 0 at the start; stays 1 once a wait ran out
    unsigned epoch = 0;
    bool late = false;                     // a wait ran out (uniform over the block)
    __device__ int rank() const { return blockIdx.x; }
    __device__ int size() const { return gridDim.x; }
    // Sum over the team; `fin(total)` runs in thread 0 before the block goes on.
    // Writes before it (any thread's) are visible to the team after it.
    // meanwhile(first, step) is work on other data that the block's warps
    // first, first + step, .. do while the total is on its way.
    template <typename F>
    __device__ void total(T v, T* scratch /* 33 */, const F& fin) {
        total(v, scratch, fin, [](int, int) {});
    }
    template <typename F, typename G>
    __device__ void total(T v, T* scratch /* 33 */, const F& fin, const G& meanwhile) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        ++epoch;
        v = warp_total1(v);
        if (lane == 0) scratch[warp] = v;
        __syncthreads();
        if (warp == 0) {
            const int nb = gridDim.x;
            const T b = warp_total1(lane < nw ? scratch[lane] : (T)0);
            TeamSlot* s = slots + (epoch & 1) * nb;
            if (lane == 0) {
                team_post(s + blockIdx.x, to_bits(b), epoch);
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" :: "l"(count) : "memory");
                const unsigned want = epoch * (unsigned)nb;
                unsigned seen = want - 1;
                for (int left = *bad ? 0 : kTeamPolls; left > 0; --left) {
                    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
                    if (team_arrived(seen, want)) break;
                }
                if (!team_arrived(seen, want)) *bad = 1;
                team_fence();
            }
            __syncwarp();
            T u[kTeamMax / 32];
#pragma unroll
            for (int q = 0; q < kTeamMax / 32; ++q) {
                unsigned long long bits = 0, e;
                if (lane + 32 * q < nb) team_peek(s + lane + 32 * q, bits, e);
                from_bits(bits, u[q]);
            }
            const T t = warp_total(u);
            team_fence();
            if (lane == 0) fin(t);
        } else {
            meanwhile(warp - 1, nw - 1);
        }
        __syncthreads();
        late = *bad != 0;
    }
};

// Cluster team: one cluster is the whole grid; partials go to every block's
// shared memory, the wait is the hardware's cluster barrier.
template <typename T>
struct ClusterTeam {
    T* box;                                // shared: 2 x 16
    int par = 0;
    bool late = false;
    __device__ static unsigned rank_() {
        unsigned r;
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
        return r;
    }
    __device__ static unsigned size_() {
        unsigned r;
        asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
        return r;
    }
    __device__ int rank() const { return (int)rank_(); }
    __device__ int size() const { return (int)size_(); }
    __device__ static void put(double* p, unsigned rank, double v) {
        asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\t"
                     "st.shared::cluster.f64 [a], %2;\n\t}"
                     :: "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank), "d"(v) : "memory");
    }
    __device__ static void put(float* p, unsigned rank, float v) {
        asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, %1;\n\t"
                     "st.shared::cluster.f32 [a], %2;\n\t}"
                     :: "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank), "f"(v) : "memory");
    }
    __device__ static void sync() {
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    }
    template <typename F>
    __device__ void total(T v, T* scratch, const F& fin) {
        total(v, scratch, fin, [](int, int) {});
    }
    template <typename F, typename G>
    __device__ void total(T v, T* scratch, const F& fin, const G& meanwhile) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
        const int nb = size();
        v = warp_total1(v);
        if (lane == 0) scratch[warp] = v;
        __syncthreads();
        if (warp == 0) {
            const T b = warp_total1(lane < nw ? scratch[lane] : (T)0);
            if (lane < nb) put(box + par * 16 + rank_(), (unsigned)lane, b);
        } else {
            meanwhile(warp - 1, nw - 1);
        }
        sync();
        if (warp == 0) {
            const T t = warp_total1(lane < nb ? box[par * 16 + lane] : (T)0);
            if (lane == 0) fin(t);
        }
        __syncthreads();
        par ^= 1;
    }
};

// Where a block's data lies: the gathered vector p always in shared memory with
// `pad` rows of its neighbours (or zeros) on both sides, the others there as
// far as they fit, else in the solve's global vectors.
struct ResLayout {
    int per;           // slices of a block
    int pad;           // reach rounded up to 32
    int r_in, q_in, x_in;
    int nval;          // slices whose matrix values are kept in shared memory
};

__host__ __device__ inline size_t res_bytes(const ResLayout& l, int W, size_t el) {
    const size_t rows = 32 * (size_t)l.per;
    return (2 * (size_t)l.pad + rows * (size_t)(1 + l.r_in + l.q_in + l.x_in) +
            (size_t)l.nval * 32 * W) * el + 8 * (size_t)l.per * W;
}

// Largest layout within `budget` bytes for `nblk` blocks; false if the gathered
// vector alone does not fit.
__host__ __device__ inline bool res_layout(int n, int W, int reach, int nblk, size_t el,
                                           size_t budget, ResLayout* l) {
    const int ns = (n + 31) / 32;
    l->per = (ns + nblk - 1) / nblk;
    l->pad = (reach + 31) & ~31;
    l->r_in = l->q_in = l->x_in = l->nval = 0;
    if (res_bytes(*l, W, el) > budget) return false;
    l->r_in = 1;
    if (res_bytes(*l, W, el) > budget) l->r_in = 0;
    l->q_in = 1;
    if (res_bytes(*l, W, el) > budget) l->q_in = 0;
    l->x_in = 1;
    if (res_bytes(*l, W, el) > budget) l->x_in = 0;
    const size_t used = res_bytes(*l, W, el), slice = el * 32 * W;
    const size_t fit = (budget - used) / slice;
    l->nval = (int)(fit < (size_t)l->per ? fit : (size_t)l->per);
    return true;
}

template <typename T> struct Vec16;
template <> struct Vec16<float> {
    static constexpr int N = 4;
    using V = float4;
    __device__ static void load(const float* p, float (&o)[4]) {
        const float4 v = *reinterpret_cast<const float4*>(p);
        o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
    }
    __device__ static void store(float* p, const float (&o)[4]) {
        *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
    }
};
template <> struct Vec16<double> {
    static constexpr int N = 2;
    using V = double2;
    __device__ static void load(const double* p, double (&o)[2]) {
        const double2 v = *reinterpret_cast<const double2*>(p);
        o[0] = v.x; o[1] = v.y;
    }
    __device__ static void store(double* p, const double (&o)[2]) {
        *reinterpret_cast<double2*>(p) = make_double2(o[0], o[1]);
    }
};

// One block's part of a CG iteration: its rows [lo, lo + rows) of the system.
// The struct lies in shared memory and each phase copies what it uses, so that
// no phase holds another's registers (64 per thread at 1,024 threads).  Vector
// phases read and write 16 bytes per thread; the last rows % 2 or % 4 go one by
// one.  `p` is the start of the dynamic shared memory in every call: p[pad + i]
// is row lo + i, the other vectors' [i].
template <typename T>
struct ResBlock {
    using X = Vec16<T>;
    int lo, rows, reach, pad, W, nsl, nval;
    int below, halo;                     // neighbours' rows needed: before, in all
    int val_at, slot_at;                 // values (elements) and slot words (bytes) from p on
    T *r, *q, *x;
    const T* gval;                       // values of the block's slices
    T* rg;                               // residual of the whole system, for the neighbours
    bool publish;                        // r lies in shared memory: edge rows go to rg
    OffsetList list;

    // Splits the shared memory (thread 0), copies the block's slot words and
    // values and clears p.  All threads; ends with a barrier.
    __device__ void setup(T* p, const ResLayout& L, int n, int s_lo, int s_hi, int W_, int reach_,
                          const OffsetList& list_, const int2* slot, const T* val, T* r_g, T* q_g,
                          T* x_g) {
        const int cap = 32 * L.per, n_p = cap + 2 * L.pad;
        if (threadIdx.x == 0) {
            W = W_;
            reach = reach_;
            pad = L.pad;
            list = list_;
            nsl = s_hi - s_lo;
            lo = s_lo * 32;
            rows = nsl > 0 ? min(n, s_hi * 32) - lo : 0;
            const int e_lo = max(0, lo - reach), e_hi = min(n, lo + rows + reach);
            below = nsl > 0 ? lo - e_lo : 0;
            halo = nsl > 0 ? below + e_hi - (lo + rows) : 0;
            T* next = p + n_p;
            rg = r_g;
            publish = L.r_in != 0;
            r = L.r_in ? next : r_g + lo;
            next += L.r_in ? cap : 0;
            q = L.q_in ? next : q_g + lo;
            next += L.q_in ? cap : 0;
            x = L.x_in ? next : x_g + lo;
            next += L.x_in ? cap : 0;
            val_at = (int)(next - p);
            slot_at = (int)((val_at + (size_t)L.nval * 32 * W) * sizeof(T));
            gval = val + (size_t)s_lo * W * 32;
            nval = min(L.nval, nsl);
        }
        for (int i = threadIdx.x; i < n_p; i += blockDim.x) p[i] = 0;
        __syncthreads();
        int2* sslot = slots(p);
        for (int i = threadIdx.x; i < nsl * W_; i += blockDim.x) sslot[i] = __ldg(slot + s_lo * W_ + i);
        T* sval = p + val_at;
        const T* gv = gval;
        const int nv = nval * W_ * 32;
        for (int i = threadIdx.x * X::N; i < nv; i += blockDim.x * X::N) {
            T v[X::N];
            X::load(gv + i, v);
            X::store(sval + i, v);
        }
        __syncthreads();
    }
    __device__ int2* slots(T* p) const {
        return reinterpret_cast<int2*>(reinterpret_cast<unsigned char*>(p) + slot_at);
    }

    __device__ void halo_fresh(T* p) const {       // p = r outside the own rows
        const int h = halo, b = below, l = lo, m = rows, at = pad;
        const T* g = rg;
        for (int j = threadIdx.x; j < h; j += blockDim.x) {
            const int i = j < b ? j - b : m + j - b;
            p[at + i] = __ldcg(g + l + i);
        }
    }
    __device__ T update_r(T alpha) const {     // r -= alpha q; returns this thread's part of r.r
        T acc = 0;
        T* const rr = r;
        const T* const qq = q;
        T* const out = rg + lo;
        const int m = rows, full = m / X::N * X::N, near = publish ? reach : 0;
        for (int i = threadIdx.x * X::N; i < full; i += blockDim.x * X::N) {
            T a[X::N], b[X::N];
            X::load(rr + i, a);
            X::load(qq + i, b);
#pragma unroll
            for (int u = 0; u < X::N; ++u) {
                a[u] = fma(-alpha, b[u], a[u]);
                acc = fma(a[u], a[u], acc);
            }
            X::store(rr + i, a);
            if (i < near || (near && i + X::N > m - near)) X::store(out + i, a);
        }
        for (int i = full + threadIdx.x; i < m; i += blockDim.x) {
            const T a = fma(-alpha, qq[i], rr[i]);
            acc = fma(a, a, acc);
            rr[i] = a;
            if (near) out[i] = a;
        }
        return acc;
    }
    __device__ void update_x(T* p, T alpha, int w0, int step) const {   // x += alpha p, by warps w0, w0 + step, ..
        T* const xx = x;
        const T* const pp = p + pad;
        const int m = rows, full = m / X::N * X::N;
        const int t = w0 * 32 + (threadIdx.x & 31), hop = step * 32 * X::N;
        int i = t * X::N;
        constexpr int kFly = 4;          // x may lie in global memory: several loads in flight
        for (; i + (kFly - 1) * hop < full; i += kFly * hop) {
            T a[kFly][X::N];
#pragma unroll
            for (int f = 0; f < kFly; ++f) X::load(xx + i + f * hop, a[f]);
#pragma unroll
            for (int f = 0; f < kFly; ++f) {
                T b[X::N];
                X::load(pp + i + f * hop, b);
#pragma unroll
                for (int u = 0; u < X::N; ++u) a[f][u] = fma(alpha, b[u], a[f][u]);
                X::store(xx + i + f * hop, a[f]);
            }
        }
        for (; i < full; i += hop) {
            T a[X::N], b[X::N];
            X::load(xx + i, a);
            X::load(pp + i, b);
#pragma unroll
            for (int u = 0; u < X::N; ++u) a[u] = fma(alpha, b[u], a[u]);
            X::store(xx + i, a);
        }
        for (i = full + t; i < m; i += step * 32) xx[i] = fma(alpha, pp[i], xx[i]);
    }
    // p = r + beta p on the own rows and the halo; the neighbours' rows of r are
    // on their way while the own rows are formed.
    __device__ void direction(T* p, T beta) const {
        constexpr int kAhead = sizeof(T) == 4 ? 2 : 4;
        T ahead[kAhead];
        const int bd = blockDim.x, h = halo, nb = below, m = rows;
        const T* const g = rg + lo;
        const T* const rr = r;
        T* const pp = p + pad;
        const bool few = h <= kAhead * bd;
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int j = threadIdx.x + u * bd;
            ahead[u] = few && j < h ? __ldcg(g + (j < nb ? j - nb : m + j - nb)) : (T)0;
        }
        const int full = m / X::N * X::N;
        for (int i = threadIdx.x * X::N; i < full; i += bd * X::N) {
            T a[X::N], b[X::N];
            X::load(pp + i, a);
            X::load(rr + i, b);
#pragma unroll
            for (int u = 0; u < X::N; ++u) a[u] = fma(beta, a[u], b[u]);
            X::store(pp + i, a);
        }
        for (int i = full + threadIdx.x; i < m; i += bd) pp[i] = fma(beta, pp[i], rr[i]);
        if (few) {
#pragma unroll
            for (int u = 0; u < kAhead; ++u) {
                const int j = threadIdx.x + u * bd;
                if (j < h) {
                    T* at = pp + (j < nb ? j - nb : m + j - nb);
                    *at = fma(beta, *at, ahead[u]);
                }
            }
        } else {
            for (int j = threadIdx.x; j < h; j += bd) {
                const int i = j < nb ? j - nb : m + j - nb;
                pp[i] = fma(beta, pp[i], __ldcg(g + i));
            }
        }
    }
    // G slices of the product q = A p, `step` apart: values at v, rows of p at pp.
    template <int WM, int G>
    __device__ __forceinline__ static void some(const T* v, const T* pp, T* qq, int s, int step,
                                                int Wn, int m, const int (&off)[WM], T& acc) {
        const int lane = threadIdx.x & 31;
        T a[G][WM], b[G][WM];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const T* at = v + (s + g * step) * Wn * 32 + lane;
#pragma unroll
            for (int k = 0; k < WM; ++k) a[g][k] = k < Wn ? at[k * 32] : (T)0;
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const T* at = pp + (s + g * step) * 32 + lane;
#pragma unroll
            for (int k = 0; k < WM; ++k) b[g][k] = k < Wn ? at[off[k]] : (T)0;
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int i = (s + g * step) * 32 + lane;
            T ax = 0;
#pragma unroll
            for (int k = 0; k < WM; ++k)
                if (k < Wn) ax = fma(a[g][k], b[g][k], ax);
            if (i < m) {
                qq[i] = ax;
                acc = fma(pp[i], ax, acc);
            }
        }
    }
    // All slices have the same offsets: a row without an entry at one multiplies
    // its stored zero by what lies there (shared memory always holds a value).
    // GF slices of values from global memory are in flight per warp.
    template <int WM, int G, int GF>
    __device__ __forceinline__ T product_same(T* p) const {
        int off[WM];
        const int Wn = W, m = rows, nv = nval, ns = nsl, nw = blockDim.x >> 5;
#pragma unroll
        for (int k = 0; k < WM; ++k) off[k] = k < Wn ? list.off[k] : 0;
        T* const qq = q;
        const T* const pp = p + pad;
        const T* const sv = p + val_at;
        const T* const gv = gval;
        int s = threadIdx.x >> 5;
        T acc = 0;
        for (; s + (G - 1) * nw < nv; s += G * nw) some<WM, G>(sv, pp, qq, s, nw, Wn, m, off, acc);
        for (; s < nv; s += nw) some<WM, 1>(sv, pp, qq, s, nw, Wn, m, off, acc);
        for (; s + (GF - 1) * nw < ns; s += GF * nw) some<WM, GF>(gv, pp, qq, s, nw, Wn, m, off, acc);
        for (; s < ns; s += nw) some<WM, 1>(gv, pp, qq, s, nw, Wn, m, off, acc);
        return acc;
    }
    __device__ T product_slots(T* p) const {
        const int lane = threadIdx.x & 31, nw = blockDim.x >> 5, Wn = W;
        const int2* ss = slots(p);
        T acc = 0;
        for (int s = threadIdx.x >> 5; s < nsl; s += nw) {
            const int i = s * 32 + lane;
            const T* v = (s < nval ? p + val_at : gval) + (size_t)s * Wn * 32 + lane;
            T ax = 0;
            for (int k = 0; k < Wn; ++k) {
                const int2 m = ss[s * Wn + k];
                if ((m.y >> lane) & 1) ax = fma(v[k * 32], p[pad + i + m.x], ax);
            }
            if (i < rows) {
                q[i] = ax;
                acc = fma(p[pad + i], ax, acc);
            }
        }
        return acc;
    }
    // q = A p on the own rows; returns this thread's part of p.q.
    template <int GF>
    __device__ __forceinline__ T product(T* p) const {
        constexpr int G = GF >= 4 ? 2 : 1;
        if (list.count > 0 && W <= 5) return product_same<5, G, GF>(p);
        if (list.count > 0 && W <= 9) return product_same<9, 1, 1>(p);
        return product_slots(p);
    }
};

}  // namespace sa
