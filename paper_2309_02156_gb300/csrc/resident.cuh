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

namespace sa {

constexpr int kTeamMax = 160;              // blocks of a grid team
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
                unsigned seen = 0;
                for (int left = kTeamPolls; left > 0; --left) {
                    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
                    if (seen >= want) break;
                }
                if (seen < want) *bad = 1;
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

// Where a block's data lies: the gathered vector always in shared memory, the
// others there as far as they fit (else in the context's global vectors).
struct ResLayout {
    int per;           // slices of a block
    int ext;           // entries of the gathered vector's shared array
    int r_in, q_in, x_in;
    int nval;          // slices whose matrix values are kept in shared memory
};

// Shared bytes of a layout for element size `el` and W slots per slice.
__host__ __device__ inline size_t res_bytes(const ResLayout& l, int W, size_t el) {
    const size_t rows = 32 * (size_t)l.per;
    size_t words = (size_t)l.ext + rows * (size_t)(l.r_in + l.q_in + l.x_in) +
                   (size_t)l.nval * 32 * W;
    return ((words * el + 7) & ~(size_t)7) + 8 * (size_t)l.per * W;
}

// Largest layout within `budget` bytes for `nblk` blocks; false if the gathered
// vector alone does not fit.
inline bool res_layout(int n, int W, int reach, int nblk, size_t el, size_t budget, ResLayout* l) {
    const int ns = (n + 31) / 32;
    l->per = (ns + nblk - 1) / nblk;
    const long long rows = 32LL * l->per, want = rows + 2LL * reach;
    l->ext = (int)(want < n + 32LL ? want : n + 32LL);
    l->r_in = l->q_in = l->x_in = l->nval = 0;
    if (res_bytes(*l, W, el) > budget) return false;
    int* which[3] = {&l->r_in, &l->q_in, &l->x_in};
    for (int* w : which) {
        *w = 1;
        if (res_bytes(*l, W, el) > budget) *w = 0;
    }
    const size_t used = res_bytes(*l, W, el), slice = el * 32 * W;
    const size_t fit = used + 8 < budget ? (budget - used - 8) / slice : 0;
    l->nval = (int)(fit < (size_t)l->per ? fit : (size_t)l->per);
    return true;
}

// Row sums of the slot-form product over this block's slices: `get(c)` reads
// entry c - row .. as an index into the gathered array (base + local row +
// offset); epi(local row, sum, live).
template <typename T, int WM, typename Epi>
__device__ __forceinline__ void res_product(const int2* sslot, const T* sval, const T* gval,
                                            const T* vec, int base, int nsl, int nval, int W,
                                            int rows, const Epi& epi) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int s = warp; s < nsl; s += nw) {
        const int i = s * 32 + lane;
        const T* vv = s < nval ? sval + (size_t)s * W * 32 + lane : gval + (size_t)s * W * 32 + lane;
        T ax = 0;
        if constexpr (WM > 0) {
            T v[WM], x[WM];
#pragma unroll
            for (int k = 0; k < WM; ++k) v[k] = k < W ? vv[k * 32] : (T)0;
#pragma unroll
            for (int k = 0; k < WM; ++k) {
                x[k] = 0;
                if (k < W) {
                    const int2 m = sslot[s * W + k];
                    if ((m.y >> lane) & 1) x[k] = vec[base + i + m.x];
                }
            }
#pragma unroll
            for (int k = 0; k < WM; ++k)
                if (k < W) ax = fma(v[k], x[k], ax);
        } else {
            for (int k = 0; k < W; ++k) {
                const int2 m = sslot[s * W + k];
                if ((m.y >> lane) & 1) ax = fma(vv[k * 32], vec[base + i + m.x], ax);
            }
        }
        epi(i, ax, i < rows);
    }
}

}  // namespace sa
