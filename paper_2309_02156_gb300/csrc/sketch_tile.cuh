// The sketched block of 32-row tiles, by teams of four warps (the steps are
// described at sketch_block_kernel): used by the single-sequence sketch kernel
// and by the batched step.
#pragma once

#include "common.cuh"

namespace sa {

// Sketch entries of column j (row j of A), in acceptance order, packed as
// row | sign << 15 (sign bit set for -1).
__device__ __forceinline__ void sketch_column_packed(int j, int s, int zeta, uint64_t seed,
                                                     uint16_t* out) {
    uint64_t taken0 = 0, taken1 = 0;                  // rows already taken (s <= 128)
    int cnt = 0;
    const uint64_t gamma = 0x9E3779B97F4A7C15ull;
    for (int c = 0; c < 256 && cnt < zeta; ++c) {
        const uint64_t ctr = (uint64_t)j * 256ull + (uint64_t)(c + 1);
        const uint64_t h = mix64(seed + ctr * gamma);
        const int q = (int)(((h >> 32) * (uint64_t)s) >> 32);
        const uint64_t bit = 1ull << (q & 63);
        const bool dup = ((q < 64 ? taken0 : taken1) & bit) != 0;
        if (!dup) {
            if (q < 64) taken0 |= bit; else taken1 |= bit;
            out[cnt] = (uint16_t)(q | ((h & 1ull) ? 0x8000 : 0));
            ++cnt;
        }
    }
    for (int q = 0; cnt < zeta && q < s; ++q) {      // exhausted: smallest unused rows
        const uint64_t bit = 1ull << (q & 63);
        if (((q < 64 ? taken0 : taken1) & bit) == 0) {
            if (q < 64) taken0 |= bit; else taken1 |= bit;
            out[cnt] = (uint16_t)q;
            ++cnt;
        }
    }
}

constexpr int kSkTeamWarps = 4;      // warps of a team (one 32-row tile at a time)
constexpr int kSkTeamThreads = kSkTeamWarps * 32;
constexpr int kSkMaxTeams = 8;       // teams per block (one block per SM)
constexpr int kSkRowsPerWarp = 8;    // rows of a tile per warp
constexpr int kSkWarpStage = 64;     // CSR entries of a warp's rows staged in shared memory
constexpr int kSkFastRow = 5;        // rows up to this many entries take the unrolled path
constexpr int kSkU = 2;              // product entries per lane in flight (32 warps per SM: 64 registers)
constexpr int kSkValueBits = 52;     // |quantised value| < 2^52 (the bits of an FP64 mantissa)
constexpr int kSkMaxTiles = 33;      // tiles per team: <= 33 * 32 terms per accumulator, < 2^63
constexpr size_t kSkSmemCap = 220 * 1024;

// Bytes of one team's shared region: integer accumulator (s x ncol), the
// tile's Y (32 x ncol doubles, quantised in place), per warp the staged CSR
// values (8 bytes each) and columns, the tile's sketch entries, and per
// column the fixed-point exponent and status.
__host__ __device__ inline size_t sketch_team_bytes(int s, int ncol) {
    return 8 * (size_t)s * ncol + 8 * 32 * (size_t)ncol +
           (size_t)kSkTeamWarps * kSkWarpStage * 12 + 2 * 32 * (size_t)kMaxZeta +
           8 * (size_t)ncol;
}

// y (finite) as a fixed-point integer with F fraction bits, rounded to
// nearest (halves away from zero), by integer operations on its bits.  The
// caller guarantees |y| 2^F < 2^kSkValueBits.
__device__ __forceinline__ long long quantize(double y, int F) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(y);
    const int eb = (int)((bits >> 52) & 0x7ff);
    unsigned long long mant = bits & 0xfffffffffffffull;
    if (eb) mant |= 1ull << 52;
    const int sh = (eb ? eb - 1075 : -1074) + F;
    unsigned long long r;
    if (sh >= 0) {
        r = mant << sh;
    } else if (sh > -64) {
        const int d = -sh;
        r = (mant + (1ull << (d - 1))) >> d;
    } else {
        r = 0;
    }
    const long long v = (long long)r;
    return (bits >> 63) ? -v : v;
}

// w / 2^d rounded to nearest (halves up), for an accumulator |w| < 2^63.
__device__ __forceinline__ long long shift_round(long long w, int d) {
    if (d <= 0) return w;
    if (d >= 63) return 0;
    return (w + (1ll << (d - 1))) >> d;
}

__device__ __forceinline__ void team_sync(int team) {
    asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "r"(kSkTeamThreads) : "memory");
}

__device__ __forceinline__ unsigned long long warp_max_u64(unsigned long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
        v = w > v ? w : v;
    }
    return v;
}


// Arrays of one team within its shared region (sketch_team_bytes).
template <typename T>
struct SketchTeam {
    long long* Wi;
    double* Ys;
    T* valW;                             // of the calling warp
    int* colW;
    uint16_t* skS;
    int* Fk;
    int* stk;                            // bit 0: column has values, bit 1: non-finite
    __device__ SketchTeam(unsigned char* base, int s, int ncol, int tw) {
        Wi = reinterpret_cast<long long*>(base);
        Ys = reinterpret_cast<double*>(Wi + s * ncol);
        unsigned char* stg = reinterpret_cast<unsigned char*>(Ys + 32 * ncol);
        valW = reinterpret_cast<T*>(stg + (size_t)tw * kSkWarpStage * 8);
        colW = reinterpret_cast<int*>(stg + (size_t)kSkTeamWarps * kSkWarpStage * 8) + tw * kSkWarpStage;
        skS = reinterpret_cast<uint16_t*>(stg + (size_t)kSkTeamWarps * kSkWarpStage * 12);
        Fk = reinterpret_cast<int*>(skS + 32 * kMaxZeta);
        stk = Fk + ncol;
    }
    // Accumulator, scales and status cleared (by the team's threads).
    __device__ void clear(int wsz, int ncol, int tt) const {
        for (int i = tt; i < wsz; i += kSkTeamThreads) Wi[i] = 0;
        for (int k = tt; k < ncol; k += kSkTeamThreads) {
            Fk[k] = 0;
            stk[k] = 0;
        }
    }
};

// (sketch entry, column) of the flat index q = z (M + 1) + k of a row's scatter
// pairs, by all threads of the block; needs a barrier before use.
__device__ __forceinline__ void sketch_pairs(int* zk, int zeta, int ncol) {
    for (int q = threadIdx.x; q < zeta * ncol; q += blockDim.x) zk[q] = ((q / ncol) << 8) | (q % ncol);
}

// Tiles tile0, tile0 + tile_step, .. below tile_end into the team's accumulator.
template <typename T, typename XT>
__device__ __forceinline__ void sketch_team_tiles(
    const SketchTeam<T>& tm, int team, const int* zk, const int* __restrict__ rowptr,
    const int* __restrict__ colind, const T* __restrict__ val, const XT* __restrict__ X, int ldx,
    const double* __restrict__ b, int n, int nnz, int M, int s, int zeta, uint64_t seed,
    long long tile0, long long tile_step, long long tile_end, int& flag) {
    const int tt = threadIdx.x % kSkTeamThreads, tw = tt >> 5, lane = threadIdx.x & 31;
    const int ncol = M + 1, per_row = zeta * ncol;
    long long* const Wi = tm.Wi;
    double* const Ys = tm.Ys;
    T* const valW = tm.valW;
    int* const colW = tm.colW;
    uint16_t* const skS = tm.skS;
    int* const Fk = tm.Fk;
    int* const stk = tm.stk;
    const int nent = kSkRowsPerWarp * M;
    for (long long tile = tile0; tile < tile_end; tile += tile_step) {
        const int row0 = (int)(tile * 32);
        const int cnt = min(32, n - row0);
        const int r0 = row0 + tw * kSkRowsPerWarp;
        const int wcnt = max(0, min(kSkRowsPerWarp, n - r0));
        // (a) this warp's rows
        int rs = 0, re = 0;
        if (lane < wcnt) {
            rs = max(0, min(__ldg(rowptr + r0 + lane), nnz));
            re = max(rs, min(__ldg(rowptr + r0 + lane + 1), nnz));
            sketch_column_packed(r0 + lane, s, zeta, seed,
                                 skS + (tw * kSkRowsPerWarp + lane) * kMaxZeta);
        }
        const int e0 = __shfl_sync(0xffffffffu, rs, 0);
        const int e1 = max(e0, __shfl_sync(0xffffffffu, re, max(wcnt - 1, 0)));
        // Row pointers that decrease may name entries outside [e0, e1): not staged.
        const bool staged = e1 - e0 <= kSkWarpStage &&
                            __all_sync(0xffffffffu, lane >= wcnt || (rs >= e0 && re <= e1));
        if (staged) {
            for (int e = e0 + lane; e < e1; e += 32) {
                colW[e - e0] = __ldg(colind + e);
                valW[e - e0] = __ldg(val + e);
            }
        }
        if (lane < kSkRowsPerWarp)
            Ys[(tw * kSkRowsPerWarp + lane) * ncol + M] = lane < wcnt ? __ldg(b + r0 + lane) : 0.0;
        __syncwarp();
        // (b) Y[:, 0:M] = A X on the warp's rows, kSkU entries per lane at a time
        // (the loop is uniform over the warp: the shuffles need every lane)
        for (int eb0 = 0; eb0 < nent; eb0 += kSkU * 32) {
            const int eb = eb0 + lane;
            int rr[kSkU], kk[kSkU], st[kSkU], ln[kSkU];
            T acc[kSkU];
            int maxlen = 0;
#pragma unroll
            for (int u = 0; u < kSkU; ++u) {
                const int e = eb + 32 * u;
                const bool in = e < nent;
                const int r = in ? e / M : 0;
                rr[u] = r;
                kk[u] = in ? e - r * M : 0;
                const int a = __shfl_sync(0xffffffffu, rs, r);
                const int z = __shfl_sync(0xffffffffu, re, r);
                st[u] = a;
                ln[u] = (in && r < wcnt) ? z - a : 0;
                maxlen = max(maxlen, ln[u]);
                acc[u] = 0;
            }
            if (maxlen <= kSkFastRow) {
                T xv[kSkU][kSkFastRow], vv[kSkU][kSkFastRow];
#pragma unroll
                for (int t = 0; t < kSkFastRow; ++t) {
#pragma unroll
                    for (int u = 0; u < kSkU; ++u) {
                        xv[u][t] = 0;
                        vv[u][t] = 0;
                        if (t < ln[u]) {
                            const int e = st[u] + t;
                            const int c = staged ? colW[e - e0] : __ldg(colind + e);
                            if ((unsigned)c < (unsigned)n) {
                                vv[u][t] = staged ? valW[e - e0] : __ldg(val + e);
                                xv[u][t] = (T)__ldg(X + (size_t)c * ldx + kk[u]);
                            } else {
                                flag = 1;
                            }
                        }
                    }
                }
#pragma unroll
                for (int t = 0; t < kSkFastRow; ++t) {
#pragma unroll
                    for (int u = 0; u < kSkU; ++u)
                        if (t < ln[u]) acc[u] = fma(vv[u][t], xv[u][t], acc[u]);
                }
            } else {
                for (int t = 0; t < maxlen; ++t) {
#pragma unroll
                    for (int u = 0; u < kSkU; ++u) {
                        if (t < ln[u]) {
                            const int e = st[u] + t;
                            const int c = staged ? colW[e - e0] : __ldg(colind + e);
                            const T v = staged ? valW[e - e0] : __ldg(val + e);
                            if ((unsigned)c < (unsigned)n)
                                acc[u] = fma(v, (T)__ldg(X + (size_t)c * ldx + kk[u]), acc[u]);
                            else
                                flag = 1;
                        }
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kSkU; ++u)
                if (eb + 32 * u < nent)
                    Ys[(tw * kSkRowsPerWarp + rr[u]) * ncol + kk[u]] =
                        rr[u] < wcnt ? (double)acc[u] : 0.0;
        }
        team_sync(team);
        // (c) column scales and fixed-point values; warp tw owns columns tw, tw + 4, ...
        long long* Yq = reinterpret_cast<long long*>(Ys);
        for (int k = tw; k < ncol; k += kSkTeamWarps) {
            const double y = Ys[lane * ncol + k];
            const unsigned long long mx = warp_max_u64(
                lane < cnt ? ((unsigned long long)__double_as_longlong(y) & 0x7fffffffffffffffull)
                           : 0ull);
            const bool nonfinite = mx >= 0x7ff0000000000000ull;
            const bool use = mx != 0 && !nonfinite;
            const int has = stk[k] & 1;
            int F = Fk[k];
            if (use) {
                const int emax = (int)(mx >> 52) - 1023;          // mx < 2^(emax + 1)
                const int Fn = (kSkValueBits - 1) - emax;
                if (!has) {
                    F = Fn;
                } else if (Fn < F) {
                    const int d = F - Fn;
                    for (int q = lane; q < s; q += 32)
                        Wi[q * ncol + k] = shift_round(Wi[q * ncol + k], d);
                    F = Fn;
                }
            }
            Yq[lane * ncol + k] = (use && lane < cnt) ? quantize(y, F) : 0;
            __syncwarp();
            if (lane == 0) {
                Fk[k] = F;
                stk[k] |= (use ? 1 : 0) | (nonfinite ? 2 : 0);
            }
        }
        team_sync(team);
        // (d) W += S[:, r] Yq[r, :] for the tile's rows (integer atomics); the
        // (row, sketch entry, column) triples are walked with the (entry,
        // column) of each flat index taken from the block's table zk.
        {
            int r = 0, q = tt;
            while (q >= per_row) {
                q -= per_row;
                ++r;
            }
            for (; r < cnt;) {
                const int t = zk[q];
                const int z = t >> 8, k = t & 0xff;
                const long long v = Yq[r * ncol + k];
                if (v != 0) {
                    const unsigned e = skS[r * kMaxZeta + z];
                    atomicAdd(reinterpret_cast<unsigned long long*>(&Wi[(int)(e & 0x7fff) * ncol + k]),
                              (unsigned long long)((e & 0x8000) ? -v : v));
                }
                q += kSkTeamThreads;
                while (q >= per_row) {
                    q -= per_row;
                    ++r;
                }
            }
        }
        team_sync(team);
    }
}

}  // namespace sa
