// Sparse-sign row sketch and the sketched block W = S [A X | b].
//
// S (s x n) has zeta nonzeros +-1/sqrt(zeta) per column.  Column j draws its
// candidate rows from SplitMix64 outputs 256 j + c + 1 (c = 0, 1, ...):
// row = ((h >> 32) * s) >> 32, sign = bit 0 of h, repeated rows skipped; if
// 256 candidates fall short, the smallest unused rows are taken with sign +1.
// The sketch replaces the n-row reduced least-squares problem of Algorithm 1
// (min ||A(t_i) X y - b(t_i)||) by its s-row image; the paper itself
// sketches columns instead (Section 2.2), so this construction is this
// library's own.
//
// Layout: the history ring X is row-major, n rows of ldx >= M values (slot k
// of row i at X[i * ldx + k]), so the M values a CSR neighbour contributes are
// one contiguous read.  W is row-major s x (M + 1): W[q * (M+1) + k] for
// history slot k < M and W[q * (M+1) + M] for b.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "sketch_tile.cuh"

namespace sa {

__global__ void sketch_columns_kernel(int n, int s, int zeta, uint64_t seed,
                                      uint16_t* packed, int32_t* rows_out, int8_t* signs_out) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    uint16_t e[kMaxZeta];
    sketch_column_packed(j, s, zeta, seed, e);
    for (int k = 0; k < zeta; ++k) {
        if (packed) packed[(size_t)j * zeta + k] = e[k];
        if (rows_out) rows_out[(size_t)j * zeta + k] = e[k] & 0x7fff;
        if (signs_out) signs_out[(size_t)j * zeta + k] = (e[k] & 0x8000) ? (int8_t)-1 : (int8_t)1;
    }
}

void launch_sketch_columns(int n, int s, int zeta, uint64_t seed, uint16_t* packed,
                           int32_t* rows, int8_t* signs, cudaStream_t st) {
    const int threads = 256;
    sketch_columns_kernel<<<(n + threads - 1) / threads, threads, 0, st>>>(
        n, s, zeta, seed, packed, rows, signs);
}

namespace {

int sketch_teams(int s, int ncol) {
    const size_t t = kSkSmemCap / sketch_team_bytes(s, ncol);
    return t < 1 ? 1 : (t > (size_t)kSkMaxTeams ? kSkMaxTeams : (int)t);
}

}  // namespace

// W = S [A X | b] in one pass over A and X, with S generated on the fly.
//
// A block (one per SM) runs up to eight teams of four warps; each team takes
// 32-row tiles in turn (tiles are dealt to the grid's teams cyclically, so
// that at any time the whole GPU works on one window of consecutive rows and
// the X rows a stencil shares between rows far apart, r and r +- the grid
// side, are still in L2 when their second reader comes).  For a tile:
//  (a) warp w takes rows 8w .. 8w+7: their CSR entries (staged in shared
//      memory) and sketch columns (zeta entries each, generated from the
//      counters), and b;
//  (b) it forms Y = A X on those rows, the 8 x M products spread over its
//      lanes, four at a time;
//  (c) the warps split the M + 1 columns: for each, the tile's largest
//      magnitude sets a fixed-point scale (values below 2^52, chosen from the
//      running maximum of the column; when a larger value arrives the
//      accumulated column is shifted to the new scale) and the column is
//      turned into integers;
//  (d) the team adds +-v into its 64-bit accumulator at the zeta sketch rows
//      of each row (shared-memory atomics: integer sums do not depend on
//      their order, so the result is deterministic), leaving the FP64 pipe
//      (the limiting unit of this GPU for FP64 work) to the products.
// At the end the block's teams are converted back to FP64 and summed in team
// order into partial[blk] (s (M+1) values); a column with a non-finite value
// becomes NaN.  A team takes at most kSkMaxTiles tiles (grid sizing), so an
// accumulator holds at most 1056 terms below 2^52 and stays below 2^63.
template <typename T, typename XT>
__global__ void __launch_bounds__(kSkMaxTeams * kSkTeamThreads, 1)
sketch_block_kernel(const int* __restrict__ rowptr, const int* __restrict__ colind,
                    const T* __restrict__ val, const XT* __restrict__ X, int ldx,
                    const double* __restrict__ b, int n, int nnz, int M, int s, int zeta,
                    uint64_t seed, double* __restrict__ partial, int* bad) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nteams = blockDim.x / kSkTeamThreads;
    const int team = threadIdx.x / kSkTeamThreads, tt = threadIdx.x % kSkTeamThreads;
    const int tw = tt >> 5;
    const int ncol = M + 1, wsz = s * ncol;
    const size_t tb = sketch_team_bytes(s, ncol);
    unsigned char* base_ptr = smem_raw + (size_t)team * tb;
    const SketchTeam<T> tm(base_ptr, s, ncol, tw);
    __shared__ int zk[kMaxZeta * (kMaxM + 1)];
    sketch_pairs(zk, zeta, ncol);
    tm.clear(wsz, ncol, tt);
    __syncthreads();
    int flag = 0;
    sketch_team_tiles<T, XT>(tm, team, zk, rowptr, colind, val, X, ldx, b, n, nnz, M, s, zeta, seed,
                             (long long)blockIdx.x * nteams + team, (long long)gridDim.x * nteams,
                             ((long long)n + 31) / 32, flag);
    if (flag) atomicOr(bad, 1);
    __syncthreads();
    double* out = partial + (size_t)blockIdx.x * wsz;
    for (int i = threadIdx.x; i < wsz; i += blockDim.x) {
        const int k = i % ncol;
        double acc = 0.0;
        bool nan = false;
        for (int t = 0; t < nteams; ++t) {
            const unsigned char* tp = smem_raw + (size_t)t * tb;
            const long long* Wt = reinterpret_cast<const long long*>(tp);
            const int* Ft = reinterpret_cast<const int*>(tp + 8 * (size_t)wsz + 8 * 32 * (size_t)ncol +
                                                         (size_t)kSkTeamWarps * kSkWarpStage * 12 +
                                                         2 * 32 * (size_t)kMaxZeta);
            const int st = Ft[ncol + k];
            nan |= (st & 2) != 0;
            if (st & 1) acc += scalbn((double)Wt[i], -Ft[k]);
        }
        out[i] = nan ? __longlong_as_double(0x7ff8000000000000ll) : acc;
    }
}

// W[i] = (1/sqrt(zeta)) * sum over blocks of partial[blk][i] (fixed order).
__global__ void sketch_reduce_kernel(const double* __restrict__ partial, int nblk, int wsz,
                                     double inv_sqrt_zeta, double* __restrict__ W) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= wsz) return;
    W[i] = sum_over_blocks(partial, nblk, wsz, i) * inv_sqrt_zeta;
}

// Blocks of the sketch kernel: one per SM, more when needed so that no team
// takes more than kSkMaxTiles tiles of 32 rows (its accumulators stay below
// 2^63), never more than the tiles need.
int sketch_grid(int n, int s, int M) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int teams = sketch_teams(s, M + 1);
    const long long ntiles = ((long long)n + 31) / 32;
    long long nblk = std::min<long long>(sms, (ntiles + teams - 1) / teams);
    const long long need = (ntiles + (long long)kSkMaxTiles * teams - 1) / ((long long)kSkMaxTiles * teams);
    if (need > nblk) nblk = need;
    return nblk > 0 ? (int)nblk : 1;
}

int sketch_grid_beside(int n, int s, int M) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int nblk = sketch_grid(n, s, M);
    const long long ntiles = ((long long)n + 31) / 32;
    const long long most = (long long)kSkMaxTiles * sketch_teams(s, M + 1) * (nblk - 1);
    return nblk == sms && nblk > 1 && ntiles <= most ? nblk - 1 : nblk;
}

size_t sketch_partial_doubles(int n, int s, int M) {
    return (size_t)sketch_grid(n, s, M) * s * (M + 1);
}

template <typename T, typename XT>
static void launch_sketch_impl(const int* rowptr, const int* colind, const T* val, const XT* X,
                               int ldx, const double* b, int n, int nnz, int M, int s, int zeta,
                               uint64_t seed, double* partial, int nblk, double* W, int* bad,
                               cudaStream_t st) {
    const int wsz = s * (M + 1);
    // Teams for these columns (at least as many as the grid was sized for,
    // so that no team takes more than kSkMaxTiles tiles).
    const int teams = sketch_teams(s, M + 1);
    const size_t smem = (size_t)teams * sketch_team_bytes(s, M + 1);
    // The attribute is per device: set it on every call (cheap, host only), to
    // one value for all sizes (other threads launch the kernel too).
    cudaFuncSetAttribute(sketch_block_kernel<T, XT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)kSkSmemCap);
    sketch_block_kernel<T, XT><<<nblk, teams * kSkTeamThreads, smem, st>>>(
        rowptr, colind, val, X, ldx, b, n, nnz, M, s, zeta, seed, partial, bad);
    const double inv = 1.0 / sqrt((double)zeta);
    sketch_reduce_kernel<<<(wsz + 127) / 128, 128, 0, st>>>(partial, nblk, wsz, inv, W);
}

void launch_sketch_f64(const int* rowptr, const int* colind, const double* val, const double* X,
                       int ldx, const double* b, int n, int nnz, int M, int s, int zeta,
                       uint64_t seed, double* partial, int nblk, double* W, int* bad,
                       cudaStream_t st) {
    launch_sketch_impl<double, double>(rowptr, colind, val, X, ldx, b, n, nnz, M, s, zeta, seed,
                                       partial, nblk, W, bad, st);
}

void launch_sketch_f32(const int* rowptr, const int* colind, const float* val, const float* X,
                       int ldx, const double* b, int n, int nnz, int M, int s, int zeta,
                       uint64_t seed, double* partial, int nblk, double* W, int* bad,
                       cudaStream_t st) {
    launch_sketch_impl<float, float>(rowptr, colind, val, X, ldx, b, n, nnz, M, s, zeta, seed,
                                     partial, nblk, W, bad, st);
}

}  // namespace sa
