// TSMM for any M, N <= 64 with the results per thread, the row lanes and the
// grid chosen per launch, for products that the width-specialised kernels do
// not cover or are too coarse for.
//
// What bounds it: the FP64 pipe, and at few rows how evenly the rows spread.
// The other kernels walk K with a grid stride, several rows per thread and
// pass: complex 64 x 64 takes 62 us a pass of 608 CTAs whether that pass holds
// 9000 rows or 1000, and 200003 rows of complex 23 x 11 are 7.15 passes that
// take the time of 8 (rows past the end are multiplied as zeros).  Here a CTA
// owns a contiguous range of rows, a pass with fewer rows costs only their
// warps, and short products get as many CTAs of as few rows as fill every
// SM once.
//
// Thread (r, q) computes results q, q + tpr, ... (T of them) of rows r, r + L,
// ... of its CTA's range, two rows at a time while there are two, with
// alpha * C staged in shared memory (Sec. 4.2) and the next columns of A
// loaded while the present ones are multiplied.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "fp64_common.cuh"
#include "tsm_internal.h"

namespace tsm {
namespace {

constexpr int kMaxBlock = 512;

template <int T, bool CPLX, bool GEN>
__global__ void __launch_bounds__(kMaxBlock) k_mm(const TsmmArgs a, const int tpr, const int L, const int64_t rows) {
    constexpr int CC = CPLX ? 2 : 1;
    constexpr int MC = CPLX ? 2 : 4;  // columns of A per register set
    extern __shared__ __align__(16) double cs[];  // alpha * C, M x N (x CC)
    const int M = a.M, N = a.N;
    tsmm_begin(a);
    tsmm_stage_c<CC>(a, cs);
    const int r = threadIdx.x / tpr, q = threadIdx.x - r * tpr;
    const unsigned lanes = __ballot_sync(0xffffffffu, r < L);
    if (r >= L) return;
    const int64_t k0 = rows * blockIdx.x, k1 = k0 + rows < a.K ? k0 + rows : a.K;
    const int64_t sa = a.lda * CC, sb = a.ldb * CC;

    auto process = [&](auto count, int64_t k, bool live) {
        constexpr int U = decltype(count)::value;
        const double* __restrict__ ar[U];
        double* br[U];
        double acc[U][T][CC];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            // the second row is past the range in some threads of a range's last warp: those repeat the first
            const int64_t ku = u && k + L < k1 ? k + L : k;
            ar[u] = a.A + ku * sa;
            br[u] = a.B + ku * sb;
        }
        double av[2][MC][U][CC];
        auto load = [&](int s, int m0) {
#pragma unroll
            for (int mm = 0; mm < MC; ++mm)
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int c = 0; c < CC; ++c) av[s][mm][u][c] = __ldg(ar[u] + min(m0 + mm, M - 1) * CC + c);
        };
        load(0, 0);
        // the old B values open the FMA chains (tsmm_acc_init)
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < T; ++j) {
                const int n = q + j * tpr;
                double o[2] = {0.0, 0.0};
                if (!a.beta_zero && live && (j < T - 1 || n < N))
#pragma unroll
                    for (int c = 0; c < CC; ++c) o[c] = br[u][n * CC + c];
                tsmm_acc_init<CC, GEN>(a, o[0], o[1], acc[u][j][0], acc[u][j][CC - 1]);
            }
        auto use = [&](int s, int m0) {
#pragma unroll
            for (int mm = 0; mm < MC; ++mm) {
                const int m = m0 + mm;
                if (m >= M) break;
                const double* row = cs + (m * N + q) * CC;
#pragma unroll
                for (int j = 0; j < T; ++j) {
                    // only the last of a thread's results can lie past N
                    if (j == T - 1 && q + j * tpr >= N) break;
                    if (!CPLX) {
                        const double cr = row[j * tpr];
#pragma unroll
                        for (int u = 0; u < U; ++u) acc[u][j][0] = fma(av[s][mm][u][0], cr, acc[u][j][0]);
                    } else {
                        const double2 c = *reinterpret_cast<const double2*>(row + j * tpr * CC);
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            const double xr = av[s][mm][u][0], xi = av[s][mm][u][CC - 1];
                            acc[u][j][0] = fma(xr, c.x, acc[u][j][0]);
                            acc[u][j][0] = fma(-xi, c.y, acc[u][j][0]);
                            acc[u][j][CC - 1] = fma(xr, c.y, acc[u][j][CC - 1]);
                            acc[u][j][CC - 1] = fma(xi, c.x, acc[u][j][CC - 1]);
                        }
                    }
                }
            }
        };
        for (int m0 = 0; m0 < M; m0 += 2 * MC) {
            load(1, m0 + MC);
            use(0, m0);
            load(0, m0 + 2 * MC);
            use(1, m0 + MC);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < T; ++j) {
                const int n = q + j * tpr;
                if ((u ? k + L < k1 : live) && (j < T - 1 || n < N)) tsmm_store_plain<CC>(br[u], n, acc[u][j][0], acc[u][j][CC - 1]);
            }
    };
    // One choice per warp, as a warp that takes both paths pays for both;
    // threads past the range repeat its last row and store nothing.
    for (int64_t k = k0 + r; __any_sync(lanes, k < k1); k += 2 * (int64_t)L) {
        if (__any_sync(lanes, k + L < k1)) process(std::integral_constant<int, 2>(), min(k, k1 - 1), k < k1);
        else process(std::integral_constant<int, 1>(), min(k, k1 - 1), k < k1);
    }
}

typedef void (*Kernel)(const TsmmArgs, int, int, int64_t);

template <bool CPLX, bool GEN>
Kernel kernel_for(int T) {
    switch (T) {
        case 1: return k_mm<1, CPLX, GEN>;
        case 2: return k_mm<2, CPLX, GEN>;
        case 3: return k_mm<3, CPLX, GEN>;
        case 4: return k_mm<4, CPLX, GEN>;
        default: break;
    }
    if (CPLX) return nullptr;
    return k_mm<5, false, GEN>;
}
constexpr int kResMax = 5, kResMaxCplx = 4;  // results per thread with an instantiation (128 registers at 8)
// Time over slots of a long product at 1, 2, ... results per thread.
constexpr double kCharge[] = {1.075, 1.04, 1.035, 1.03, 1.035};
constexpr double kChargeCplx[] = {1.03, 1.03, 1.025, 1.02};

struct MmShape {
    int T, tpr, L, block, grid;
    int64_t rows;  // per CTA
    double cost;  // time of a long product over its useful FMAs'
};

size_t mm_smem(int M, int N, int cplx) { return (size_t)M * N * (cplx ? 2 : 1) * sizeof(double); }

// The limit is set to the same value every time: one set to a launch's own
// need could be lowered by another thread before that launch.
cudaError_t allow_smem(const void* kernel, size_t smem) {
    return smem > 48 * 1024 ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)
                            : cudaSuccess;
}

template <bool CPLX>
int mm_resident(int T, int block, int M, int N) {
    const size_t smem = mm_smem(M, N, CPLX);
    const Kernel k = kernel_for<CPLX, false>(T);
    if (allow_smem((const void*)k, smem) != cudaSuccess) return 0;
    return resident_ctas((const void*)k, block, smem);
}

// Row lanes of a full CTA for each count of threads per row: as many as fit
// with the fewest idle lanes in the last warp.
struct Lanes {
    int L[65];
    Lanes() {
        for (int tpr = 1; tpr <= 64; ++tpr) {
            int best = 1;
            double bf = 0.0;
            for (int l = 1; l * tpr <= kMaxBlock; ++l) {
                const double fill = (double)(l * tpr) / ((l * tpr + 31) / 32 * 32);
                if (fill > bf - 1e-9 || (fill > 0.995 * bf && l > best * 5 / 4)) {
                    bf = fill;
                    best = l;
                }
            }
            L[tpr] = best;
        }
    }
};

// Results per thread: the fewest unused FP64 slots (idle and masked lanes
// cost as much as live ones), among those that leave an SM at least 256
// threads with a row each; one result per thread if none does.  The charge
// for what a thread loads per FMA is measured (real 39 x 23, 157000 rows;
// complex 10 x 17, 500000 rows), as is the one for short ranges, whose first
// loads and last stores nothing overlaps: complex 33 x 20, 30000 rows take
// 147 us as one pass of 102 row lanes, 137 as four of 25.  CTAs of up to 512
// threads beat those of 256 by 1 to 4 % (fewer last warps of a range).
template <bool CPLX>
MmShape mm_shape(int M, int N, int64_t K) {
    static const Lanes full;
    const int64_t sms = device_info().sm_count, rows_sm = std::max<int64_t>((K + sms - 1) / sms, 1);
    MmShape best = {0, 0, 0, 0, 0, 0, 0.0};
    double bc = 1e30;
    for (int T = 1; T <= (CPLX ? kResMaxCplx : kResMax) && T <= N; ++T) {
        const int tpr = (N + T - 1) / T;
        if ((T - 1) * tpr >= N) continue;  // a thread's last result alone may lie past N
        if (T > 1 && rows_sm * tpr < 256) continue;
        const int L = rows_sm * tpr <= kMaxBlock ? (int)rows_sm : full.L[tpr];
        const int block = (L * tpr + 31) / 32 * 32;
        const double slots = (double)T * tpr / N * block / (L * tpr);
        const double passes = std::max(1.0, (double)rows_sm / (2 * L));
        const double c = slots * ((CPLX ? kChargeCplx : kCharge)[T - 1] + 0.06 / passes);
        if (c < bc) {
            bc = c;
            best = MmShape{T, tpr, L, block, 0, 0, c};
        }
    }
    const int64_t passes = (rows_sm + best.L - 1) / best.L;
    const int64_t cps = std::min<int64_t>(std::max(mm_resident<CPLX>(best.T, best.block, M, N), 1), passes);
    best.rows = std::max<int64_t>((K + sms * cps - 1) / (sms * cps), 1);
    best.grid = (int)std::max<int64_t>((K + best.rows - 1) / best.rows, 1);
    return best;
}

template <bool CPLX, bool GEN>
cudaError_t launch_as(const TsmmArgs& a, const MmShape& s, int grid, int64_t rows, cudaStream_t st) {
    size_t smem = mm_smem(a.M, a.N, CPLX);
    const Kernel k = kernel_for<CPLX, GEN>(s.T);
    cudaError_t e = allow_smem((const void*)k, smem);
    if (e != cudaSuccess) return e;
    // Shared memory that leaves room for this grid's CTAs per SM and no more:
    // with CTAs of the neighbouring kernels waiting on some SMs, the placement
    // would else put two on one SM and none on another.  Complex 33 x 20, 1000
    // rows inside a Gram-Schmidt step: 47.3 us as placed, 22.9 spread.
    const int sms = device_info().sm_count, cps = (grid + sms - 1) / sms;
    if (cps < resident_ctas((const void*)k, s.block, smem))
        smem = std::max<size_t>(smem, (size_t)228 * 1024 / (cps + 1) + 1024);
    if ((e = allow_smem((const void*)k, smem)) != cudaSuccess) return e;
    // the shortest start early at any grid: their CTAs are soon placed
    if ((double)a.M * a.N * (CPLX ? 4 : 1) * (double)a.K < 1e7)
        return launch_early(pdl_enabled(), k, grid, s.block, smem, st, a, s.tpr, s.L, rows);
    return launch_pdl(k, grid, s.block, smem, st, a, s.tpr, s.L, rows);
}

// A grid other than the shape's own cuts K into that many ranges.
template <bool CPLX>
cudaError_t launch_mm(const TsmmArgs& a, int grid, cudaStream_t st) {
    const MmShape s = mm_shape<CPLX>(a.M, a.N, a.K);
    const int64_t rows = grid == s.grid ? s.rows : std::max<int64_t>((a.K + grid - 1) / grid, 1);
    return tsmm_general_beta(a) ? launch_as<CPLX, true>(a, s, grid, rows, st)
                                : launch_as<CPLX, false>(a, s, grid, rows, st);
}

template <bool CPLX>
Variant make_mm() {
    Variant v;
    memset(&v, 0, sizeof(v));
    snprintf(v.info.name, sizeof(v.info.name), "tsmm_%s_row", CPLX ? "c64" : "r64");
    v.info.kind = TSM_KIND_TSMM;
    v.info.dtype = CPLX ? TSM_C64 : TSM_R64;
    v.info.tile_n = CPLX ? kResMaxCplx : kResMax;
    v.info.threads_per_row = 64;  // the largest; the launch picks the value
    v.info.unroll = 2;
    v.info.block = kMaxBlock;
    v.info.runtime_tile = 1;
    v.tsmm = launch_mm<CPLX>;
    v.occupancy = [](int M, int N) {
        const MmShape s = mm_shape<CPLX>(M, N, (int64_t)1 << 24);
        return mm_resident<CPLX>(s.T, s.block, M, N);
    };
    v.grid = [](int M, int N, int64_t K) { return mm_shape<CPLX>(M, N, K).grid; };
    v.resolve = [](int M, int N, tsm_variant_info* info) {
        const MmShape s = mm_shape<CPLX>(M, N, (int64_t)1 << 24);
        info->tile_n = s.T;
        info->threads_per_row = s.tpr;
        info->block = s.block;
    };
    return v;
}

}  // namespace

double mm_cost(int M, int N, int64_t K, int cplx) {
    return cplx ? mm_shape<true>(M, N, K).cost : mm_shape<false>(M, N, K).cost;
}

void register_mm_variants(std::vector<Variant>& tsmm) {
    tsmm.push_back(make_mm<false>());
    tsmm.push_back(make_mm<true>());
}

}  // namespace tsm
