// TSMTTSM for any M, N <= 64 with the tile, its orientation and the CTA size
// chosen per launch, and a reduction made for short products.
//
// What bounds it: the FP64 pipe (2 FMA per cycle and SM).  A guarded tile
// entry and an idle lane of an active warp take their slot there like useful
// ones, so the shapes without a kernel of their own lose what their tile
// pads; loads are cheap beside it (a 1 x 5 tile loads 6 values for 5 FMAs of
// 16 cycles a warp).  So every thread owns a narrow strip, one column of one
// operand against T consecutive-stride columns of the other, and the rule
// below picks T (a template parameter), which operand it runs along, and the
// number of row lanes, hence the CTA size, that leave the fewest FP64 slots
// unused.  37 x 53 runs as 37 x 6 strips of 9: 2 % padding, where 2 x 5 tiles in
// CTAs of 256 threads leave 14 % unused.
//
// Short products are bound by their tails instead.  The row lanes of a CTA
// are summed all strip entries at a time (the other kernels go entry by
// entry, two barriers per level each), and the CTAs' partials always by the
// final kernel, whose few CTAs are already waiting when this one ends (the
// last CTA alone, or groups of CTAs in two levels, took 2 to 5 us more).
// Every order is fixed by the shape and the grid, so results repeat bit for
// bit.  A lane's rows are one chain of FMAs: real 37 x 53, 300007 rows has an
// error of 1.1e-15 against 64 bits, 8.7e-16 with the tile kernel's shorter ones.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "fp64_common.cuh"
#include "tsm_internal.h"

namespace tsm {
namespace {

constexpr int kMaxBlock = 512;
constexpr int kChunk = 8;      // doubles of a thread's strip reduced at a time

struct RowShape {
    int T;        // strip length
    int along_m;  // the strip runs along M (else along N)
    int P, L;     // threads per row lane, row lanes
    int block;    // CTA size, a multiple of 32
    double slots; // FP64 slots per useful FMA
};

// Strip lengths with an instantiation.
constexpr int kLen[] = {1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 13};
constexpr int kLenMaxCplx = 7;  // complex strips hold two accumulators per entry

// Fewest FP64 slots per useful FMA: padding of the strip's last entries
// times the idle lanes of the CTA's last warp, plus a charge for loads (two
// slots' worth per load over the strip's FMAs: 1 + T loads for T (4 T) FMAs
// of 16 cycles each), CTAs near 256 threads, and registers.
RowShape find_row_shape(int M, int N, int cplx) {
    RowShape best = {0, 0, 1, 1, 32, 0.0};  // T = 0: more threads per row than a CTA holds
    double bc = 1e30;
    for (int am = 0; am < 2; ++am) {
        const int V = am ? N : M, W = am ? M : N;
        for (int T : kLen) {
            if (T > W || (cplx && T > kLenMaxCplx)) continue;
            const int parts = (W + T - 1) / T, P = V * parts;
            if (P > kMaxBlock) continue;
            for (int L = 1; P * L <= kMaxBlock; ++L) {
                const int block = (P * L + 31) / 32 * 32;
                const double fill = (double)P * L / block;
                const double pad = (double)parts * T / W;
                const double load = 1.0 + (1.0 + T) / T * (cplx ? 0.02 : 0.06);
                double c = pad / fill * load;
                if (block < 192 || block > 320) c *= 1.02;
                if (!cplx && T >= 8) c *= 1.03;  // 90 and more registers: half the warps of T <= 7
                if (c < bc - 1e-9 || (c < bc + 1e-9 && block > best.block && block <= 256)) {
                    bc = c;
                    best = RowShape{T, am, P, L, block, pad / fill};
                }
            }
        }
    }
    return best;
}

// The same, kept per shape (the search takes a few microseconds).
const RowShape& row_shape(int M, int N, int cplx) {
    static std::once_flag once[2][64][64];
    static RowShape shape[2][64][64];
    std::call_once(once[cplx][M - 1][N - 1],
                   [&] { shape[cplx][M - 1][N - 1] = find_row_shape(M, N, cplx); });
    return shape[cplx][M - 1][N - 1];
}

template <int T, int U, bool CPLX, bool CONJ>
__global__ void __launch_bounds__(kMaxBlock) k_row(const TsmttsmArgs a, const int along_m, const int P,
                                                   const int L) {
    constexpr int CC = CPLX ? 2 : 1, E = T * CC;
    __shared__ double red[kMaxBlock / 2 * kChunk];
    tsmttsm_begin(a);
    const int V = along_m ? a.N : a.M, W = along_m ? a.M : a.N;
    const int parts = (W + T - 1) / T;
    const int t = threadIdx.x, lane = t / P, p = t - lane * P;
    const int v = p % V, w = p / V;  // entries (v, w + j * parts)
    const bool active = lane < L;
    // operand columns of this thread; entries past W repeat column w, and
    // are not stored
    const int64_t sv = (along_m ? a.ldb : a.lda) * CC, sw = (along_m ? a.lda : a.ldb) * CC;
    const double* __restrict__ pv = (along_m ? a.B : a.A) + v * CC;
    const double* __restrict__ pw = (along_m ? a.A : a.B) + w * CC;
    int off[T];
#pragma unroll
    for (int j = 0; j < T; ++j) off[j] = w + j * parts < W ? j * parts * CC : 0;

    double acc[T][CC];
#pragma unroll
    for (int j = 0; j < T; ++j)
#pragma unroll
        for (int c = 0; c < CC; ++c) acc[j][c] = 0.0;
    const int64_t G = gridDim.x;
    const int64_t k0 = a.K * (int64_t)blockIdx.x / G, k1 = a.K * ((int64_t)blockIdx.x + 1) / G;
    auto step = [&](const double(&x)[CC], const double(&y)[T][CC]) {
#pragma unroll
        for (int j = 0; j < T; ++j) {
            if (!CPLX) {
                acc[j][0] = fma(x[0], y[j][0], acc[j][0]);
            } else {
                // x y, or conj(x) y; with the strip along M, y is A's and the
                // sign of the imaginary part is set after the loop
                const double xr = x[0], xi = x[CC - 1], yr = y[j][0], yi = y[j][CC - 1];
                acc[j][0] = fma(xr, yr, acc[j][0]);
                acc[j][0] = fma(CONJ ? xi : -xi, yi, acc[j][0]);
                acc[j][CC - 1] = fma(xr, yi, acc[j][CC - 1]);
                acc[j][CC - 1] = fma(CONJ ? -xi : xi, yr, acc[j][CC - 1]);
            }
        }
    };
    if (active) {
        // Two register sets of U rows in turn: the next U rows' loads are in
        // flight while this set is multiplied.  (Without, the warps of a CTA
        // wait for their rows together: 37 x 53 at 14 warps per SM ran at half
        // speed.)  Rows past the end repeat the first and are not used.
        double x[2][U][CC], y[2][U][T][CC];
        auto load = [&](int s, int64_t k) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t ku = k + (int64_t)u * L < k1 ? k + (int64_t)u * L : k0;
                const double* rv = pv + ku * sv;
                const double* rw = pw + ku * sw;
#pragma unroll
                for (int c = 0; c < CC; ++c) x[s][u][c] = __ldg(rv + c);
#pragma unroll
                for (int j = 0; j < T; ++j)
#pragma unroll
                    for (int c = 0; c < CC; ++c) y[s][u][j][c] = __ldg(rw + off[j] + c);
            }
        };
        auto use = [&](int s, int64_t k) {
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (k + (int64_t)u * L < k1) step(x[s][u], y[s][u]);
        };
        const int64_t next = (int64_t)U * L;
        int64_t k = k0 + lane;
        if (k < k1) load(0, k);
        for (; k < k1; k += 2 * next) {
            load(1, k + next);
            use(0, k);
            load(0, k + 2 * next);
            use(1, k + next);
        }
    }

    if (CONJ && along_m)
#pragma unroll
        for (int j = 0; j < T; ++j) acc[j][CC - 1] = -acc[j][CC - 1];

    pdl_trigger();  // the main loop is done
    pdl_wait();     // the previous launch on the stream may still use the workspace
    // Row lanes: chunks of kChunk strip entries, a fixed-pairing tree (lane l
    // absorbs lane l + h), the upper lanes' values passed through shared
    // memory.  Every thread of the CTA takes part in the barriers.
    const int MN = a.M * a.N, MNc = MN * CC;
    double* part = a.ws + (int64_t)blockIdx.x * MNc;
    double* ac = &acc[0][0];
    for (int n = L; n > 1;) {
        const int h = (n + 1) >> 1;
        const int q = (lane - h) * P + p;  // slot of an upper lane; (n - h) P <= kMaxBlock / 2 of them
#pragma unroll
        for (int e0 = 0; e0 < E; e0 += kChunk) {
            if (lane >= h && lane < n)
#pragma unroll
                for (int e = 0; e < kChunk; ++e)
                    if (e0 + e < E) red[e * (kMaxBlock / 2) + q] = ac[e0 + e];
            __syncthreads();
            if (lane + h < n)
#pragma unroll
                for (int e = 0; e < kChunk; ++e)
                    if (e0 + e < E) ac[e0 + e] += red[e * (kMaxBlock / 2) + lane * P + p];
            __syncthreads();
        }
        n = h;
    }
    if (lane == 0)
#pragma unroll
        for (int j = 0; j < T; ++j) {
            const int y = w + j * parts;
            if (y >= W) continue;
            const int o = along_m ? y * a.N + v : v * a.N + y;
#pragma unroll
            for (int c = 0; c < CC; ++c) part[o * CC + c] = acc[j][c];
        }
    // the partials are summed by the final kernel, launched behind this one
}

typedef void (*Kernel)(const TsmttsmArgs, int, int, int);

template <int T, int U, bool CPLX>
Kernel kernel_of(bool conj) {
    return CPLX && conj ? (Kernel)k_row<T, U, CPLX, true> : (Kernel)k_row<T, U, CPLX, false>;
}

// Rows per register set: a few for the shortest strips, else one.
template <bool CPLX>
constexpr int rows_per_set(int T) {
    return T == 1 ? (CPLX ? 2 : 4) : (T <= 3 && !CPLX ? 2 : 1);
}
template <bool CPLX>
Kernel kernel_for(int T, bool conj) {
    switch (T) {
        case 1: return kernel_of<1, rows_per_set<CPLX>(1), CPLX>(conj);
        case 2: return kernel_of<2, rows_per_set<CPLX>(2), CPLX>(conj);
        case 3: return kernel_of<3, rows_per_set<CPLX>(3), CPLX>(conj);
        case 4: return kernel_of<4, 1, CPLX>(conj);
        case 5: return kernel_of<5, 1, CPLX>(conj);
        case 6: return kernel_of<6, 1, CPLX>(conj);
        case 7: return kernel_of<7, 1, CPLX>(conj);
        default: break;
    }
    if (CPLX) return nullptr;
    switch (T) {
        case 8: return kernel_of<8, 1, false>(false);
        case 9: return kernel_of<9, 1, false>(false);
        case 10: return kernel_of<10, 1, false>(false);
        default: return kernel_of<13, 1, false>(false);
    }
}

// Registers a thread, in the units they are handed out in (0: unknown).
template <bool CPLX>
int registers(int T) {
    static std::atomic<int> known[16];
    int r = known[T].load(std::memory_order_relaxed);
    if (!r) {
        cudaFuncAttributes at;
        if (cudaFuncGetAttributes(&at, (const void*)kernel_for<CPLX>(T, false)) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        known[T].store(r = (at.numRegs + 7) / 8 * 8, std::memory_order_relaxed);
    }
    return r;
}

double row_work(int M, int N, int64_t K, int cplx) { return (double)K * M * N * (cplx ? 4 : 1); }

// Dynamic shared memory (unused) that leaves room for no more than `cps` CTAs
// on an SM.  A grid of cps x SMs CTAs then is at full residency and may start
// early (pdl_allowed), and is spread evenly when it does.
size_t limit_smem(int cps) { return (size_t)228 * 1024 / (cps + 1) + 1024 - sizeof(double) * kMaxBlock / 2 * kChunk; }

template <bool CPLX>
cudaError_t launch_row(const TsmttsmArgs& a, int grid, cudaStream_t s) {
    const RowShape& r = row_shape(a.M, a.N, CPLX);
    const Kernel k = kernel_for<CPLX>(r.T, a.conj != 0);
    const int sms = device_info().sm_count, cps = (grid + sms - 1) / sms;
    size_t smem = 0;
    if (cps < resident_ctas((const void*)k, r.block, 0)) {
        smem = limit_smem(cps);
        if (smem > 48 * 1024) {
            // (the largest value ever used: a limit of each launch's own could be
            // lowered by another thread before the launch)
            const cudaError_t e =
                cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit_smem(1));
            if (e != cudaSuccess) return e;
        }
    }
    // the shortest start early at any grid: one CTA per SM is soon placed
    if (row_work(a.M, a.N, a.K, CPLX) < 1e7)
        return launch_early(pdl_enabled(), k, grid, r.block, smem, s, a, r.along_m, r.P, r.L);
    return launch_pdl(k, grid, r.block, smem, s, a, r.along_m, r.P, r.L);
}

template <bool CPLX>
int occ_row(int M, int N) {
    const RowShape& r = row_shape(M, N, CPLX);
    return resident_ctas((const void*)kernel_for<CPLX>(r.T, false), r.block, 0);
}

// CTAs per SM by the work: one below 6 10^6 FMAs (3 10^6 if a CTA has no more
// than six warps to hide its loads with), or where two would leave a CTA of
// more fewer than 64 rows for its partial; two below 10^8; else what fits.
// Three cases in the middle differ:
//   two CTAs that fill the register file leave no room for the CTAs of the
//     neighbours that wait on the SM, and some start a wave late (complex strips
//     of 6 and 7 in CTAs of 256): one.  Complex 2 x 12, 78231 rows 27.9 / 20.0 us
//     (two / one), 56 x 1, 40972 rows 29.0 / 23.3;
//   real CTAs of more than ten warps with strips of five and more hold an SM's
//     FMAs alone, up to 5 10^7 and 60000 rows: real 35 x 35, 19610 rows 56.8 / 44.2,
//     48 x 11, 36707 rows 45.6 / 35.1, 24 x 29, 25177 rows 32.7 / 32.8, but 5 x 59,
//     68213 rows 35.7 / 39.2;
//   operands that do not fit L2 (129 MB) wait for DRAM, which real CTAs with
//     fewer than 1200 FMAs per set of rows do not cover: three.  Real 64 x 2, 334665
//     rows 103 / 83 (two / three), 8 x 8, 902858 rows 137 / 111, 17 x 10, 446205
//     rows 234 / 170; with more FMAs real 32 x 5, 398825 rows 114 / 120.
// Measured (us, one / two / what fits): real 6 x 6 at 50000 rows 9.1 / 10.6 /
// 16.7, complex 50 x 50 at 5000 rows 99.6 / 108 / 99.6, real 22 x 22 at 52291
// rows 80.6 / 52.7 / 60.6, complex 17 x 33 at 200000 rows 1211 / 849 / 788;
// one / two: real 43 x 17 (192 threads) at 9575 rows 26.6 / 19.9, real 16 x 16
// at 27343 rows 21.8 / 19.5, real 8 x 8 at 109375 rows 21.7 / 19.0, complex
// 16 x 16 at 3906 rows 11.4 / 13.6, complex 32 x 32 at 4882 rows 42.1 / 43.8.
template <bool CPLX>
int grid_row(int M, int N, int64_t K) {
    const int sms = device_info().sm_count;
    const int occ = std::max(occ_row<CPLX>(M, N), 1);
    const double fma = row_work(M, N, K, CPLX);
    int cps = occ;
    const bool few_warps = row_shape(M, N, CPLX).block <= 192;
    if (fma < (few_warps ? 3e6 : 6e6) || (!few_warps && K < 128 * (int64_t)sms)) {
        cps = 1;
    } else if (fma < 1e8) {
        const RowShape& r = row_shape(M, N, CPLX);
        const int set = r.block * r.T * rows_per_set<CPLX>(r.T);
        const double bytes = 8.0 * (CPLX ? 2 : 1) * (M + N) * (double)K;
        // (a waiting CTA of the final kernel: 64 threads of 48 registers at most)
        const bool room = 2 * r.block * registers<CPLX>(r.T) + 64 * 48 <= 65536;
        if (!room || (!CPLX && r.T >= 5 && r.block > 320 && fma < 5e7 && K < 60000))
            cps = 1;
        else
            cps = !CPLX && set < 1200 && bytes > 9.5e7 ? 3 : 2;
    }
    return sms * std::min(cps, occ);
}

template <bool CPLX>
Variant make_row() {
    Variant v;
    memset(&v, 0, sizeof(v));
    snprintf(v.info.name, sizeof(v.info.name), "tsmttsm_%s_row", CPLX ? "c64" : "r64");
    v.info.kind = TSM_KIND_TSMTTSM;
    v.info.dtype = CPLX ? TSM_C64 : TSM_R64;
    v.info.tile_m = 1;
    v.info.tile_n = CPLX ? kLenMaxCplx : 13;
    v.info.unroll = 2;
    v.info.block = kMaxBlock;
    v.info.runtime_tile = 1;
    v.tsmttsm = launch_row<CPLX>;
    v.occupancy = occ_row<CPLX>;
    v.grid = grid_row<CPLX>;
    v.final_pass = true;
    v.resolve = [](int M, int N, tsm_variant_info* info) {
        const RowShape& r = row_shape(M, N, CPLX);
        info->tile_m = r.along_m ? r.T : 1;
        info->tile_n = r.along_m ? 1 : r.T;
        info->block = r.block;
    };
    v.supports = [](int M, int N) { return row_shape(M, N, CPLX).T > 0; };
    return v;
}

}  // namespace

double row_slots(int M, int N, int cplx) { return row_shape(M, N, cplx).slots; }
double row_long_cost(int M, int N, int cplx) {
    const RowShape& r = row_shape(M, N, cplx);
    if (!cplx) return r.T == 1 ? 1.3 : r.block <= 192 ? 1.2 : 1.09;
    if (r.T > 3) return 1.05;
    // short strips leave the pipe idle where the SM's four schedulers do not
    // have equally many warps
    const int warps = r.block / 32 * std::max(occ_row<true>(M, N), 1);
    return std::max(1.05, (warps + 3) / 4 * 4.0 / warps);
}

void register_row_variants(std::vector<Variant>& tsmttsm) {
    tsmttsm.push_back(make_row<false>());
    tsmttsm.push_back(make_row<true>());
}

}  // namespace tsm
