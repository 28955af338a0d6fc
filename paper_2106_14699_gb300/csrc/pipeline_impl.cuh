// Template bodies of the per-(precision, size) entry points; included by the
// kernels_<prec>_<sizes>.cu units, which instantiate Sized<T, SZ> for a few
// sizes each.
#pragma once
#include "pipeline.cuh"
#include "rows_tm.cuh"
#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

namespace cmif {

// Sizes with the 16-lane variant of the column transforms (FP32 only).
template <typename T, int SZ>
constexpr bool kHasColVariant = std::is_same<T, float>::value && SZ >= 1024 && is_pow2(SZ);

// Shared memory of an SM (each block takes 1 KB more than it asks for) and the most one block may have.
constexpr size_t kSmemPerSm = 228 * 1024, kSmemPerBlock = 227 * 1024;

// Opt the kernel in to `bytes` of dynamic shared memory.  Without the attribute,
// static plus dynamic shared memory must stay within 48 KB, so a kernel with a
// little static memory (a work index, an abort flag) fails to launch just below
// 48 KB of dynamic memory: set it from 32 KB up.
template <typename K>
static cudaError_t ensure_smem(K kernel, size_t bytes) {
    if (bytes <= 32 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Blocks of a kernel that share an SM, asked for once (any host thread; all find the same number).
template <typename K>
static cudaError_t blocks_per_sm(std::atomic<int>& known, K kernel, int threads, size_t smem, int* out) {
    *out = known.load(std::memory_order_relaxed);
    if (*out > 0) return cudaSuccess;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kernel, threads, smem);
    if (e != cudaSuccess) return e;
    *out = std::max(1, *out);
    known.store(*out, std::memory_order_relaxed);
    return cudaSuccess;
}

template <typename T, int Q>
static cudaError_t launch_fwd_rows(const int32_t* X, const uint8_t* MX, const double* WX, int H, int W, int K, int Qs,
                                   cpx<T>* T1, const Tw<T>& tw, DevStatus* st, int conditional, int* popc,
                                   const unsigned char* need, cudaStream_t s) {
    using C = FwdRowsCfg<T, Q>;
    auto kern = k_fwd_rows<T, Q>;
    cudaError_t e = ensure_smem(kern, C::smem(Q, true));
    if (e != cudaSuccess) return e;
    dim3 grid(H, ((K + 1) / 2 + C::TPB - 1) / C::TPB);
    kern<<<grid, C::THREADS, C::smem(W, WX != nullptr), s>>>(X, MX, WX, H, W, K, Qs, T1, tw, st, conditional, popc,
                                                             need);
    return cudaGetLastError();
}

template <typename T, int P, int MMAX>
static cudaError_t launch_fwd_cols(const cpx<T>* T1, int H, int K, int Qh, int Qs, cpx<T>* F, const Tw<T>& tw,
                                   const DevStatus* st, int conditional, T out_scale, const unsigned char* need,
                                   int slices, int num_sms, cudaStream_t s) {
    using C = ColCfg<T, P, MMAX>;
    auto kern = k_fwd_cols<T, P, MMAX>;
    cudaError_t e = ensure_smem(kern, C::smem(P));
    if (e != cudaSuccess) return e;
    const long long items = (long long)((Qh + C::TPB - 1) / C::TPB) * K;
    long long slots = items;
    if (C::PIPE && num_sms > 0) {  // persistent: every resident block slot
        static std::atomic<int> known{0};
        int by_regs = 0;
        e = blocks_per_sm(known, kern, C::THREADS, 0, &by_regs);
        if (e != cudaSuccess) return e;
        const int by_smem = (int)(kSmemPerSm / (C::smem(H) + 1024));
        slots = (long long)std::max(1, std::min(by_regs, by_smem)) * num_sms;
    }
    kern<<<(int)std::min(items, slots), C::THREADS, C::smem(H), s>>>(T1, H, K, Qh, Qs, F, tw, st, conditional, out_scale, need, slices);
    return cudaGetLastError();
}

// The table of e^{-2 pi i k / N}, N = 2^l or 3 2^l.
template <typename T>
static const cpx<T>* tw_table(const Tw<T>& tw, int N) {
    return N % 3 == 0 ? tw.n3[ilog2_of(N / 3)] : tw.n[ilog2_of(N)];
}

template <typename T, int P, bool VOL, int MMAX>
static cudaError_t launch_pair_cols(const Geom& g, const PipeArgs<T>& a, cudaStream_t s) {
    using C = PairColsCfg<T, P, MMAX>;
    auto kern = k_pair_cols<T, P, VOL, MMAX>;
    const size_t smem = pair_cols_smem<T, P, MMAX>();
    cudaError_t e = ensure_smem(kern, smem);
    if (e != cudaSuccess) return e;
    // persistent grid: every resident block slot of the device, at most one per item
    static std::atomic<int> known{0};
    int per_sm = 0;
    e = blocks_per_sm(known, kern, C::THREADS, smem, &per_sm);
    if (e != cudaSuccess) return e;
    const long long np = a.plist ? a.chunk_cap : (long long)g.KA * g.KB;  // list mode: at most chunk_cap pairs
    const long long items = np * ((g.Ys + C::TPB - 1) / C::TPB) * (VOL ? (g.Dz + C::NDZ - 1) / C::NDZ : g.units);
    const int bps = a.cols_bps > 0 && a.cols_bps < per_sm ? a.cols_bps : per_sm;
    const long long slots = a.num_sms > 0 ? (long long)bps * a.num_sms : items;
    const int grid = (int)(items < slots ? items : slots);
    // a map's one launch counts in its status word, which is zeroed with it; the list launches
    // of the second precision, several per map, have a counter of their own
    int* ctr = &a.st->work;
    if (a.plist) {
        ctr = a.work_ctr;
        e = cudaMemsetAsync(ctr, 0, sizeof(int), s);
        if (e != cudaSuccess) return e;
    }
    kern<<<grid, C::THREADS, smem, s>>>(a.FA, a.FB, g.KA, g.KB, g.Qh, g.HA, g.HB, g.R, g.r0, g.r1, a.Y, a.tw,
                                        tw_table(a.tw, g.Q), a.st, a.conditional, ctr, g.DA, g.DB, g.R2, a.plist, a.lrange,
                                        a.chunk_off, a.chunk_cap, VOL ? 1 : g.units, g.split);
    return cudaGetLastError();
}

// Teams per block of the one-warp Tensor-Memory row kernel (rows_tm.cuh): blocks of 8 where two
// of them share an SM.  At Q = 2048 a block of 16 is the better one for more than 32 pairs when
// every row has an SM of its own, and the slower one beyond.  Time with 16 over time with 8, MI,
// outputs of 151 rows / 155 rows / 999 rows: 7 x 7 labels 0.97 / 1.18 / 1.27, 8 x 8 0.86 / 1.03 /
// 1.08, 11 x 11 0.90 / 1.09 / 1.14, 16 x 16 0.85 / 1.01 / 1.04 (2047 rows 1.01: 1.524 against
// 1.509 ms); AUTO and several angles per launch alike.  NMI, whose blocks of 8 spill, has no such
// line (151 / 999 rows: 8 x 8 0.84 / 1.06, 16 x 16 0.79 / 1.00) and takes 16 beyond 32 pairs.
template <int Q, bool NMI>
static int rows_tm_teams(const Geom& g, const PipeArgs<float>& a) {
    const int rows = g.units * (g.r1 - g.r0);
    if (a.tm_cols > 256) return 16;
    return Q == 2048 && g.KA * g.KB > 32 && (NMI || rows <= a.num_sms) ? 16 : 8;
}

template <int Q, bool NMI, int MODE, int NT>
static cudaError_t launch_rows_tm(const Geom& g, const PipeArgs<float>& a, cudaStream_t s) {
    using C = RowTmCfg<Q, NT>;
    auto kern = k_pair_rows_tm<Q, NMI, MODE, NT>;
    cudaError_t e = ensure_smem(kern, C::SMEM);
    if (e != cudaSuccess) return e;
    const bool ext = MODE == 2;
    CUtensorMap ymap;
    e = make_row_map(&ymap, a.Y, C::L, g.R, g.KA * g.KB);
    if (e != cudaSuccess) return e;
    const int grid = std::min(a.rows_grid, C::BLOCKS * a.num_sms);
    kern<<<grid, C::THREADS, C::SMEM, s>>>(ymap, g, a.tw, a.mi, a.n, a.st, a.tm_cols,
                                           ext && a.wait_polls > 0 ? a.wait_polls : kDefaultWaitPolls,
                                           ext ? a.withhold_row : -1, ext ? a.conditional : 0,
                                           ext ? a.ov : nullptr, ext ? a.ov_slot : nullptr,
                                           ext ? a.pair_res : nullptr);
    return cudaGetLastError();
}

template <int Q, bool NMI, int MODE>
static cudaError_t launch_rows_tm_mode(const Geom& g, const PipeArgs<float>& a, cudaStream_t s) {
    if constexpr (Q == 4096) {
        return launch_rows_tm<Q, NMI, MODE, 8>(g, a, s);
    } else if constexpr (Q % 3 == 0) {
        return launch_rows_tm<Q, NMI, MODE, 4>(g, a, s);
    } else {
        return rows_tm_teams<Q, NMI>(g, a) == 8 ? launch_rows_tm<Q, NMI, MODE, 8>(g, a, s)
                                                : launch_rows_tm<Q, NMI, MODE, 16>(g, a, s);
    }
}

template <typename T, int Q, bool NMI>
static cudaError_t launch_pair_rows_v(const Geom& g, const PipeArgs<T>& a, cudaStream_t s) {
    using C = RowCfg<T, Q>;
    if constexpr (std::is_same<T, float>::value && tm_rows(Q)) {
        if (a.tm_cols > 0 && !a.counts) {  // debug count maps: the generic kernel below
            const bool ext = a.ov_slot || a.pair_res || a.conditional || a.wait_polls > 0 || a.withhold_row >= 0;
            // the multi-unit kernel lives in its own translation unit (kernels_f32_rows_units.cu):
            // compiled next to the plain one, it changed the plain kernel's register allocation
            if (!ext && g.units > 1) return launch_rows_tm_units<Q, NMI>(g, a, s);
            return ext ? launch_rows_tm_mode<Q, NMI, 2>(g, a, s) : launch_rows_tm_mode<Q, NMI, 0>(g, a, s);
        }
    }
    size_t smem = pair_rows_smem<T, Q>(g.KB, a.cb_smem);
    if (a.cb_smem) {
        auto kern = k_pair_rows<T, Q, true, NMI>;
        // A map of few rows: a cluster of blocks per row, as many as the labels and the
        // resident blocks allow (64^2, K = 8, 127 rows: 1 block per row 16.5 us).  The blocks
        // of a cluster also hold a row of partial sums: where those do not fit, one block per
        // row.  (Where they leave fewer blocks per SM the split stays: 37 rows of 32 x 32
        // labels at Q = 512, exact, 8 blocks per row 164 us, 4 190 us.)
        const int ntask = g.units * (g.r1 - g.r0);
        const size_t smem_split = (smem + 15) / 16 * 16 + Q * (sizeof(EntAcc<NMI>) + sizeof(int));
        int split = 1;
        if (smem_split <= kSmemPerBlock)
            while (split < 8 && 2 * split <= g.KA && (long long)ntask * 2 * split <= a.rows_cap) split *= 2;
        if (split == 1) {
            cudaError_t e = ensure_smem(kern, smem);
            if (e != cudaSuccess) return e;
            kern<<<a.rows_grid, C::THREADS, smem, s>>>(a.Y, g, a.tw, a.cb_global, a.mi, a.n, a.counts, a.st,
                                                       a.prec_slot, a.conditional, a.ov, a.ov_slot, a.pair_res, 1);
            return cudaGetLastError();
        }
        smem = smem_split;
        cudaError_t e = ensure_smem(kern, smem);
        if (e != cudaSuccess) return e;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = split;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(ntask * split);
        cfg.blockDim = dim3(C::THREADS);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = s;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kern, (const cpx<T>*)a.Y, g, a.tw, a.cb_global, a.mi, a.n, a.counts, a.st,
                                  a.prec_slot, a.conditional, (const int32_t*)a.ov, a.ov_slot, a.pair_res, split);
    } else if constexpr (Q > 512) {  // Q <= 512: K_B (<= 64) x Q floats always fit in shared memory
        auto kern = k_pair_rows<T, Q, false, NMI>;
        cudaError_t e = ensure_smem(kern, smem);
        if (e != cudaSuccess) return e;
        kern<<<a.rows_grid, C::THREADS, smem, s>>>(a.Y, g, a.tw, a.cb_global, a.mi, a.n, a.counts, a.st,
                                                   a.prec_slot, a.conditional, a.ov, a.ov_slot, a.pair_res, 1);
    } else {
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// MI or NMI epilogue (CMIF_FLAG_NMI)
template <typename T, int Q>
static cudaError_t launch_pair_rows(const Geom& g, const PipeArgs<T>& a, cudaStream_t s) {
    return a.nmi ? launch_pair_rows_v<T, Q, true>(g, a, s) : launch_pair_rows_v<T, Q, false>(g, a, s);
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::fwd_rows(const Geom& g, const PipeArgs<T>& a, bool b_side, cudaStream_t s) {
    const double* wb = a.weighted ? a.WB : nullptr;
    const double* wa = a.weighted ? a.WA : nullptr;
    // volumes: the D slices of H rows are D * H rows of one image
    return b_side ? launch_fwd_rows<T, SZ>(a.B, a.MB, wb, g.DB * g.HB, g.WB, g.KB, g.Qs, a.T1B, a.tw, a.st,
                                           a.conditional, a.popB, a.needB, s)
                  : launch_fwd_rows<T, SZ>(a.A, a.MA, wa, g.DA * g.HA, g.WA, g.KA, g.Qs, a.T1A, a.tw, a.st,
                                           a.conditional, a.popA, a.needA, s);
}

// 1 / n for the unnormalised transforms (residues: n a power of two, 2^31 = 1)
template <typename T>
static T inverse_of(double n) {
    if constexpr (std::is_same<T, m31>::value) return m31_of(1u << (31 - (int)std::lround(std::log2(n))));
    else return T(1.0 / n);
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::fwd_cols(const Geom& g, const PipeArgs<T>& a, bool b_side, cudaStream_t s) {
    // B's spectra carry the 1/(P Q) of the unnormalised inverse transform (a power of two: exact)
    // volumes: K * D slice planes of H rows each (plane index label * D + z)
    auto go = [&](auto mm) {
        constexpr int MM = decltype(mm)::value;
        return b_side ? launch_fwd_cols<T, SZ, MM>(a.T1B, g.HB, g.KB * g.DB, g.Qh, g.Qs, a.FB, a.tw, a.st,
                                                   a.conditional, inverse_of<T>((double)g.P * (double)g.Q), a.needB,
                                                   g.DB, a.num_sms, s)
                      : launch_fwd_cols<T, SZ, MM>(a.T1A, g.HA, g.KA * g.DA, g.Qh, g.Qs, a.FA, a.tw, a.st,
                                                   a.conditional, T(1), a.needA, g.DA, a.num_sms, s);
    };
    if constexpr (kHasColVariant<T, SZ>) {
        if (a.col_m == 16) return go(std::integral_constant<int, 16>{});
    }
    return go(std::integral_constant<int, max_m<T>()>{});
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::pair_cols(const Geom& g, const PipeArgs<T>& a, cudaStream_t s) {
    if constexpr (kHasColVariant<T, SZ>) {
        if (a.col_m == 16)
            return g.Dz > 1 ? launch_pair_cols<T, SZ, true, 16>(g, a, s) : launch_pair_cols<T, SZ, false, 16>(g, a, s);
    }
    constexpr int MM = max_m<T>();
    return g.Dz > 1 ? launch_pair_cols<T, SZ, true, MM>(g, a, s) : launch_pair_cols<T, SZ, false, MM>(g, a, s);
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::pair_rows(const Geom& g, const PipeArgs<T>& a, cudaStream_t s) {
    return launch_pair_rows<T, SZ>(g, a, s);
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::pair_rows_counts(const Geom& g, const PipeArgs<T>& a, cudaStream_t s) {
    using C = RowCntCfg<T, SZ>;
    auto kern = k_pair_rows_counts<T, SZ>;
    cudaError_t e = ensure_smem(kern, C::SMEM);
    if (e != cudaSuccess) return e;
    const long long tasks = (long long)a.chunk_cap * (g.r1 - g.r0);
    const long long blocks = std::min<long long>((tasks + C::NT - 1) / C::NT, 8LL * (a.num_sms > 0 ? a.num_sms : 152));
    kern<<<(int)std::max<long long>(1, blocks), C::THREADS, C::SMEM, s>>>(a.Y, g, a.tw, a.lrange, a.chunk_off,
                                                                          a.chunk_cap, a.ov, a.st);
    return cudaGetLastError();
}

template <typename T, int SZ>
size_t Sized<T, SZ>::rows_smem(int KB, bool cb_smem) {
    return pair_rows_smem<T, SZ>(KB, cb_smem);
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::rows_max_blocks(int KB, bool cb_smem, int* out) {
    const size_t smem = pair_rows_smem<T, SZ>(KB, cb_smem);
    if (cb_smem) {
        auto kern = k_pair_rows<T, SZ, true, false>;
        cudaError_t e = ensure_smem(kern, smem);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kern, RowCfg<T, SZ>::THREADS, smem);
    }
    if constexpr (SZ > 512) {
        auto kern = k_pair_rows<T, SZ, false, false>;
        cudaError_t e = ensure_smem(kern, smem);
        if (e != cudaSuccess) return e;
        return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kern, RowCfg<T, SZ>::THREADS, smem);
    } else {
        return cudaErrorInvalidValue;  // not reached: the B-marginals always fit in shared memory
    }
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::pair_rows_w(const Geom& g, const PipeArgs<T>& a, cudaStream_t s) {
    using C = RowWCfg<SZ>;
    cudaError_t e = ensure_smem(k_pair_rows_w<SZ>, C::SMEM);
    if (e != cudaSuccess) return e;
    k_pair_rows_w<SZ><<<a.rows_grid_w, C::THREADS, C::SMEM, s>>>(a.Y, g, a.tw, a.cbw, a.mi, a.nw, a.st);
    return cudaGetLastError();
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::rows_w_max_blocks(int* out) {
    using C = RowWCfg<SZ>;
    cudaError_t e = ensure_smem(k_pair_rows_w<SZ>, C::SMEM);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, k_pair_rows_w<SZ>, C::THREADS, C::SMEM);
}

template <typename T, int SZ>
int Sized<T, SZ>::tm_cols(int KA, int KB) {
    if constexpr (std::is_same<T, float>::value && tm_rows(SZ)) {
        const int need = tm_cols_needed(tm_swapped(SZ, KA, KB) ? KA : KB, SZ);
        return need <= 512 ? tm_alloc_cols(need) : 0;
    } else {
        (void)KA;
        (void)KB;
        return 0;
    }
}

template <typename T, int SZ>
cudaError_t Sized<T, SZ>::tm_max_blocks(int tm_cols, int* out) {
    *out = 0;
    if constexpr (std::is_same<T, float>::value && tm_rows(SZ)) {
        // The blocks that share an SM: as many as the kernel is bounded for (registers; shared
        // memory is less than that), within the SM's 512 TMEM columns.  (The occupancy query
        // answers 1 for a kernel that allocates Tensor Memory.)
        constexpr int NT = SZ % 3 == 0 ? 4 : 8;
        *out = std::min(RowTmCfg<SZ, NT>::BLOCKS, 512 / tm_cols);
        return cudaSuccess;
    } else {
        (void)tm_cols;
        return cudaSuccess;
    }
}

}  // namespace cmif
