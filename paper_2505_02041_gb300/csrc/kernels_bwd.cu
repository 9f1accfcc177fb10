// kernels_bwd.cu -- adjoint HRC kernels for sm_103a (standalone launches of
// the bodies in bwd_bodies.cuh) and the backward launch sequence.
#include <type_traits>

#include <cstring>

#include "bwd_bodies.cuh"
#include "launch.h"

namespace hrc {

template <int P, int C, class GIN>
__global__ void __launch_bounds__(256) k_adj_sum(Plan pl, const GIN *__restrict__ gF) {
    __shared__ __align__(16) unsigned char smem[sizeof(typename Prec<P>::A) * C * 32 * 33];
    body_adj_sum<P, C, GIN>(pl, gF, blockIdx.x, blockIdx.y, smem);
}

// Row and v-block of this block (see the forward merge kernels).
__device__ __forceinline__ void row_block_b(const Plan &pl, long long &row, int &vb) {
    if (pl.vmajor) { row = blockIdx.y; vb = blockIdx.x; }
    else { row = blockIdx.x; vb = blockIdx.y; }
}

// Level 0 (odd shifts), four v per thread like the levels above.
template <int P, int C>
__global__ void __launch_bounds__(512) k_adj_R0(Plan pl, RowSplitB rs) {
    long long row;
    int vb;
    row_block_b(pl, row, vb);
    body_adj_R0<P, C>(pl, rs, row, vb);
}

template <int P, int C, bool ENV>
__global__ void __launch_bounds__(512) k_adj_T0(Plan pl, RowSplitB rs) {
    long long row;
    int vb;
    row_block_b(pl, row, vb);
    body_adj_T0<P, C, ENV>(pl, rs, row, vb);
}

// Levels n >= 1: four v per thread.  With a pair of v these kernels issued in
// about 65 % of the slots, most of it addresses and range tests, so a thread that
// shares them over four entries is faster (40-46 % of the slots, waiting for
// loads instead) -- provided that a shifted range is tested once for all its
// rows (rows4, shifted4, interval4): with a
// test per channel the merge-up reverse took 513 us instead of 387 (1024^2,
// C = 3, fp32).  Pairs -> quads, us, C = 3 / C = 1 at 1024^2 fp32: merge-down
// reverse 272 -> 247 / 188 -> 144, merge-up reverse 374 -> 366 / 260 -> 196;
// bf16 C = 3: 277 -> 240, 354 -> 323.  (C = 4: see k_adj_merge_up.)
template <int P, int C>
__global__ void __launch_bounds__(512) k_adj_R4(Plan pl, RowSplitB rs, int n) {
    long long row;
    int vb;
    row_block_b(pl, row, vb);
    body_adj_R4<P, C>(pl, rs, n, row, vb);
}

template <int P, int C, bool ENV>
__global__ void __launch_bounds__(512) k_adj_T4(Plan pl, RowSplitB rs, int n) {
    long long row;
    int vb;
    row_block_b(pl, row, vb);
    body_adj_T4<P, C, ENV>(pl, rs, n, row, vb);
}

template <int P, int C, bool ENV>
__global__ void __launch_bounds__(512) k_adj_merge_up4(Plan pl, RowSplitB rs, int n) {
    long long row;
    int vb;
    row_block_b(pl, row, vb);
    body_adj_merge_up4<P, C, ENV>(pl, rs, n, row, vb);
}

// The merge-up reverse of four channels, and of fp64, takes a pair of v per
// thread: quads need 96-100 registers (fp64 62-128 and spills) against 40 (fp64
// 36-100).  Quads / pairs, us: C = 4 1024^2 fp32 542 / 474, bf16 455 / 436,
// 512^2 fp32 137 / 120, 256^2 51 / 43, whole backward of 32 batched scenes of
// 256^2 fp32 2321 / 2013; fp64 256^2 C = 1 .. 4 70 / 65, 106 / 92, 133 / 117,
// 166 / 143.  Single C = 4 grids below 128^2 keep the quads (64^2 18 / 20).
template <int P, int C> constexpr bool amu_pairs() { return C == 4 || P == P_FP64; }

template <int P, int C, bool ENV>
__global__ void __launch_bounds__(512) k_adj_merge_up(Plan pl, RowSplitB rs, int n) {
    long long row;
    int vb;
    row_block_b(pl, row, vb);
    body_adj_merge_up<P, C, ENV>(pl, rs, n, row, vb);
}

template <int P, int C, class IN>
__global__ void __launch_bounds__(ADJ_THREADS, 3) k_adj_trace(Plan pl, const IN *__restrict__ e, const IN *__restrict__ s,
                                                   IN *__restrict__ ge, IN *__restrict__ gs, int pair,
                                                   const __grid_constant__ CUtensorMap tme,
                                                   const __grid_constant__ CUtensorMap tms, int use_tma) {
    extern __shared__ __align__(128) unsigned char tb_smem[];
    body_adj_trace<P, C, IN>(pl, e, s, ge, gs, pair, blockIdx.x, blockIdx.y, tb_smem, use_tma ? &tme : nullptr,
                             use_tma ? &tms : nullptr, 3, pair == 1);
}

// Both pairs' adjoint traces in one launch.  FB = 2: block b < n0 takes tile b
// of pair 0 (into ge / gs), the others pair 1 (into the planes of frame 2).
// FB = 1: every frame its own blocks and planes, frames 0 .. 3 in order.
// k_adj_combine adds the planes.
template <int P, int C, class IN, int FB>
__global__ void __launch_bounds__(ADJ_THREADS, 3) k_adj_trace_all(Plan pl, const IN *__restrict__ e,
                                                                  const IN *__restrict__ s, IN *ge, IN *gs, int n0, int n1,
                                                                  int nx0, int nx1, const __grid_constant__ CUtensorMap me0,
                                                                  const __grid_constant__ CUtensorMap ms0,
                                                                  const __grid_constant__ CUtensorMap me1,
                                                                  const __grid_constant__ CUtensorMap ms1, int use_tma) {
    extern __shared__ __align__(128) unsigned char tb_smem[];
    constexpr int BF = 2 / FB;                            // blocks per tile
    const int b = (int)blockIdx.x, pair = b >= BF * n0, r = pair ? b - BF * n0 : b, nt = pair ? n1 : n0;
    const int half = FB == 1 && r >= nt, t = half ? r - nt : r, nx = pair ? nx1 : nx0, q = 2 * pair + half;
    if (FB == 1 || pair) {
        ge = adj_part<IN>(pl, q, 0);
        gs = adj_part<IN>(pl, q, 1);
    }
    body_adj_trace<P, C, IN>(pl, e, s, ge, gs, pair, t % nx, t / nx, tb_smem, use_tma ? (pair ? &me1 : &me0) : nullptr,
                             use_tma ? (pair ? &ms1 : &ms0) : nullptr, FB == 2 ? 3 : 1 << half, false, FB == 1 || pair);
}

// dL/de and dL/dsigma from the planes of k_adj_trace_all: (q0 + q1) + (q2 + q3).
template <int C, class IN, int FB>
__global__ void __launch_bounds__(256) k_adj_combine(Plan pl, IN *__restrict__ ge, IN *__restrict__ gs) {
    const long long HW = (long long)pl.W * pl.H, n = (C + 1) * HW;
    const IN *pe[4], *ps[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        pe[q] = adj_part<IN>(pl, q, 0);
        ps[q] = adj_part<IN>(pl, q, 1) - C * HW;
    }
    for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL) {
        const bool es = i < C * HW;
        IN *o = (es ? ge : gs - C * HW) + i;
        if constexpr (FB == 2) {
            *o += (es ? pe[2] : ps[2])[i];
        } else {
            IN v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = (es ? pe[q] : ps[q])[i];
            *o = (v[0] + v[1]) + (v[2] + v[3]);
        }
    }
}

// ---------------------------------------------------------------------------
// Host-side launcher of the whole backward pass.
// ---------------------------------------------------------------------------
namespace {

RowSplitB split_rows(const Plan &pl, int kind, int n) {
    // kind 0: R_0 rows (q, x); 1: rows of gR_{n+1} (q, x', j); 2: rows of gT_n (q, x, k);
    // 3: rows of gT_{n-1} for the level-n merge-up reverse
    RowSplitB rs;
    long long acc = 0;
    for (int q = 0; q < 4; ++q) {
        rs.start[q] = acc;
        const QuadGeom &g = pl.q[q];
        long long rows = 0;
        if (kind == 0) rows = g.N >= 1 ? g.Un[0] : 0;
        else if (kind == 1) rows = (n + 1 < g.N) ? (long long)(g.Un[n + 1] - 1) * (2 << n) : 0;
        else if (kind == 2)   // level 0: odd columns only
            rows = (g.N >= 1 && n <= g.N && !adj_T_fused(n, g.N))
                       ? (n == 0 ? (long long)(g.Un[0] / 2) * 2 : (long long)(g.Un[n] - 1) * ((1 << n) + 1)) : 0;
        else rows = (n >= 3 && n <= g.N) ? (long long)(g.Un[n - 1] - 1) * ((1 << (n - 1)) + 1) : 0;
        acc += rows;
    }
    rs.start[4] = acc;
    return rs;
}

dim3 row_grid_b(const Plan &pl, long long rows, int per_block) {
    int Vmax = 0;
    for (int q = 0; q < 4; ++q) Vmax = pl.q[q].V > Vmax ? pl.q[q].V : Vmax;
    const unsigned vb = (unsigned)((Vmax + per_block - 1) / per_block);
    return pl.vmajor ? dim3(vb, (unsigned)rows) : dim3((unsigned)rows, vb);
}

}  // namespace

template <int P, int C>
static cudaError_t bwd_impl(const Plan &pl, const RayTable &rt, const void *e, const void *s, const void *gF,
                            void *ge, void *gs, bool recompute, cudaStream_t st, int *launches, Recorder *rec) {
    using IN = typename std::conditional<P == P_FP64, double, float>::type;
    // A block of quads covers the v of a block of pairs twice as wide: 512 threads
    // leave most of a row's threads without work and, from C = 2 on, too few
    // blocks on an SM (backward, fp32, us, 512 / 256 threads: C = 3 1024^2 951 /
    // 858, 256^2 133 / 107, 4096x64 845 / 650; C = 1 4096x64 505 / 544).
    const int mt = C >= 2 && pl.mthreads > 256 ? 256 : pl.mthreads;
    const bool env = plan_has_env(pl);   // kernels compiled for an environment map
    int Nmax = 0, Nmin = pl.q[0].N;
    for (int q = 0; q < 4; ++q) {
        Nmax = pl.q[q].N > Nmax ? pl.q[q].N : Nmax;
        Nmin = pl.q[q].N < Nmin ? pl.q[q].N : Nmin;
    }
    const double ab = P == P_FP64 ? 8.0 : 4.0;
    const double img = double(pl.W) * pl.H;
    // live columns x >= 1 only (column 0 is dead)
    auto gTbytes = [&](int q, int n) {
        const QuadGeom &g = pl.q[q];
        return (n < 0 || n > g.N) ? 0.0 : double(t_live_rows(n, g.Un[n])) * g.V * (pl.C + 1) * ab;
    };
    auto gRbytes = [&](int q, int n) {
        const QuadGeom &g = pl.q[q];
        return (n < 0 || n >= g.N) ? 0.0 : double(g.Un[n] - 1) * (1 << n) * g.V * pl.C * ab;
    };
    // T_0..T_N and R_1..R_{N-1}: recomputed from (e, s), or the ones the last
    // forward left in the plan's buffers (the inputs unchanged since, by
    // contract).
    if (recompute) {
        cudaError_t err = launch_forward(pl, rt, e, s, nullptr, st, launches, rec);
        if (err != cudaSuccess) return err;
    }
    {
        double by = img * pl.C * ab;
        for (int q = 0; q < 4; ++q) by += gRbytes(q, 0);
        rec->begin(K_ADJ_SUM, 0, by);
        k_adj_sum<P, C, IN><<<dim3((pl.W + 31) / 32, (pl.H + 31) / 32), 256, 0, st>>>(pl, (const IN *)gF);
        rec->end();
        ++*launches;
    }
    for (int n = 0; n + 1 < Nmax; ++n) {
        RowSplitB rs = split_rows(pl, 1, n);
        if (rs.start[4] == 0) continue;
        double by = 0;
        for (int q = 0; q < 4; ++q)
            if (n + 1 < pl.q[q].N)
                by += gRbytes(q, n) + gRbytes(q, n + 1) + bytes_T(pl, q, n) / (pl.C + 1) / 2 +
                      bytes_T(pl, q, n + 1) / (pl.C + 1) / 2;
        rec->begin(K_ADJ_MERGE_DOWN, n, by);
        if (n >= 1) k_adj_R4<P, C><<<row_grid_b(pl, rs.start[4], 4 * mt), mt, 0, st>>>(pl, rs, n);
        else k_adj_R0<P, C><<<row_grid_b(pl, rs.start[4], 4 * mt), mt, 0, st>>>(pl, rs);
        rec->end();
        ++*launches;
    }
    for (int n = 0; n <= Nmax; ++n) {
        RowSplitB rs = split_rows(pl, 2, n);
        if (rs.start[4] == 0) continue;
        double by = 0;
        for (int q = 0; q < 4; ++q)
            if (pl.q[q].N >= 1 && n <= pl.q[q].N && !adj_T_fused(n, pl.q[q].N))
                by += gTbytes(q, n) + gRbytes(q, n) + gRbytes(q, n - 1) + bytes_R(pl, q, n) + bytes_R(pl, q, n + 1);
        rec->begin(K_ADJ_MERGE_DOWN, n, by);
        if (n >= 1) {
            if (env) k_adj_T4<P, C, true><<<row_grid_b(pl, rs.start[4], 4 * mt), mt, 0, st>>>(pl, rs, n);
            else k_adj_T4<P, C, false><<<row_grid_b(pl, rs.start[4], 4 * mt), mt, 0, st>>>(pl, rs, n);
        } else {
            if (env) k_adj_T0<P, C, true><<<row_grid_b(pl, rs.start[4], 4 * mt), mt, 0, st>>>(pl, rs);
            else k_adj_T0<P, C, false><<<row_grid_b(pl, rs.start[4], 4 * mt), mt, 0, st>>>(pl, rs);
        }
        rec->end();
        ++*launches;
    }
    for (int n = Nmax; n >= 3; --n) {
        RowSplitB rs = split_rows(pl, 3, n);
        if (rs.start[4] == 0) continue;
        double by = 0;
        for (int q = 0; q < 4; ++q)
            if (n <= pl.q[q].N)   // merge-up reverse + the fused merge-down part of level n-1
                by += gTbytes(q, n - 1) + gTbytes(q, n) + bytes_T(pl, q, n - 1) + gRbytes(q, n - 1) +
                      gRbytes(q, n - 2) + bytes_R(pl, q, n - 1) + bytes_R(pl, q, n);
        rec->begin(K_ADJ_MERGE_UP, n, by);
        bool pairs = false;
        if constexpr (amu_pairs<P, C>()) {
            pairs = P == P_FP64 || !pl.solo || pl.W * pl.H >= 128 * 128;
            // Grids 8 times as long as wide: every row gets the blocks of the
            // longest, most of them empty; twice the threads halve those (fp32, us,
            // 128 / 256 threads: 4096x64 684 / 379, 2048x128 209 / 172, 1024^2 474 /
            // 483; fp64 C = 4 987 / 1110, so not there).
            const int lo = pl.W < pl.H ? pl.W : pl.H, hi = pl.W < pl.H ? pl.H : pl.W;
            const int mp = hi >= 8 * lo && hi > 2 * mt && mt <= 256 && !(P == P_FP64 && C == 4) ? 2 * mt : pl.mthreads;
            if (pairs) {
                const dim3 grid = row_grid_b(pl, rs.start[4], 2 * mp);
                if (env) k_adj_merge_up<P, C, true><<<grid, mp, 0, st>>>(pl, rs, n);
                else k_adj_merge_up<P, C, false><<<grid, mp, 0, st>>>(pl, rs, n);
            }
        }
        if constexpr (P != P_FP64) {
            const dim3 grid = row_grid_b(pl, rs.start[4], 4 * mt);
            if (!pairs && env) k_adj_merge_up4<P, C, true><<<grid, mt, 0, st>>>(pl, rs, n);
            else if (!pairs) k_adj_merge_up4<P, C, false><<<grid, mt, 0, st>>>(pl, rs, n);
        }
        rec->end();
        ++*launches;
    }
    {
        using A = typename Prec<P>::A;
        const size_t smem = adj_trace_smem<A, C>();
        const int nx0 = pair_tiles_x(0, pl.W), nx1 = pair_tiles_x(1, pl.W);
        const int n0 = nx0 * pair_tiles_y(0, pl.H), n1 = nx1 * pair_tiles_y(1, pl.H);
        // Both pairs in one launch and their sum in a second one: two launches
        // of 4.5 waves each (1024^2, 456 blocks resident) become one of 9, and
        // pair 1 no longer reads what pair 0 wrote.  While a block per tile and
        // frame fits the GPU at once (3 blocks per SM at C <= 3, 2 at C = 4, 1 in
        // fp64, of 152), a tile's two frames are halved too.  Adjoint trace in all, C = 3, fp32,
        // us, one pair after the other / pairs at once / frames at once:
        // 64^2 40.9 / 24.4 / 17.3, 256^2 44.0 / 30.2 / 35.9, 512^2 97 / 79 / 85,
        // 1024^2 269 / 254 / 309, 2048^2 987 / 966 / 1216; on either side of the
        // lines, pairs / frames at once: fp64 C = 1 128^2 117 / 82, 144^2 118 /
        // 145, C = 4 170 / 108, 174 / 203; C = 4 fp32 176^2 28.2 / 22.5, 200^2 34.7 /
        // 36.5; C = 1 224^2 25.5 / 22.1, 256^2 24.5 / 28.6.  The planes need dL/dR_1
        // buffers (N >= 2 in every frame).
        const bool all = Nmin >= 2;
        if (all) {
            const int room = 152 * (P == P_FP64 ? 1 : (C == 4 ? 2 : 3));
            const bool one = pl.solo && 2 * (n0 + n1) <= room;   // a frame per block
            const double planes = one ? 4.0 : 2.0;
            double by = img * (pl.C + 1) * ab * (1.0 + planes);   // the inputs, the planes written
            for (int q = 0; q < 4; ++q)
                for (int n = 0; n <= 2; ++n) by += gTbytes(q, n);
            rec->begin(K_ADJ_TRACE, 0, by);
            CUtensorMap m[4];
            std::memset(m, 0, sizeof(m));
            const int use_tma = (P != P_FP64 && encode_image_maps(pl, e, s, PT_RU, PT_RV, m[0], m[1]) &&
                                 encode_image_maps(pl, e, s, PT_RV, PT_RU, m[2], m[3])) ? 1 : 0;
            const IN *ei = (const IN *)e, *si = (const IN *)s;
            IN *geo = (IN *)ge, *gso = (IN *)gs;
            const long long nb = ((long long)(pl.C + 1) * pl.W * pl.H + 255) / 256;
            const unsigned cb = (unsigned)(nb < 2432 ? nb : 2432);
            if (one)
                k_adj_trace_all<P, C, IN, 1><<<2 * (n0 + n1), ADJ_THREADS, smem, st>>>(pl, ei, si, geo, gso, n0, n1, nx0, nx1,
                                                                                    m[0], m[1], m[2], m[3], use_tma);
            else
                k_adj_trace_all<P, C, IN, 2><<<n0 + n1, ADJ_THREADS, smem, st>>>(pl, ei, si, geo, gso, n0, n1, nx0, nx1, m[0],
                                                                              m[1], m[2], m[3], use_tma);
            rec->end();
            rec->begin(K_ADJ_TRACE, 1, img * (pl.C + 1) * ab * (planes + 1.0));   // the planes read, the sums
            if (one) k_adj_combine<C, IN, 1><<<cb, 256, 0, st>>>(pl, geo, gso);
            else k_adj_combine<C, IN, 2><<<cb, 256, 0, st>>>(pl, geo, gso);
            rec->end();
            *launches += 2;
        }
        for (int pair = 0; pair < 2 && !all; ++pair) {
            // the inputs, the gradients written; pair 1 adds to them
            double by = img * (pl.C + 1) * ab * (pair == 0 ? 2.0 : 3.0);
            for (int q = 2 * pair; q < 2 * pair + 2; ++q)
                for (int n = 0; n <= 2; ++n) by += gTbytes(q, n);
            dim3 grid(pair_tiles_x(pair, pl.W), pair_tiles_y(pair, pl.H));
            rec->begin(K_ADJ_TRACE, pair, by);
            CUtensorMap me, ms;
            std::memset(&me, 0, sizeof(me));
            std::memset(&ms, 0, sizeof(ms));
            const int use_tma = (P != P_FP64 && encode_image_maps(pl, e, s, pair == 0 ? PT_RU : PT_RV,
                                                                  pair == 0 ? PT_RV : PT_RU, me, ms))
                                    ? 1 : 0;
            k_adj_trace<P, C, IN><<<grid, ADJ_THREADS, smem, st>>>(pl, (const IN *)e, (const IN *)s, (IN *)ge, (IN *)gs,
                                                                   pair, me, ms, use_tma);
            rec->end();
            ++*launches;
        }
    }
    return cudaGetLastError();
}

template <int P>
static cudaError_t bwd_prec(const Plan &pl, const RayTable &rt, const void *e, const void *s, const void *gF,
                            void *ge, void *gs, bool rc, cudaStream_t st, int *launches, Recorder *rec) {
    switch (pl.C) {
    case 1: return bwd_impl<P, 1>(pl, rt, e, s, gF, ge, gs, rc, st, launches, rec);
    case 2: return bwd_impl<P, 2>(pl, rt, e, s, gF, ge, gs, rc, st, launches, rec);
    case 3: return bwd_impl<P, 3>(pl, rt, e, s, gF, ge, gs, rc, st, launches, rec);
    default: return bwd_impl<P, 4>(pl, rt, e, s, gF, ge, gs, rc, st, launches, rec);
    }
}

template <int P>
static cudaError_t prepare_bwd_prec() {
    using IN = typename std::conditional<P == P_FP64, double, float>::type;
    using A = typename Prec<P>::A;
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *fn, size_t bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    set((const void *)k_adj_trace<P, 1, IN>, adj_trace_smem<A, 1>());
    set((const void *)k_adj_trace_all<P, 1, IN, 1>, adj_trace_smem<A, 1>());
    set((const void *)k_adj_trace_all<P, 1, IN, 2>, adj_trace_smem<A, 1>());
    set((const void *)k_adj_trace<P, 2, IN>, adj_trace_smem<A, 2>());
    set((const void *)k_adj_trace_all<P, 2, IN, 1>, adj_trace_smem<A, 2>());
    set((const void *)k_adj_trace_all<P, 2, IN, 2>, adj_trace_smem<A, 2>());
    set((const void *)k_adj_trace<P, 3, IN>, adj_trace_smem<A, 3>());
    set((const void *)k_adj_trace_all<P, 3, IN, 1>, adj_trace_smem<A, 3>());
    set((const void *)k_adj_trace_all<P, 3, IN, 2>, adj_trace_smem<A, 3>());
    set((const void *)k_adj_trace<P, 4, IN>, adj_trace_smem<A, 4>());
    set((const void *)k_adj_trace_all<P, 4, IN, 1>, adj_trace_smem<A, 4>());
    set((const void *)k_adj_trace_all<P, 4, IN, 2>, adj_trace_smem<A, 4>());
    return e;
}

cudaError_t prepare_backward_kernels() {
    cudaError_t e = prepare_bwd_prec<P_FP32>();
    if (e == cudaSuccess) e = prepare_bwd_prec<P_FP16>();
    if (e == cudaSuccess) e = prepare_bwd_prec<P_BF16>();
    if (e == cudaSuccess) e = prepare_bwd_prec<P_FP64>();
    return e;
}

cudaError_t launch_backward(const Plan &pl, const RayTable &rt, const void *e, const void *s, const void *gF,
                            void *ge, void *gs, bool recompute, cudaStream_t st, int *launches, Recorder *rec) {
    switch (pl.prec) {
    case P_FP32: return bwd_prec<P_FP32>(pl, rt, e, s, gF, ge, gs, recompute, st, launches, rec);
    case P_FP16: return bwd_prec<P_FP16>(pl, rt, e, s, gF, ge, gs, recompute, st, launches, rec);
    case P_BF16: return bwd_prec<P_BF16>(pl, rt, e, s, gF, ge, gs, recompute, st, launches, rec);
    default: return bwd_prec<P_FP64>(pl, rt, e, s, gF, ge, gs, recompute, st, launches, rec);
    }
}

}  // namespace hrc
