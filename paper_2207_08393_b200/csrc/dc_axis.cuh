// Readout axis of 3-D problems with an arbitrary mask whose lengths dc_brick.cuh does not take: transform, k-space work,
// inverse transform, in place on the workspace that the middle passes of dc_mid.cuh leave as (unit, q, n0, n2), the rows q in their order (raw
// ky = q / BY + RY * (q % BY)).  A block takes KC neighbouring kz columns of one (unit, q): n0 pieces of 8 KC bytes
// that lie n2 apart, so a tile's pieces share DRAM pages (with the volume's natural order they lie a plane apart:
// 96 x 160 x 128, 6 coils: 306 us for both calls against 150 us here).  Bound by HBM: 16 bytes per element, 24 with
// measurements.  One exchange buffer: the second stage and its inverse work in place on the runs they read.
// Mask weights are requested first, the measurements they admit are copied to shared memory while the transform runs.
#pragma once
#include "size_ops.cuh"

namespace gleam {

enum AxisMode { AXIS_MID = 0, AXIS_ADJ = 1, AXIS_GRADY = 2 };

struct AxisArgs {
    cf* W;
    const cf* y; cf* ky_out;       // measurements (may be null) / k-space output (AXIS_GRADY), (B,C,T,n0,n1,n2)
    const float* mask;             // (B,T,n0,n1,n2), or (B,T,n1,n2) if mask_plane
    int mask_plane;
    float scale, scale2;           // g / sqrt(Ntot) (times eta: AXIS_GRADY), 1 / Ntot
    int C, T, n1, n2, ry;
    long long nunits;
};

template <class P, int KC>
struct Axis {
    static constexpr int N = P::N;
    static constexpr int TH = KC * P::MAXBF;                      // a multiple of 32 (below) for every plan with KC >= 16
    static constexpr int THREADS = (TH + 31) / 32 * 32;
    static constexpr int X_ELEMS = (P::S == 2) ? P::R0 * P::LS1 * KC : 0;
    static constexpr size_t BYTES = sizeof(cf) * (X_ELEMS + (P::S == 2 ? N : 0));
    static constexpr size_t Y_BYTES = sizeof(cf) * P::RL * THREADS;
    static constexpr int REGS = (2 * cmax(P::R0, P::RL) + P::RL + 32 + 7) / 8 * 8;
    // Blocks that the register bound keeps resident.  Butterflies of 15 and 16 points get two blocks of 256 threads and 128
    // registers: with three (80 registers) weights and addresses are spilled and fewer loads are in flight (forward / VJP, us a
    // pass: 256 x 256 x 160, 8 coils 799 / 503 -> 466 / 388, 240 x 96 x 96 150 / 115 -> 114 / 98, 192 x 96 x 128 145 / 119 -> 127 /
    // 107, 160 x 160 x 128, 6 coils 160 / 125 -> 142 / 114).  Smaller ones want the blocks (with one fewer 96 x 160 x 128 82 / 70
    // -> 111 / 97, 64 x 160 x 128 39 / 33 -> 43 / 35); a 640-point block of 512 threads has 128 registers at most and spills 148 B.
    static constexpr int BLOCKS = cmax(1, cmin(cmin(cmax(P::R0, P::RL) > 12 ? 2 : 16, 2048 / THREADS), 65536 / (THREADS * REGS)));
};

template <class P, int KC, int MODE>
__global__ void __launch_bounds__(Axis<P, KC>::THREADS, Axis<P, KC>::BLOCKS)
axis_kernel(const AxisArgs a) {
    grid_dependency_wait();
    using AX = Axis<P, KC>;
    constexpr int N = P::N, R0 = P::R0, RL = P::RL, BF0 = P::BF0, BFL = P::BFL, LS1 = P::LS1;
    extern __shared__ __align__(16) float2 smem[];
    cf* sX = smem;
    cf* sTw = smem + AX::X_ELEMS;                                 // stage twiddles, [k][j]
    cf* sY = sTw + (P::S == 2 ? N : 0);                           // measurements, slots of the thread's own
    const int tid = threadIdx.x, l = tid % KC, jt = tid / KC;
    const unsigned tiles = (unsigned)((a.n2 + KC - 1) / KC);
    const unsigned o = blockIdx.x / tiles;                        // unit * n1 + q
    const int i = (int)(blockIdx.x - o * tiles) * KC + l;
    const bool ok = i < a.n2, act0 = ok && jt < BF0, actL = ok && jt < BFL;
    const unsigned unit = o / (unsigned)a.n1;
    const int q = (int)(o - unit * (unsigned)a.n1), by = a.n1 / a.ry;
    const unsigned bc = unit / (unsigned)a.T;
    const long long bt = (long long)(bc / (unsigned)a.C) * a.T + (unit - bc * (unsigned)a.T);
    const int s1 = shift_half(q / by + a.ry * (q % by), a.n1), s2 = shift_half(i, a.n2);
    const long long plane = (long long)a.n1 * a.n2, V = N * plane, at = (long long)s1 * a.n2 + s2;
    cf* w = a.W + (long long)o * N * a.n2 + i;

    float mv[RL];
    if (actL && MODE != AXIS_GRADY) {
        const float* mk = a.mask + bt * V + at;
#pragma unroll
        for (int k = 0; k < RL; ++k) mv[k] = mk[shift_half(jt + BFL * k, N) * plane];
    }
    cf v[R0];
    if (MODE != AXIS_ADJ) {
#pragma unroll
        for (int m = 0; m < R0; ++m) v[m] = act0 ? w[(jt + BF0 * m) * a.n2] : make_float2(0.f, 0.f);
    }
    if (P::S == 2) for (int e = tid; e < N; e += AX::THREADS) sTw[e] = unit_root_fwd<N>(((e / BF0) * (e % BF0)) % N);
    if (actL && MODE != AXIS_GRADY && a.y) {
        // measurements at unsampled positions are not read (they may hold anything)
        const cf* yy = a.y + unit * V + at;
#pragma unroll
        for (int k = 0; k < RL; ++k)
            if (mv[k] != 0.f) cp_async8(sY + k * AX::THREADS + tid, yy + shift_half(jt + BFL * k, N) * plane);
    }
    cp_async_commit();
    cf u[RL];
    if (MODE != AXIS_ADJ) {
        Dft<R0, -1>::run(v);
        if (P::S == 2) {
            __syncthreads();
            if (jt < BF0) {
#pragma unroll
                for (int k = 0; k < R0; ++k) sX[(k * LS1 + jt) * KC + l] = (k == 0) ? v[0] : cmul(v[k], sTw[k * BF0 + jt]);
            }
            __syncthreads();
            if (jt < BFL) {
#pragma unroll
                for (int m = 0; m < RL; ++m) u[m] = sX[(jt * LS1 + m) * KC + l];
                Dft<RL, -1>::run(u);
            }
        } else {
#pragma unroll
            for (int k = 0; k < RL; ++k) u[k] = v[k % R0];
        }
    }
    cp_async_wait<0>();
    if (MODE == AXIS_GRADY) {
        if (actL) {
            const float* mk = a.mask + (a.mask_plane ? bt * plane : bt * V) + at;
            cf* dst = a.ky_out + unit * V + at;
#pragma unroll
            for (int k = 0; k < RL; ++k) {
                const int s0 = shift_half(jt + BFL * k, N);
                dst[s0 * plane] = cscale(u[k], (((s0 + s1 + s2) & 1) ? -a.scale : a.scale) * mk[a.mask_plane ? 0 : s0 * plane]);
            }
        }
        return;
    }
    if (actL) {
#pragma unroll
        for (int k = 0; k < RL; ++k) {
            const float wt = mv[k] * mv[k] * a.scale2;
            if (a.y) {
                const cf yv = (mv[k] != 0.f) ? sY[k * AX::THREADS + tid] : make_float2(0.f, 0.f);
                const float f = (((shift_half(jt + BFL * k, N) + s1 + s2) & 1) ? -a.scale : a.scale) * mv[k];
                u[k] = (MODE == AXIS_ADJ) ? make_float2(-f * yv.x, -f * yv.y) : make_float2(fmaf(wt, u[k].x, -f * yv.x), fmaf(wt, u[k].y, -f * yv.y));
            } else {
                u[k] = cscale(u[k], wt);
            }
        }
    }
    if (P::S == 2) {
        if (MODE == AXIS_ADJ) __syncthreads();                    // the twiddles are visible
        if (jt < BFL) {
            Dft<RL, +1>::run(u);
#pragma unroll
            for (int m = 0; m < RL; ++m) sX[(jt * LS1 + m) * KC + l] = u[m];
        }
        __syncthreads();
        if (jt < BF0) {
#pragma unroll
            for (int k = 0; k < R0; ++k) { const cf r = sX[(k * LS1 + jt) * KC + l]; v[k] = (k == 0) ? r : cmulc(r, sTw[k * BF0 + jt]); }
        }
    } else {
#pragma unroll
        for (int k = 0; k < R0; ++k) v[k] = u[k % RL];
    }
    if (act0) {
        Dft<R0, +1>::run(v);
#pragma unroll
        for (int m = 0; m < R0; ++m) w[(jt + BF0 * m) * a.n2] = v[m];
    }
}

struct AxisOps {
    int n0;
    cudaError_t (*launch)(int mode, const AxisArgs&, cudaStream_t);
};

// KC: 32 columns (256-byte pieces) where the exchange buffer and the block stay small, 16 otherwise.
template <class P>
struct AxisImpl {
    static constexpr int KC = (P::N <= 128 && P::MAXBF <= 16) ? 32 : 16;
    using AX = Axis<P, KC>;
    template <int MODE> static cudaError_t go(const AxisArgs& a, cudaStream_t s) {
        static PerDevice done;
        cudaError_t e = ensure_smem(axis_kernel<P, KC, MODE>, AX::BYTES + AX::Y_BYTES, done);
        if (e != cudaSuccess) return e;
        const long long blocks = a.nunits * a.n1 * ((a.n2 + KC - 1) / KC);
        if (blocks <= 0) return cudaSuccess;
        if (blocks > 2147483647LL) return cudaErrorInvalidConfiguration;
        return launch_overlapped(true, axis_kernel<P, KC, MODE>, dim3((unsigned)blocks), dim3(AX::THREADS), AX::BYTES + (a.y ? AX::Y_BYTES : 0), s, a);
    }
    static cudaError_t launch(int mode, const AxisArgs& a, cudaStream_t s) {
        switch (mode) {
            case AXIS_MID: return go<AXIS_MID>(a, s);
            case AXIS_ADJ: return go<AXIS_ADJ>(a, s);
            case AXIS_GRADY: return go<AXIS_GRADY>(a, s);
        }
        return cudaErrorInvalidValue;
    }
};

}  // namespace gleam
