// K-space part of 3-D problems with an arbitrary mask in one pass over the workspace (unit, k0, j, n0, n2) of the row-tile
// passes: radix-BY stage of ky, readout transform, mask and measurements, and the mirror image back.  A block holds a
// brick of BY x n0 x W elements (W neighbouring kz of one unit and k0 group) in shared memory; the ky stages are dealt to
// all threads, the readout stages of a k1 belong to one warp, and all work in place on the slots they read.  Against the
// three launches it replaces (MID_FWD, the readout pass of dc_axis.cuh and MID_INV) the workspace is read and written once
// instead of three times.  Forward / VJP call, us: 6 coils of 96 x 160 x 128 206 / 193 -> 160 / 143, 8 of 128 x 128 x 128 333 /
// 322 -> 220 / 199, 8 of 48 x 320 x 320 671 / 632 -> 547 / 495, 4 of 320 x 120 x 96 317 / 283 -> 245 / 223, 4 of 32 x 96 x 96
// 30 / 30 -> 26 / 25.  Bound by issue and what keeps it from its slots: at 6 coils of 96 x 160 x 128, two bricks an SM, 51 %
// (forward) and 52 % (VJP) active, next to the FP32 pipe at 34 and 40 % and L2 at 7.2 and 6.2 TB/s; the ky stages and the copies
// before and after them alternate.  One to four bricks fit an SM, a single one in 39 of the 146 variants.
//
// The bricks leave little of L1, and a load occupies a line of it until it is served: loading the brick through registers
// left too few requests in flight (VJP of the first 156 us), and so did measurements one by one (forward 176 us).
// Both are copied 16 bytes at a time past L1.
#pragma once
#include "size_ops.cuh"
#include "dc_entry.h"

namespace gleam {

struct BrickArgs {
    cf* V;
    const cf* y;                   // measurements (B,C,T,n0,n1,n2); null: VJP
    const float* mask;             // (B,T,n0,n1,n2)
    int adjoint;                   // minus A^H y's k-space alone, nothing is read from the workspace
    float scale, scale2;           // g / sqrt(Ntot), 1 / Ntot
    int C, T, n1, n2, ry;
    long long nunits;
};

template <class P, int BY>
struct Brick {
    static constexpr int N = P::N, R0 = P::R0, RL = P::RL, BF0 = P::BF0;
    static constexpr size_t LIMIT = 227 * 1024;
    static constexpr size_t bytes(int w, int ls) { return sizeof(cf) * ((size_t)BY * R0 * ls * w + N + BY); }
    // Columns: pieces of 128 bytes in global memory where two blocks of them fit an SM, else the widest that fit.  Two blocks
    // of 4 columns instead of one of 8 measured slower (4 coils of 160 x 320 x 128, VJP 394 -> 433 us), 4 columns instead of
    // the three passes faster (4 of 184 x 184 x 92 318 / 291 -> 244 / 230 us).
    static constexpr int W = 2 * (bytes(16, RL) + 1024) <= LIMIT ? 16 : bytes(8, odd_up(RL)) <= LIMIT ? 8 : 4;
    static constexpr int LS = W == 16 ? RL : odd_up(RL);       // run of a second-stage butterfly; with 8 columns two runs share the banks
    static constexpr int ROW = R0 * LS;                        // slots of a readout line
    static constexpr size_t BYTES = bytes(W, LS);
    // Where the three passes are slower, over 187 volumes of all pairs of lengths (three passes / brick, forward and VJP together
    // unless stated).  Not for single-stage readouts, which occur in small tests only; radix 32 (384 points spill 204 B and read
    // 548 B back, the variants taken at most 84 B and 200 B: 3 coils of 384 x 96 x 96, forward 269 -> 307 us); 16 x 15 and 16 x 16
    // points (two large butterflies in few registers: 0.90 to 1.14, mean 1.0); 23 points of ky next to smaller ones of the readout
    // (0.94 to 1.31, mean 1.04).  23-point readouts gain most, 1.02 to 2.0.
    // A^H y has the readout pass and one middle pass to replace: 0.92 to 1.33 with 80 to 128 points, 1.04 to 2.5 with
    // 23-point stages, 0.78 to 1.2 elsewhere.
    static constexpr bool FITS = P::S == 2 && RL <= 23 && !(R0 == 16 && (RL == 15 || RL == 16)) && (BY != 23 || RL == 23) && BYTES <= LIMIT;
    static constexpr bool ADJOINT = RL == 23 || (N >= 80 && N <= 128);
    static constexpr int slot(int i0) { return (i0 / BF0) * LS + i0 % BF0; }
    // The readout stages of UC columns of one k1 belong to one warp, which needs no block barrier between them.
    static constexpr int UC = W == 16 && BY < 10 ? 8 : W;
    static constexpr int UNITS = BY * (W / UC);
    static constexpr int RMAX = cmax(BY, cmax(R0, RL));
    static constexpr bool PRIME = RMAX > 4 && RMAX % 2 == 1 && smallest_odd_factor(RMAX) == RMAX;
    static constexpr int REGS = ((PRIME ? 4 : 2) * RMAX + 32 + 7) / 8 * 8;
    static constexpr int BLOCKS = cmax(1, cmin(4, (int)(LIMIT / (BYTES + 1024))));
    // warps: the fewest that give the fewest rounds of butterflies, within the registers
    static constexpr int rounds(int items, int each) { return (items + each - 1) / each; }
    static constexpr int cost(int warps) {
        return 2 * (BY * rounds(N * W, 32 * warps) + rounds(UNITS, warps) * (R0 * rounds(BF0 * UC, 32) + RL * rounds(R0 * UC, 32)));
    }
    static constexpr int pick() {
        int best = 4;
        for (int n = 5; n <= 24; ++n) if (32 * n * BLOCKS * REGS <= 65536 && 32 * n * BLOCKS <= 2048 && cost(n) < cost(best)) best = n;
        return 32 * best;
    }
    static constexpr int THREADS = pick();
};

// v[k] times tw[k], or its conjugate (DIR = +1), for k > 0; two twiddles a load
template <int R, int DIR>
__device__ __forceinline__ void twiddle_pairs(cf (&v)[R], const cf* tw) {
#pragma unroll
    for (int k = 0; k < R; k += 2) {
        if (k + 1 == R) { v[k] = DIR < 0 ? cmul(v[k], tw[k]) : cmulc(v[k], tw[k]); break; }
        const float4 t = *reinterpret_cast<const float4*>(tw + k);
        const cf a = make_float2(t.x, t.y), b = make_float2(t.z, t.w);
        if (k > 0) v[k] = DIR < 0 ? cmul(v[k], a) : cmulc(v[k], a);
        v[k + 1] = DIR < 0 ? cmul(v[k + 1], b) : cmulc(v[k + 1], b);
    }
}

template <class P, int BY>
__global__ void __launch_bounds__(Brick<P, BY>::THREADS, Brick<P, BY>::BLOCKS)
brick_kernel(const BrickArgs a) {
    grid_dependency_wait();
    using BR = Brick<P, BY>;
    constexpr int N = P::N, R0 = P::R0, RL = P::RL, BF0 = P::BF0, W = BR::W, LS = BR::LS, ROW = BR::ROW, TH = BR::THREADS;
    extern __shared__ __align__(16) float2 smem[];
    cf* sT = smem;                                               // (k1, readout slot, kz)
    cf* sTw = smem + BY * ROW * W;                               // readout stage twiddles, [j][k]
    cf* sKy = sTw + N;                                           // w_n1^(j k0)
    const int tid = threadIdx.x;
    const unsigned tiles = (unsigned)((a.n2 + W - 1) / W);
    const unsigned o = blockIdx.x / tiles;                       // unit * ry + k0
    const int kz0 = (int)(blockIdx.x - o * tiles) * W;
    const unsigned unit = o / (unsigned)a.ry;
    const int k0 = (int)(o - unit * (unsigned)a.ry);
    const unsigned bc = unit / (unsigned)a.T;
    const long long bt = (long long)(bc / (unsigned)a.C) * a.T + (unit - bc * (unsigned)a.T);
    // element offsets inside a volume fit 32 bits (lengths up to 640)
    const unsigned plane = (unsigned)(a.n1 * a.n2), sj = (unsigned)(N * a.n2);
    const long long V = (long long)N * plane;
    cf* w = a.V + (long long)o * BY * sj + kz0;
    // The whole brick is requested at once, past L1 (most of which is shared memory here), each pair to its place.
    if (!a.adjoint) {
        for (int t = tid; t < N * (W / 2); t += TH) {
            const int p = t % (W / 2), i0 = t / (W / 2);
            if (kz0 + 2 * p >= a.n2) continue;
            cf* e = sT + BR::slot(i0) * W + 2 * p;
            const cf* g = w + (unsigned)(i0 * a.n2 + 2 * p);
#pragma unroll
            for (int j = 0; j < BY; ++j) { cp_async16(e + j * ROW * W, g); g += sj; }
        }
        cp_async_commit();
    }
    for (int e = tid; e < N; e += TH) sTw[e] = unit_root_fwd<N>(((e / R0) * (e % R0)) % N);
    if (tid < BY) {
        double s, q;
        sincospi(2.0 * ((tid * k0) % a.n1) / a.n1, &s, &q);
        sKy[tid] = make_float2((float)q, (float)-s);
    }
    cp_async_wait<0>();
    __syncthreads();
    // forward ky stage: thread (readout position, kz)
    cf c[BY];
    if (!a.adjoint) {
#pragma unroll 1
        for (int t = tid; t < N * W; t += TH) {
            cf* e = sT + BR::slot(t / W) * W + t % W;
#pragma unroll
            for (int j = 0; j < BY; ++j) c[j] = e[j * ROW * W];
            twiddle_pairs<BY, -1>(c, sKy);
            Dft<BY, -1, true>::run(c);
#pragma unroll
            for (int k = 0; k < BY; ++k) e[k * ROW * W] = c[k];
        }
        __syncthreads();
    }
    constexpr int UC = BR::UC, WARPS = TH / 32;
    const int lane = tid & 31;
#pragma unroll 1
    for (int un = tid >> 5; un < BR::UNITS; un += WARPS) {
        const int b = un / (W / UC), l0 = (un % (W / UC)) * UC;
        cf* line = sT + b * ROW * W + l0;
        const int s1 = shift_half(k0 + a.ry * b, a.n1);
        const float* mk = a.mask + bt * V + (unsigned)(s1 * a.n2);
        const cf* yy = a.y + unit * V + (unsigned)(s1 * a.n2);
        if (!a.adjoint) {
            // first readout stage
#pragma unroll 1
            for (int t = lane; t < BF0 * UC; t += 32) {
                const int l = t % UC, jt = t / UC;
                cf* e = line + jt * W + l;
                cf v[R0];
#pragma unroll
                for (int m = 0; m < R0; ++m) v[m] = e[m * LS * W];
                Dft<R0, -1, true>::run(v);
                twiddle_pairs<R0, -1>(v, sTw + jt * R0);
#pragma unroll
                for (int k = 0; k < R0; ++k) e[k * LS * W] = v[k];
            }
            __syncwarp();
        }
        // Second readout stage, k-space work, its inverse.  The measurements come to the slots that the butterfly has read
        // while it runs, two neighbouring kz at a time where one of them was sampled; what lies at an unsampled position may
        // be anything and is not used.
#pragma unroll 1
        for (int t = lane; t - lane < R0 * UC; t += 32) {
            const int l = t % UC, jt = t / UC, s2 = shift_half(kz0 + l0 + l, a.n2);
            const bool ok = t < R0 * UC && kz0 + l0 + l < a.n2;
            auto offset = [&](int k, int kz) -> unsigned {       // of the centred readout position of jt + R0 k
                if (RL % 2 == 0) return jt * plane + kz + (unsigned)(k < RL / 2 ? k + RL / 2 : k - RL / 2) * (R0 * plane);
                return (unsigned)shift_half(jt + R0 * k, N) * plane + kz;
            };
            float mv[RL];
#pragma unroll
            for (int k = 0; k < RL; ++k) mv[k] = ok ? mk[offset(k, s2)] : 0.f;
            cf* e = line + jt * LS * W + l;
            cf u[RL];
            if (!a.adjoint && ok) {
#pragma unroll
                for (int m = 0; m < RL; ++m) u[m] = e[m * W];
            }
            if (a.y) {
                unsigned bits = 0u;
#pragma unroll
                for (int k = 0; k < RL; ++k) bits |= (mv[k] != 0.f ? 1u : 0u) << k;
                if (a.n2 % 4 == 0) {                             // pairs stay pairs under the half shift
                    __syncwarp();                                // both lanes have read their slots (a shuffle orders no memory)
                    bits |= __shfl_xor_sync(0xffffffffu, bits, 1);
                    const int odd = lane & 1;
#pragma unroll
                    for (int k2 = 0; k2 < RL; k2 += 2) {         // shared between the lanes of the pair
                        const int k = k2 + odd;
                        if ((bits >> k) & 1u) cp_async16(e - odd + k * W, yy + offset(k, s2 - odd));
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < RL; ++k) if ((bits >> k) & 1u) cp_async8(e + k * W, yy + offset(k, s2));
                }
                cp_async_commit();
            }
            if (!a.adjoint) Dft<RL, -1, true>::run(u);
            if (a.y) {
                static_assert(N % 2 == 0 && R0 % 2 == 0, "one sign for all k");
                const float sign = ((shift_half(jt, N) + s1 + s2) & 1) ? -a.scale : a.scale;
                cp_async_wait<0>();
                __syncwarp();
#pragma unroll
                for (int k = 0; k < RL; ++k) {
                    const cf yv = (mv[k] != 0.f) ? e[k * W] : make_float2(0.f, 0.f);
                    const float f = sign * mv[k], wt = mv[k] * mv[k] * a.scale2;
                    u[k] = a.adjoint ? make_float2(-f * yv.x, -f * yv.y) : make_float2(fmaf(wt, u[k].x, -f * yv.x), fmaf(wt, u[k].y, -f * yv.y));
                }
            } else {
#pragma unroll
                for (int k = 0; k < RL; ++k) u[k] = cscale(u[k], mv[k] * mv[k] * a.scale2);
            }
            Dft<RL, +1, true>::run(u);
            if (ok) {
#pragma unroll
                for (int m = 0; m < RL; ++m) e[m * W] = u[m];
            }
        }
        __syncwarp();
#pragma unroll 1
        for (int t = lane; t < BF0 * UC; t += 32) {
            const int l = t % UC, jt = t / UC;
            cf* e = line + jt * W + l;
            cf v[R0];
#pragma unroll
            for (int k = 0; k < R0; ++k) v[k] = e[k * LS * W];
            twiddle_pairs<R0, +1>(v, sTw + jt * R0);
            Dft<R0, +1, true>::run(v);
#pragma unroll
            for (int m = 0; m < R0; ++m) e[m * LS * W] = v[m];
        }
    }
    __syncthreads();
    for (int t = tid; t < N * W; t += TH) {
        const int l = t % W, i0 = t / W;
        if (kz0 + l >= a.n2) continue;
        const cf* e = sT + BR::slot(i0) * W + l;
#pragma unroll
        for (int k = 0; k < BY; ++k) c[k] = e[k * ROW * W];
        Dft<BY, +1, true>::run(c);
        twiddle_pairs<BY, +1>(c, sKy);
        const unsigned at = (unsigned)(i0 * a.n2 + l);
#pragma unroll
        for (int j = 0; j < BY; ++j) w[at + j * sj] = c[j];
    }
}

// *taken: the call was launched here (the brick fits an SM and BY is one of a two-stage ky plan)
template <class P>
struct BrickImpl {
    template <int BY> static cudaError_t go(const BrickArgs& a, cudaStream_t s, bool* taken) {
        using BR = Brick<P, BY>;
        if constexpr (!BR::FITS) return cudaSuccess;
        else {
            if (a.adjoint && !BR::ADJOINT) return cudaSuccess;
            static PerDevice done;
            cudaError_t e = ensure_smem(brick_kernel<P, BY>, BR::BYTES, done);
            if (e != cudaSuccess) return e;
            const long long blocks = a.nunits * a.ry * ((a.n2 + BR::W - 1) / BR::W);
            if (blocks > 2147483647LL) return cudaSuccess;
            *taken = true;
            if (blocks <= 0) return cudaSuccess;
            if ((e = prof_mark(GLEAM_K_COL_MID_FULL, s)) != cudaSuccess) return e;
            return launch_overlapped(true, brick_kernel<P, BY>, dim3((unsigned)blocks), dim3(BR::THREADS), BR::BYTES, s, a);
        }
    }
    static cudaError_t launch(const BrickArgs& a, cudaStream_t s, bool* taken) {
        *taken = false;
        if (a.ry < 2) return cudaSuccess;                    // a single-stage ky has no k0 groups
        switch (a.n1 / a.ry) {
            case 4: return go<4>(a, s, taken);
            case 5: return go<5>(a, s, taken);
            case 6: return go<6>(a, s, taken);
            case 8: return go<8>(a, s, taken);
            case 10: return go<10>(a, s, taken);
            case 12: return go<12>(a, s, taken);
            case 15: return go<15>(a, s, taken);
            case 16: return go<16>(a, s, taken);
            case 20: return go<20>(a, s, taken);
            case 23: return go<23>(a, s, taken);
            default: return cudaSuccess;
        }
    }
};

typedef cudaError_t (*BrickLaunch)(const BrickArgs&, cudaStream_t, bool* taken);

}  // namespace gleam
