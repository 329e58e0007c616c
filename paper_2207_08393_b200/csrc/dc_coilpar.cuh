// One-pass row kernel for 2-D problems with few lines: the coils of a line group are transformed by different warps of
// one block instead of one after another by one warp.
//
// Latency-bound: with a warp per group the call lasts C coils, each a chain of loads, two exchanges and four butterfly
// stages (0.6 to 1.5 us), on a nearly empty GPU.  Here warp w takes the coils w, w + W, ...; the coil images come to
// rest in shared memory, and the conjugate-sensitivity sum then runs over the coils in order, spread over all threads
// by image element: the same operations in the same order as in the other one-pass kernels.
// One 64 x 64 slice of 8 coils: prepared step 12.5 -> 4.3 us, VJP 4.7 -> 3.4 us in a replayed chain.
#pragma once
#include "dc_warpline.cuh"

namespace gleam {

template <class P>
struct CoilPar {
    static constexpr int N = P::N, R0 = P::R0, RL = P::RL, S = P::S;
    static constexpr int TPL = pow2_ceil(cmax(P::BF0, P::BFL));   // lanes per line
    static constexpr int LW = 32 / TPL;                           // lines per group
    static constexpr int EXL = (S == 2) ? P::SM_A : 0;            // exchange elements per line
    static constexpr int LINE = LW * N;
    // float2 units: x, scaled mask^2 (floats) and unit masks per line, exchange per warp, then one line group per coil
    static constexpr int OFF_M = LINE, OFF_U = OFF_M + (LINE + 1) / 2, OFF_E = OFF_U + LW * P::BFL;
    static constexpr size_t bytes(int warps, int coils) { return sizeof(cf) * (size_t)(OFF_E + warps * LW * EXL + coils * LINE); }
    static constexpr size_t LIMIT = 200 * 1024;
    // shared memory of an SM, and what a block takes beyond `bytes`: the kernel's static arrays and the 1 KB reserved
    static constexpr size_t SM_BYTES = 228 * 1024, BLOCK_BYTES = 1024 + 2 * 64 * sizeof(double) + 192;
};

// Sixteen warps have 128 registers each: butterflies of 32 points beside 16 or 20 spill 170 to 320 B (512 and 640 points, 172 B
// and 324 B without z), one reason why those lengths come here for a single round only.
template <class P, bool HAS_Z, bool ADJ>
__global__ void __launch_bounds__(512)
coilpar_kernel(const RowArgs a) {
    grid_dependency_wait();
    grid_launch_dependents();
    using CP = CoilPar<P>;
    constexpr int N = P::N, R0 = P::R0, RL = P::RL, TPL = CP::TPL, LW = CP::LW, EXL = CP::EXL, LINE = CP::LINE;
    extern __shared__ __align__(16) float2 smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, warps = blockDim.x >> 5;
    cf* sX = smem;
    float* sM = reinterpret_cast<float*>(smem + CP::OFF_M);
    UnitMask* sU = reinterpret_cast<UnitMask*>(smem + CP::OFF_U);
    cf* sE = smem + CP::OFF_E + warp * LW * EXL;
    cf* sV = smem + CP::OFF_E + warps * LW * EXL;
    __shared__ bool s_few[LW];                             // the line's sampled entries are as few as other kernels stage
    const long long row0 = (long long)blockIdx.x * LW;

    // offsets of a line of this group (identical arithmetic wherever a line index is needed)
    auto line_of = [&](int ll, long long& x_off, long long& s_off, long long& k_off, long long& bt, int& b) -> bool {
        const long long row = row0 + ll;
        if (row >= a.nrows) return false;
        bt = row / a.RPB;
        const int ri = (int)(row - bt * a.RPB);
        b = (int)(bt / a.T);
        const int t = (int)(bt - (long long)b * a.T);
        x_off = (bt * a.RPB + ri) * (long long)N;
        s_off = (((long long)(b * a.C) * a.Ts + (a.Ts > 1 ? t : 0)) * a.RPB + ri) * N;
        k_off = (((long long)(b * a.C) * a.T + t) * a.RPB + ri) * N;
        return true;
    };
    const long long s_stride = (long long)a.Ts * a.RPB * N, k_stride = (long long)a.T * a.RPB * N;

    // ---- x, mask weights and unit masks of the lines: one warp per line ----
    for (int ll = warp; ll < LW; ll += warps) {
        long long x_off = 0, s_off = 0, k_off = 0, bt = 0; int b = 0;
        const bool ok = line_of(ll, x_off, s_off, k_off, bt, b);
        if (HAS_Z) {
            const int cnt = line_units<P::BFL, RL>(a.mask + bt * N, ok, lane, sU + ll * P::BFL, ADJ ? nullptr : sM + ll * N);
            if (lane == 0) s_few[ll] = cnt <= z_stage(N);
        }
#pragma unroll 8
        for (int k0 = 0; k0 < N; k0 += 32) {
            const int k = k0 + lane;
            if (k >= N) break;
            if (!ADJ) sX[ll * N + k] = ok ? load_image(a.x, x_off + k, a.x_planar, b, a.plane) : make_float2(0.f, 0.f);
            if (!HAS_Z) { const float mv = ok ? a.mask[bt * N + shift_half(k, N)] : 0.f; sM[ll * N + k] = mv * mv * (1.0f / N); }
        }
    }
    const int l = lane / TPL, j = lane % TPL;
    const bool a0 = j < P::BF0, aL = j < P::BFL;
    long long x_off = 0, s_off = 0, k_off = 0, bt = 0; int b = 0;
    const bool row_ok = line_of(l, x_off, s_off, k_off, bt, b);
    cf tw0[R0];
    if (P::S == 2) {
#pragma unroll
        for (int k = 0; k < R0; ++k) tw0[k] = unit_root_fwd<N>((j * k) % N);
    }
    __syncthreads();

    // ---- coil images: S x, transform, k-space update, inverse transform ----
    for (int c = warp; c < a.C; c += warps) {
        cf v[R0], u[RL];
        if (!ADJ) {
            if (a0) {
                const cf* sp = a.sens + s_off + c * s_stride + j;
#pragma unroll
                for (int m = 0; m < R0; ++m) v[m] = cmul(row_ok ? sp[P::BF0 * m] : make_float2(0.f, 0.f), sX[l * N + j + P::BF0 * m]);
                Dft<R0, -1>::run(v);
            }
            if (P::S == 2) {
                if (a0) {
#pragma unroll
                    for (int k = 0; k < R0; ++k) sE[l * EXL + k * P::LS1 + j] = (k == 0) ? v[0] : cmul(v[k], tw0[k]);
                }
                __syncwarp();
                if (aL) {
#pragma unroll
                    for (int m = 0; m < RL; ++m) u[m] = sE[l * EXL + j * P::LS1 + m];
                    Dft<RL, -1>::run(u);
                }
                __syncwarp();
            } else {
#pragma unroll
                for (int k = 0; k < RL; ++k) u[k] = v[k % R0];
            }
        }
        if (aL) {
            if (HAS_Z) {
                const UnitMask um = sU[l * P::BFL + j];
                unit_update<P::BFL, RL, ADJ>(u, um.bits, sM + l * N + j, a.z + k_off + c * k_stride + um.first, s_few[l]);
            } else {
#pragma unroll
                for (int k = 0; k < RL; ++k) u[k] = cscale(u[k], sM[l * N + j + P::BFL * k]);
            }
        }
        if (P::S == 2) {
            if (aL) {
                Dft<RL, +1>::run(u);
#pragma unroll
                for (int m = 0; m < RL; ++m) sE[l * EXL + j * P::LS1 + m] = u[m];
            }
            __syncwarp();
            if (a0) {
#pragma unroll
                for (int k = 0; k < R0; ++k) { const cf r = sE[l * EXL + k * P::LS1 + j]; v[k] = (k == 0) ? r : cmulc(r, tw0[k]); }
            }
        } else {
#pragma unroll
            for (int k = 0; k < R0; ++k) v[k] = u[k % RL];
        }
        if (a0) {
            Dft<R0, +1>::run(v);
#pragma unroll
            for (int m = 0; m < R0; ++m) sV[c * LINE + l * N + j + P::BF0 * m] = v[m];
        }
        __syncwarp();
    }
    __syncthreads();

    // ---- conjugate-sensitivity sum over the coils in order, update, Re<x, out> and <out, out> per row ----
    // tasks: (line, segment of its elements), one warp each
    __shared__ double s_dot[2][64];
    const int segs = warps > LW ? warps / LW : 1;
    for (int task = warp; task < LW * segs; task += warps) {
        const int ll = task % LW, seg = task / LW;
        double dsum = 0.0, nsum = 0.0;
        if (line_of(ll, x_off, s_off, k_off, bt, b)) {
            for (int n = seg * 32 + lane; n < N; n += 32 * segs) {
                const cf* sp = a.sens + s_off + n;
                cf acc = coil_sum_start(a.aty, x_off + n);
#pragma unroll 8
                for (int c = 0; c < a.C; ++c) {
                    const cf sv = sp[c * s_stride], vv = sV[c * LINE + ll * N + n];
                    acc.x = fmaf(sv.x, vv.x, fmaf(sv.y, vv.y, acc.x));
                    acc.y = fmaf(sv.x, vv.y, fmaf(-sv.y, vv.x, acc.y));
                }
                const cf xv = ADJ ? make_float2(0.f, 0.f) : sX[ll * N + n];
                const cf ov = make_float2(fmaf(-a.eta, acc.x, xv.x), fmaf(-a.eta, acc.y, xv.y));
                store_image(a.out, x_off + n, ov, a.out_planar, b, a.plane);
                if (a.dot_rows != nullptr) { dsum += (double)xv.x * ov.x + (double)xv.y * ov.y; nsum += (double)ov.x * ov.x + (double)ov.y * ov.y; }
            }
        }
        if (a.dot_rows != nullptr) {
            for (int o = 16; o > 0; o >>= 1) { dsum += __shfl_down_sync(0xffffffffu, dsum, o); nsum += __shfl_down_sync(0xffffffffu, nsum, o); }
            if (lane == 0) { s_dot[0][task] = dsum; s_dot[1][task] = nsum; }
        }
    }
    if (a.dot_rows != nullptr) {
        __syncthreads();
        if (tid < LW && row0 + tid < a.nrows) {
            double d = 0.0, n = 0.0;
            for (int seg = 0; seg < segs; ++seg) { d += s_dot[0][seg * LW + tid]; n += s_dot[1][seg * LW + tid]; }
            a.dot_rows[row0 + tid] = d;
            a.dot_rows[a.nrows + row0 + tid] = n;
        }
    }
}

}  // namespace gleam
