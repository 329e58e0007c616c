// Warp-resident one-pass row kernel (contiguous axis) for plans whose stages need at most 32
// butterflies per line: every warp owns LW whole lines, so the stage hand-over through shared
// memory needs only __syncwarp(), warps never wait for one another, and the next coil's operands
// stream into shared memory with cp.async while the current coil is transformed.
//
//   out = x - eta * sum_c conj(S_c) Fraw^H ( m2 .* Fraw(S_c x) - z_c )
#pragma once
#include "dc_kernels.cuh"

namespace gleam {

constexpr int pow2_ceil(int v) { int p = 1; while (p < v) p *= 2; return p; }

template <class P, bool HAS_Z = false>
struct WarpLine {
    static constexpr int N = P::N, R0 = P::R0, RL = P::RL, S = P::S;
    static constexpr int BFMAX = cmax(P::BF0, P::BFL);
    static constexpr bool ELIGIBLE = (S <= 2) && (BFMAX <= 32) && (N % 2 == 0);
    static constexpr int TPL = pow2_ceil(BFMAX);          // lanes per line
    static constexpr int LW = 32 / TPL;                   // lines per warp
    static constexpr int EXL = (S == 2) ? P::SM_A : 0;    // exchange elements per line
    // per-warp shared memory, in float2 units: S[2], z[2], x, exchange, m2 (floats, N/2 float2 per line), unit masks.
    // Up to KCAP sampled z entries per line are staged (lines with more read z straight from global memory)
    static constexpr int TILE = LW * N;
    static constexpr int KCAP = z_stage(N);
    static constexpr int KSTRIDE = KCAP;
    static constexpr int KTILE = LW * KSTRIDE;
    static constexpr int OFF_S = 0, OFF_K = 2 * TILE, OFF_X = OFF_K + (HAS_Z ? 2 * KTILE : 0),
                         OFF_EX = OFF_X + TILE, OFF_M2 = OFF_EX + LW * EXL + (LW * EXL) % 2;
    static constexpr int OFF_U = OFF_M2 + TILE / 2;       // masks of the units (last-stage butterflies) of every line
    static constexpr int WARP_ELEMS = OFF_U + (HAS_Z ? LW * P::BFL : 0) + 2;
    static constexpr int WARP_ELEMS_ALIGNED = (WARP_ELEMS + 1) / 2 * 2;   // keep 16-byte alignment per warp
};

// ADJ (with z): A^H y, the image is zero and the forward stages are left out
template <class P, int WARPS, bool HAS_Z, bool ADJ>
__global__ void __launch_bounds__(WARPS * 32)
warpline_kernel(const RowArgs a) {
    grid_dependency_wait();
    using WL = WarpLine<P, HAS_Z>;
    constexpr int KCAP = WL::KCAP, KTILE = WL::KTILE, KSTRIDE = WL::KSTRIDE;
    constexpr int N = P::N, R0 = P::R0, RL = P::RL, TPL = WL::TPL, LW = WL::LW, TILE = WL::TILE;
    extern __shared__ __align__(16) float2 smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cf* wsm = smem + (size_t)warp * WL::WARP_ELEMS_ALIGNED;
    cf* sS = wsm + WL::OFF_S;
    cf* sK = wsm + WL::OFF_K;
    cf* sX = wsm + WL::OFF_X;
    cf* sE = wsm + WL::OFF_EX;
    float* sM = reinterpret_cast<float*>(wsm + WL::OFF_M2);
    UnitMask* sU = reinterpret_cast<UnitMask*>(wsm + WL::OFF_U);

    const int l = lane / TPL, j = lane % TPL;
    const bool a0 = j < P::BF0, aL = j < P::BFL;

    cf tw0[R0];
    if (P::S == 2) {
#pragma unroll
        for (int k = 0; k < R0; ++k) tw0[k] = unit_root_fwd<N>((j * k) % N);
    }

    const long long ngroups = (a.nrows + LW - 1) / LW;
    const long long wstride = (long long)gridDim.x * WARPS;
    if (wstride >= ngroups) grid_launch_dependents();      // a single round: the next launch may come in
    constexpr bool use_z = HAS_Z;

    for (long long g = (long long)blockIdx.x * WARPS + warp; g < ngroups; g += wstride) {
        // ---- element offsets of this lane's line; other lines' offsets come by shuffle ----
        const long long row = g * LW + l;
        const bool row_ok = row < a.nrows;
        const unsigned rowu = row_ok ? (unsigned)row : 0u;       // host side guarantees nrows < 2^31
        const unsigned bt = rowu / (unsigned)a.RPB;
        const int ri = (int)(rowu - bt * (unsigned)a.RPB);
        const int b = (int)(bt / (unsigned)a.T), t = (int)(bt - (unsigned)b * (unsigned)a.T);
        const long long x_off = ((long long)bt * a.RPB + ri) * N;
        const long long s_off = (((long long)(b * a.C) * a.Ts + (a.Ts > 1 ? t : 0)) * a.RPB + ri) * N;
        const long long k_off = (((long long)(b * a.C) * a.T + t) * a.RPB + ri) * N;
        const long long s_stride = (long long)a.Ts * a.RPB * N;
        const long long k_stride = (long long)a.T * a.RPB * N;

        int k_cnt = 0;       // sampled positions of this line (z; set below, when the mask row is scanned)

        auto issue_coil = [&](int c, int buf) {
#pragma unroll
            for (int ll = 0; ll < LW; ++ll) {
                const bool ok = __shfl_sync(0xffffffffu, (int)row_ok, ll * TPL) != 0;
                const long long so = __shfl_sync(0xffffffffu, s_off, ll * TPL);
                const long long ko = __shfl_sync(0xffffffffu, k_off, ll * TPL);
                const int kc = __shfl_sync(0xffffffffu, k_cnt, ll * TPL);
                if (!ok) continue;
                const cf* src = a.sens + so + c * s_stride;
                for (int i = lane; i < N / 2; i += 32) cp_async16(sS + buf * TILE + ll * N + 2 * i, src + 2 * i);
                if (use_z && kc <= KCAP) {
                    const cf* ks = a.z + ko + c * k_stride;
                    for (int i = lane; i < (kc + 1) / 2; i += 32) cp_async16(sK + buf * KTILE + ll * KSTRIDE + 2 * i, ks + 2 * i);
                }
            }
        };

        __syncwarp();   // previous group's shared-memory reads are complete
#pragma unroll
        for (int ll = 0; ll < LW; ++ll) {
            const bool ok = __shfl_sync(0xffffffffu, (int)row_ok, ll * TPL) != 0;
            const long long xo = __shfl_sync(0xffffffffu, x_off, ll * TPL);
            const long long bto = __shfl_sync(0xffffffffu, (long long)bt, ll * TPL);
            if (!ok) continue;
            if (!ADJ) {
                if (!a.x_planar) {
                    for (int i = lane; i < N / 2; i += 32) cp_async16(sX + ll * N + 2 * i, a.x + xo + 2 * i);
                } else {
                    // two-channel layout: the line's real parts and its imaginary parts are two contiguous runs
                    const long long bo = __shfl_sync(0xffffffffu, (long long)b, ll * TPL);
                    const float* xf = reinterpret_cast<const float*>(a.x) + xo + bo * a.plane;
                    float* dst = reinterpret_cast<float*>(sX + ll * N);
                    if (N % 4 == 0) {       // staged as two planes of N floats (16-byte copies), read as pairs below
                        for (int i = lane; i < N / 4; i += 32) { cp_async16(dst + 4 * i, xf + 4 * i); cp_async16(dst + N + 4 * i, xf + a.plane + 4 * i); }
                    } else {
                        for (int i = lane; i < N; i += 32) { dst[2 * i] = xf[i]; dst[2 * i + 1] = xf[a.plane + i]; }
                    }
                }
            }
            {
                // scaled mask^2 in raw k order and, with z, the masks of the units
                if (use_z) {
                    const int cnt = line_units<P::BFL, RL>(a.mask + bto * N, true, lane, sU + ll * P::BFL, ADJ ? nullptr : sM + ll * N);
                    if (l == ll) k_cnt = cnt;
                } else {
#pragma unroll
                    for (int k0 = 0; k0 < N; k0 += 32) {       // a trip count known at compile time: all loads in flight
                        const int k = k0 + lane;
                        const float mv = (k < N) ? a.mask[bto * N + shift_half(k, N)] : 0.f;
                        if (k < N) sM[ll * N + k] = mv * mv * (1.0f / N);
                    }
                }
            }
        }
        issue_coil(0, 0);
        cp_async_commit();

        cf acc[R0];
#pragma unroll
        for (int m = 0; m < R0; ++m)
            acc[m] = (a0 && row_ok) ? coil_sum_start(a.aty, x_off + j + P::BF0 * m) : make_float2(0.f, 0.f);

        for (int c = 0; c < a.C; ++c) {
            const int buf = c & 1;
            if (c + 1 < a.C) issue_coil(c + 1, buf ^ 1);
            cp_async_commit();
            cp_async_wait<1>();          // everything but the newest group (coil c+1) has landed
            __syncwarp();

            const cf* cS = sS + buf * TILE + l * N;
            const cf* cK = sK + buf * KTILE + l * KSTRIDE;
            const cf* gK = use_z ? a.z + k_off + c * k_stride : nullptr;   // this line's compact z row
            const cf* cX = sX + l * N;
            const bool x_planes = a.x_planar && (N % 4 == 0);       // x staged as two planes of floats
            auto x_at = [&](int idx) -> cf {
                if (!x_planes) return cX[idx];
                const float* xf = reinterpret_cast<const float*>(cX);
                return make_float2(xf[idx], xf[N + idx]);
            };
            cf v[R0], u[RL];
            if (ADJ) {
#pragma unroll
                for (int k = 0; k < RL; ++k) u[k] = make_float2(0.f, 0.f);
            } else {
                if (a0) {
#pragma unroll
                    for (int m = 0; m < R0; ++m) v[m] = cmul(cS[j + P::BF0 * m], x_at(j + P::BF0 * m));
                    Dft<R0, -1, !HAS_Z>::run(v);
                }
                if (P::S == 2) {
                    if (a0) {
#pragma unroll
                        for (int k = 0; k < R0; ++k)
                            sE[l * WL::EXL + k * P::LS1 + j] = (k == 0) ? v[0] : cmul(v[k], tw0[k]);
                    }
                    __syncwarp();
                    if (aL) {
#pragma unroll
                        for (int m = 0; m < RL; ++m) u[m] = sE[l * WL::EXL + j * P::LS1 + m];
                        Dft<RL, -1, !HAS_Z>::run(u);
                    }
                    __syncwarp();
                } else {
#pragma unroll
                    for (int k = 0; k < RL; ++k) u[k] = v[k % R0];
                }
            }
            {
                if (aL) {
                    const float* mm = sM + l * N + j;
                    if (!use_z) {
#pragma unroll
                        for (int k = 0; k < RL; ++k) u[k] = cscale(u[k], mm[P::BFL * k]);
                    } else {       // staged z, or straight from the line's row (lanes without a row hold no mask)
                        const UnitMask um = row_ok ? sU[l * P::BFL + j] : UnitMask{0u, 0};
                        if (k_cnt <= KCAP) unit_update<P::BFL, RL, ADJ>(u, um.bits, mm, cK + um.first, true);
                        else unit_update<P::BFL, RL, ADJ>(u, um.bits, mm, gK + um.first, false);
                    }
                }
            }
            {
                if (P::S == 2) {
                    if (aL) {
                        Dft<RL, +1, !HAS_Z>::run(u);
#pragma unroll
                        for (int m = 0; m < RL; ++m) sE[l * WL::EXL + j * P::LS1 + m] = u[m];
                    }
                    __syncwarp();
                    if (a0) {
#pragma unroll
                        for (int k = 0; k < R0; ++k) {
                            const cf r = sE[l * WL::EXL + k * P::LS1 + j];
                            v[k] = (k == 0) ? r : cmulc(r, tw0[k]);
                        }
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < R0; ++k) v[k] = u[k % RL];
                }
                if (a0) {
                    Dft<R0, +1, !HAS_Z>::run(v);
#pragma unroll
                    for (int m = 0; m < R0; ++m) {
                        const cf sv = cS[j + P::BF0 * m];
                        acc[m].x = fmaf(sv.x, v[m].x, fmaf(sv.y, v[m].y, acc[m].x));
                        acc[m].y = fmaf(sv.x, v[m].y, fmaf(-sv.y, v[m].x, acc[m].y));
                    }
                }
            }
            __syncwarp();   // all lanes are done with buffer `buf` and the exchange area
        }
        cp_async_wait<0>();
        {
            double dsum = 0.0, nsum = 0.0;       // Re<x, out>, <out, out> over this lane's elements (for the caller's inner products)
            if (a0 && row_ok) {
#pragma unroll
                for (int m = 0; m < R0; ++m) {
                    const int idx = j + P::BF0 * m;
                    const float* xf = reinterpret_cast<const float*>(sX + l * N);
                    const cf xv = ADJ ? make_float2(0.f, 0.f) : (a.x_planar && (N % 4 == 0)) ? make_float2(xf[idx], xf[N + idx]) : sX[l * N + idx];
                    const cf av = acc[m];
                    const cf ov = make_float2(fmaf(-a.eta, av.x, xv.x), fmaf(-a.eta, av.y, xv.y));
                    store_image(a.out, x_off + j + P::BF0 * m, ov, a.out_planar, b, a.plane);
                    if (a.dot_rows != nullptr) { dsum += (double)xv.x * ov.x + (double)xv.y * ov.y; nsum += (double)ov.x * ov.x + (double)ov.y * ov.y; }
                }
            }
            if (a.dot_rows != nullptr) {     // the same in every thread
                for (int o = TPL / 2; o > 0; o >>= 1) {
                    dsum += __shfl_down_sync(0xffffffffu, dsum, o, TPL);
                    nsum += __shfl_down_sync(0xffffffffu, nsum, o, TPL);
                }
                if (j == 0 && row_ok) { a.dot_rows[row] = dsum; a.dot_rows[a.nrows + row] = nsum; }
            }
        }
    }
}

}  // namespace gleam
