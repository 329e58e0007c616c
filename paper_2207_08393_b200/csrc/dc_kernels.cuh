// Kernels of the data-consistency step  out = x - eta * A^H (A x - y),  A = Omega F S  (Eq. 3 of
// the GLEAM paper with eta = 2t; sensing model Eq. 1) and of its vector-Jacobian product.
//
// All transforms inside the kernels are raw DFTs.  Centring and orthonormal scaling of F are moved
// into the k-space tables: with the shift sh(k) = (k + N/2) mod N per transformed axis,
//     A^H A   = S^H  Fraw^H  diag( M[sh(k)]^2 / N )  Fraw  S
//     A^H y   = S^H  Fraw^H  ( g (-1)^{sh(k)} M[sh(k)] y[sh(k)] / sqrt(N) ),   g = prod (-1)^{N_a/2}
// (even extents only).
//
// Row kernels (dc_warpline.cuh, dc_warpflat.cuh) transform the contiguous axis n2 of 2-D problems and carry
// the image-side work: sensitivity multiply on the way in, conjugate-sensitivity coil sum in registers on the
// way out.  The column kernel here turns y into the table z.
#pragma once
#include "fft_line.cuh"
#include "dc_entry.h"
#include "launch_overlap.cuh"
#include <stdint.h>

namespace gleam {

__device__ __forceinline__ int shift_half(int k, int n) { int h = n >> 1; return k >= n - h ? k - (n - h) : k + h; }


__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async8(void* smem_dst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gsrc) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int NKEEP> __device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(NKEEP) : "memory");
}

struct RowArgs {
    const cf* x;        // image-domain input (B,T,n0,n1,n2); null with z: a zero image (A^H y)
    const cf* sens;     // (B,C,[T],n0,n1,n2)
    cf* out;            // (B,T,n0,n1,n2)
    const float* mask;  // readout-invariant mask (B,T,n2)
    const cf* z;        // compact table of shifted, signed, masked R^H y: (B,C,T,n1,[rank < n2]), unit order; may be null
    float eta;
    int C, T, Ts;       // coils, frames, sens frames (T or 1)
    int RPB;            // rows of an image (n1)
    long long nrows;    // B*T*n1
    double* dot_rows;   // if not null, Re<x, out> of every image row, (B*T*n1), followed by <out, out> of every row
    DotForm* dot_form;  // host: if not null, the launch says how it leaves them
    int dot_blocks;     // set by the launch, if not 0 the number of examples: the sums of a whole block instead of a row, by block
    // Two-real-channel layout (B, 2, T, n0, n1, n2) float32 of the image-side arrays (the form the learned
    // prior takes and returns): real index of complex element e of example b = e + b * plane, the imaginary
    // part `plane` further on (plane = T * n0 * n1 * n2).
    int x_planar, out_planar;
    long long plane;
    // Normal-equations form of the step: when not null (only with z == null), the image A^H y (B,T,n0,n1,n2),
    // complex interleaved; the kernels that write `out` then store x - eta * (sum - aty).
    const cf* aty;
};

// Start value of the coil sum of image element e: minus the given A^H y, if there is one.  Taking it as the
// start value puts its load at the beginning of the coil loop, where its latency costs nothing, and needs no
// register of its own.
__device__ __forceinline__ cf coil_sum_start(const cf* aty, long long e) {
    if (aty == nullptr) return make_float2(0.f, 0.f);
    const cf t = aty[e];
    return make_float2(-t.x, -t.y);
}

// image-side element e (complex-element offset in the (B,T,V) array) of example b, in either layout
__device__ __forceinline__ cf load_image(const cf* x, long long e, int planar, int b, long long plane) {
    if (!planar) return x[e];
    const float* xf = reinterpret_cast<const float*>(x) + e + (long long)b * plane;
    return make_float2(xf[0], xf[plane]);
}
__device__ __forceinline__ void store_image(cf* out, long long e, cf v, int planar, int b, long long plane) {
    if (!planar) { out[e] = v; return; }
    float* of = reinterpret_cast<float*>(out) + e + (long long)b * plane;
    of[0] = v.x; of[plane] = v.y;
}

struct ColArgs {
    const cf* y;        // (B,C,T,V)
    cf* z;              // compact table (unit, n_ro, [rank < pe])
    const int* zlist;   // (B,T,pe): sampled source positions p (unshifted), by rank; null: the blocks rank themselves
    const int* zcount;  // (B,T)
    const float* mask;  // readout-invariant mask
    int es;             // element stride of the transformed axis = phase-encode positions per outer index
    int images;         // B*T
    int C, T, rank, n2;
    int unit_r0;        // rank 2: the ranks follow the units of the row kernel (below)
    int bpi;            // blocks per image: they share its (coil, tile of ranks) pairs
    float scale;        // g_ro g_pe / sqrt(N_ro N_pe)
};

// Rank order of the sampled positions of a 2-D mask row (unit order): the raw k indices k = jb + R0 k1 (k1 < RL) that
// one last-stage butterfly of the row kernel's plan N = R0 RL holds are neighbours, jb outermost.  A butterfly's z values
// are then one contiguous run of the compact row, and what it needs to know of the mask is one word: bit k1 is set where
// k is sampled.  The update reads shared memory at the sampled entries only (it used to read a rank, a weight and a z
// value for every entry: 8 x 16 coils x 640 rows of 320 at 4x, 152 -> 128 us; 256-point rows at 3x, 58 -> 36 us).
struct UnitMask { unsigned bits; int first; };       // that word, and the rank of the run's first entry
// The masks of the R0 units of one line, by one warp: lane jb < R0 reads its RL mask values (and stores their squares,
// scaled, at raw k in `weight` unless it is null).  Returns the number of sampled positions in every lane.
template <int R0, int RL>
__device__ __forceinline__ int line_units(const float* mask_row, bool ok, int lane, UnitMask* units, float* weight) {
    constexpr int N = R0 * RL;
    static_assert(R0 <= 32 && RL <= 32, "one lane per unit, one bit per entry");
    unsigned bits = 0;
    if (lane < R0) {
#pragma unroll
        for (int k1 = 0; k1 < RL; ++k1) {
            const int k = lane + R0 * k1;
            const float m = ok ? mask_row[shift_half(k, N)] : 0.f;
            if (weight != nullptr) weight[k] = m * m * (1.0f / N);
            bits |= (m != 0.f ? 1u : 0u) << k1;
        }
    }
    int incl = __popc(bits);
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += t; }
    if (lane < R0) units[lane] = UnitMask{bits, incl - __popc(bits)};
    return __shfl_sync(0xffffffffu, incl, 31);
}
// k-space update of one unit: u = w u - z at the sampled entries, 0 elsewhere (adjoint: -z).  `weight` points at the
// unit's first entry (stride R0), `z` at its run; both are read at sampled entries only.  `fused`: one rounding for the
// two operations (lines whose z values are few enough to be staged), else one each, whichever kernel the line is in.
template <int R0, int RL, bool ADJ>
__device__ __forceinline__ void unit_update(cf (&u)[RL], unsigned bits, const float* weight, const cf* z, bool fused) {
#pragma unroll
    for (int k = 0; k < RL; ++k) {
        float w = 0.f; cf q = make_float2(0.f, 0.f);
        if (bits & (1u << k)) {
            if (!ADJ) w = weight[R0 * k];
            q = *z++;
        }
        if (ADJ) u[k] = make_float2(-q.x, -q.y);
        else if (fused) u[k] = make_float2(fmaf(w, u[k].x, -q.x), fmaf(w, u[k].y, -q.y));
        else u[k] = make_float2(__fsub_rn(__fmul_rn(w, u[k].x), q.x), __fsub_rn(__fmul_rn(w, u[k].y), q.y));
    }
}
// sampled entries of a line of N points that are staged
constexpr int z_stage(int N) { return ((N + 3) / 4 + 1) / 2 * 2; }

constexpr int COLZ_SELF_MAX = 1024;   // COL_Z ranks a mask row of at most this many positions by itself


// --------------------------------------------------------------------------------------------
// z table: tiles of L sampled phase-encode positions of one unit, inverse transform along the readout axis:
//     z[r] = (g/sqrt(N_ro N_pe)) (-1)^{n_ro} (-1)^{p} M[p] * Rraw^H( (-1)^{k_ro} y[.., p] ),  p = source of rank r
// Gathers 8-byte samples; bound by the DRAM sectors and pages they touch and by the requests in flight.  A block walks over
// tiles of one image; a sample goes straight to the register of the butterfly that takes it, and other blocks fill the time
// a tile waits.  Butterflies of 20 and 23 points leave one to three blocks per SM, so there the next tile is on its way to
// shared memory (8-byte cp.async) while the current one is transformed; elsewhere that costs more than it gives.  Cold L2, us,
// staged -> direct: 256 x 256 x 160 at 7x, 6 coils 108 -> 98, 240 x 320 x 184 182 -> 162, 64 x 240 x 184 45 -> 41, 8 x 16 coils of
// 640 x 320 at 4x 90 -> 80, 4 x 8 coils x 4 of 256 x 256 39 -> 31; but 8 x 16 coils of 320 x 320 43 -> 45, 46 x 184 x 160 31 -> 39,
// 184 x 240 x 184 at 3x 211 -> 242, 368 x 320 x 320 at 3x 287 -> 326.
// Staged, two buffers take turns as "incoming tile" and "current tile"; once every thread holds its elements of the
// current one, its buffer takes the exchange of the transform.
// --------------------------------------------------------------------------------------------
template <class P, int L>
struct ColZ {
    using E = LineFFT<P, L>;
    static constexpr bool STAGED = P::S == 2 && P::RL >= 20;
    static constexpr int BUFSZ = L * (STAGED ? cmax(P::BUF, P::N) : P::BUF);
    static constexpr size_t SMEM_BYTES = sizeof(cf) * (STAGED ? 2 : P::S == 3 ? 2 : 1) * BUFSZ;
    static_assert(E::THREADS % L == 0, "a thread has one line in every stage");
    static_assert(!STAGED || P::S == 2, "the exchange takes the current tile's buffer");
    // Volumes: candidate tiles (of which the sampled ones have work) per block, 0 for one round of blocks that share all
    // tiles.  Blocks are dealt out in order, which keeps the tiles in work next to each other in y; those of a single round
    // drift apart.  Cold L2, one round -> 8 tiles per block: 320 x 320 x 256 at 12x 249 -> 234 us, at 7x 314 -> 295, but at 3.5x,
    // where a DRAM page holds more of a tile, 354 -> 376; 240 x 320 x 184 (direct) 166 -> 154.  23-point plans do not gain
    // (184 x 240 x 184 at 5x 162 -> 174).  Slices rank their mask row in every block and stay with one round.
    static constexpr int TILES = P::RL == 23 ? 0 : 8;
};

template <class P, int L>
__global__ void __launch_bounds__(LineFFT<P, L>::THREADS)
col_z_kernel(const ColArgs a) {
    grid_dependency_wait();
    // The row kernel behind this launch is scheduled when its blocks end.  Scheduled at their start, its single-warp
    // blocks piled up on the SMs with room and stayed there (8 x 16 coils of 128 x 120, forward 48 against 29 us); only
    // next to a handful of blocks the earlier start is the better one (64 x 64, 8 coils: 7.4 against 8.1 us).
    if (gridDim.x <= 64) grid_launch_dependents();
    using E = LineFFT<P, L>;
    constexpr int N = P::N, R0 = P::R0, RL = P::RL, BUFSZ = ColZ<P, L>::BUFSZ;
    constexpr bool STAGED = ColZ<P, L>::STAGED;
    extern __shared__ __align__(16) float2 smem[];
    const int tid = threadIdx.x;
    const int bt = blockIdx.x / a.bpi, t = bt % a.T, b = bt / a.T;
    const long long pe = a.es;
    const float* mk = a.mask + bt * pe;

    // Without a rank map from an earlier launch (a.zlist == null; rank 2 with at most COLZ_SELF_MAX phase-encode
    // positions) the block ranks the sampled positions of its mask row itself: it lists their source positions sh(k) in
    // unit order.
    __shared__ int s_list[COLZ_SELF_MAX];
    __shared__ unsigned s_bal[COLZ_SELF_MAX / 32];
    const bool self_ranks = a.zlist == nullptr;
    int cnt = 0;
    if (self_ranks) {
        const int lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
        const int nchunks = (a.es + 31) / 32, r0 = a.unit_r0, rl = a.es / r0;
        auto source = [&](int q) { return shift_half(q / rl + r0 * (q % rl), a.es); };        // of entry q in unit order
        // every warp marks the sampled entries of its chunks of 32 ...
        for (int c = warp; c < nchunks; c += nwarps) {
            const int q = c * 32 + lane;
            const bool on = (q < a.es) && (mk[source(q)] != 0.f);
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            if (lane == 0) s_bal[c] = bal;
        }
        __syncthreads();
        // ... then numbers them behind the entries of the chunks before
        for (int c = warp; c < nchunks; c += nwarps) {
            int before = 0;
            for (int e = 0; e < c; ++e) before += __popc(s_bal[e]);
            const unsigned bal = s_bal[c];
            const int q = c * 32 + lane;
            if ((bal >> lane) & 1u) s_list[before + __popc(bal & ((1u << lane) - 1u))] = source(q);
        }
        for (int e = 0; e < nchunks; ++e) cnt += __popc(s_bal[e]);
        __syncthreads();
    } else {
        cnt = a.zcount[bt];
    }
    const int ntiles = (cnt + L - 1) / L, items = a.C * ntiles;
    auto source_of = [&](int i) { return self_ranks ? s_list[i] : a.zlist[bt * pe + i]; };
    auto unit_of = [&](int item) { return ((long long)b * a.C + item / ntiles) * a.T + t; };
    const int l = tid % L;                             // every stage sees the same line
    auto issue = [&](int item, cf* dst) {
        const int i = (item % ntiles) * L + l;
        if (i < cnt) {
            const cf* src = a.y + (unit_of(item) * N + tid / L) * pe + source_of(i);
            for (int n = tid / L; n < N; n += E::THREADS / L) { cp_async8(dst + n * L + l, src); src += (E::THREADS / L) * pe; }
        }
        cp_async_commit();
    };

    int item = blockIdx.x % a.bpi;
    if (item >= items) return;
    const typename E::Ids d = E::ids(tid);
    typename E::Tw tw;
    E::make_tw(d, tw);
    if (STAGED) issue(item, smem);
    for (int it = 0; item < items; item += a.bpi, ++it) {
        cf* cur = smem + (STAGED ? (it % 2) * BUFSZ : 0);
        if (STAGED) {
            cp_async_wait<0>();
            __syncthreads();           // the tile is visible to all; every thread has left the one before
            if (item + a.bpi < items) issue(item + a.bpi, smem + ((it + 1) % 2) * BUFSZ);
        }
        const int i = (item % ntiles) * L + l;
        const bool ok = i < cnt;
        int p = 0, psign = 0; float mv = 0.f;
        if (ok) {
            p = source_of(i);
            mv = mk[p];
            psign = (a.rank == 2) ? (p & 1) : ((p / a.n2 + p % a.n2) & 1);
        }
        cf v[R0], u[RL];
        if (d.aL) {
            const float odd = (d.jL & 1) ? -1.f : 1.f;
            const cf* src = a.y + (unit_of(item) * N + d.jL) * pe + p;
#pragma unroll
            for (int k = 0; k < RL; ++k) {
                const cf yv = !ok ? make_float2(0.f, 0.f) : STAGED ? cur[(d.jL + P::BFL * k) * L + l] : *src;
                u[k] = cscale(yv, (P::BFL * k) % 2 ? -odd : odd);
                src += P::BFL * pe;
            }
        }
        if (P::S == 2) __syncthreads();        // the exchange buffer is free
        E::inverse(u, v, tw, d, smem + BUFSZ, cur);
        if (d.a0 && ok) {
            const float f = ((psign + d.j0) & 1) ? -a.scale * mv : a.scale * mv;
            cf* dst = a.z + (unit_of(item) * N + d.j0) * pe + i;
#pragma unroll
            for (int m = 0; m < R0; ++m) { *dst = cscale(v[m], (P::BF0 * m) % 2 ? -f : f); dst += P::BF0 * pe; }
        }
    }
}

}  // namespace gleam
