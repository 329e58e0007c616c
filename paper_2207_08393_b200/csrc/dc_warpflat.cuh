// One-pass row kernel of 2-D problems (arithmetic of dc_warpline.cuh) for two-stage plans N = R0 * RL.  In the plain
// warp-resident form the RL-point butterflies of the last forward stage, the k-space update and the first inverse
// stage keep only R0 of every max(R0, RL) lanes busy (10 of 16 for N = 160 = 10 x 16, 8 of 32 for 184 = 8 x 23).
//
// Here a warp still owns LW = 32 / RL whole lines, and the first / last image-side stages (S x, R0-point
// butterflies, twiddles; conj(S) coil sum) keep their fixed lane = (line, butterfly) assignment, so the
// coil sum stays in registers.  The k-space stages are stateless, so their work units (one RL-point
// butterfly pair with the mask update in between) are numbered across the coils,
//     unit u = coil * UPC + line * R0 + k,       UPC = LW * R0 units per coil,
// and taken 32 at a time, one per lane: every lane is busy whatever R0 is (N = 160, 8 coils: 5 rounds
// of 32 units instead of 8 rounds of 20).  The stage hand-over goes through a small ring of coil slots in
// shared memory: forward image-side stages run ahead just far enough to fill the next round, the
// inverse image-side stage of a coil runs once all its units are through.  The sensitivities are read
// from global memory straight into registers (a round ahead for the forward stage, at the start of the
// stage for the inverse one), which frees the shared memory the ring needs.
#pragma once
#include "dc_warpline.cuh"

namespace gleam {


enum FlatForm {
    FLAT_SINGLE = 0,     // one warp per block, blocks stride over the line groups
    FLAT_SM = 1,         // one block of many warps per SM, a single round
    FLAT_TAIL = 2        // blocks of four warps that stride over the groups; a block's warps share each group of the last, partial round
};

template <class P, bool HAS_Z, bool SMW = false>
struct WarpFlat {
    static constexpr int N = P::N, R0 = P::R0, RL = P::RL;
    static constexpr bool ELIGIBLE = (P::S == 2) && RL >= 2 && RL <= 32 && (N % 2 == 0);
    static constexpr int LW = 32 / RL;                     // lines per warp
    static constexpr int UPC = LW * R0;                    // k-space units per coil
    static constexpr int LANES = LW * RL;                  // lanes of the image-side stages (32 if RL is a power of two)
    static constexpr int USTRIDE = odd_up(RL);             // odd: a round's 32 units read without bank conflicts
    static constexpr int SLOTS_MIN = (32 + UPC - 1) / UPC + 1;     // coils between first forward and inverse stage
    // Where the z values of a unit wait for its butterfly: in the unit's own slots of the ring, which it has just read (RING_Z),
    // or in a staging area per coil, requested a forward stage earlier.  The first takes any number of samples, leaves the
    // staging area's shared memory to further blocks and makes the update free of branches, but the butterfly alone has to
    // cover the latency: not where so large ones leave 8 warps per SM or fewer.  Prepared step, staged -> ring: 8 x 16 coils
    // of 640 x 320 at 4x 137 -> 112 us, at 2.9x 138 -> 118, 8 x 8 of 512 x 256 52 -> 46, 2 x 12 of 384 x 320 26.1 -> 20.9, 20
    // frames x 8 of 192 x 160 21.9 -> 20.8; but 4 x 15 of 640 x 368 92 -> 98, 8 of 640 x 640 24 -> 26.5.
    static constexpr bool RING_Z = !(RL > 16 && R0 >= 16);
    // a ring whose unit count is a multiple of 16 keeps the bank pattern across the wrap; taken when small
    static constexpr int slots_aligned() {
        for (int s = SLOTS_MIN; s <= SLOTS_MIN + 3; ++s) if ((s * UPC) % 16 == 0) return s;
        return SLOTS_MIN;
    }
    static constexpr int SLOTS = (!SMW && (!HAS_Z || RING_Z) && slots_aligned() * UPC * USTRIDE * 8 <= 11 * 1024) ? slots_aligned() : SLOTS_MIN;
    static constexpr int ZS = RING_Z ? 0 : SLOTS + 1;      // staged: one forward stage ahead
    static_assert(!SMW || RING_Z, "blocks of many warps stage no z");
    static constexpr int KCAP = z_stage(N); // staged z entries per line (more: read from global memory)
    static constexpr int KSTRIDE = KCAP;
    static constexpr int KTILE = LW * KSTRIDE;
    static constexpr int MS = N + ((LW > 1 && N % 32 == 0) ? 16 : 0);   // mask row stride (floats): lines on different banks
    // shared memory of the warp, in float2 units
    static constexpr int OFF_X = 0, OFF_E = LW * N, OFF_M2 = OFF_E + SLOTS * UPC * USTRIDE + (SLOTS * UPC * USTRIDE) % 2;
    // mask weights of every raw k; with z: the units' masks, and the staged z rows
    static constexpr int OFF_U = OFF_M2 + (LW * MS + 3) / 4 * 2;
    static constexpr int OFF_K = OFF_U + (HAS_Z ? (LW * R0 + 1) / 2 * 2 : 0);
    static constexpr int OFF_CNT = OFF_K + (HAS_Z ? ZS * KTILE : 0);
    // per line: element offset of its z row (64-bit), sampled count
    static constexpr int ELEMS = (OFF_CNT + 2 * LW + 1) / 2 * 2;
    static constexpr size_t WARP_BYTES = sizeof(cf) * ELEMS;      // per warp of the block
    // Registers: coil sum, twiddles and the sensitivities of the next forward stage are held throughout (2 R0 each),
    // next to a butterfly of the image side or of the k-space round (a prime radix also holds its sums and differences).
    static constexpr bool PRIME = RL > 4 && RL % 2 == 1 && smallest_odd_factor(RL) == RL;
    static constexpr int REGS = cmax(8 * R0 + 24, 6 * R0 + (PRIME ? 4 : 2) * RL + 24);
    static constexpr int SINGLE_BLOCKS = cmax(4, cmin(RL == 32 ? 12 : 16, 65536 / (32 * ((REGS + 7) / 8 * 8)) / 4 * 4));
};

// SMW = false: one warp per block, blocks stride over the line groups.
// SMW = true (one round, one block per SM, the host sizes the grid): a block of nwhole + 4 nsplit warps.
// A warp's run time grows with the number of warps on its scheduler (the schedulers favour the oldest warp, and
// the last one to finish sets the time), so 4 k + 1 single-warp blocks per SM leave one scheduler with k + 1
// warps and the others waiting for it.  Here the first nwhole warps of the block take one group each, and every
// further set of four warps (one per scheduler) shares ONE more group, a quarter of the coils each; the partial
// coil sums are added in warp order through shared memory.  A quarter of the extra work lands on every scheduler.
// One block per SM also keeps a dependent launch from moving in next to the running one warp by warp, which
// would fill the schedulers unevenly.
// FLAT_TAIL (several rounds, the last one nearly empty): blocks of four warps, each with groups of its own in the full rounds;
// then a block's warps share one group after another as above.  The rule and its measurements: launch_warpflat_zy.
// HAS_ATY: the coil sum is kept as aty - sum, starting from the given A^H y image as loaded (no instruction depends on
// the load before the first inverse stage, so its latency is hidden even when a warp has a single group; the coil
// terms are subtracted and the update adds eta times the result: the same bits as sum - aty, since rounding is
// symmetric in the sign).  Normal-equations form of the step; never together
// with z).  A template parameter, not a run-time test of a.aty: with the test in the code the plain call measured
// 11 % slower (17.7 against 16.0 us), although it never takes that branch.
// ADJ (with z): A^H y, the image is zero; the forward stages are left out and a unit starts from minus its z values.
// Registers: sixteen warps of one block have 128 each, which the step with z of 160 points exceeds by 20 B (spilled to
// local memory; single-warp blocks without the spill are slower all the same, see launch_warpflat_zy).
// DOT: the inner products of dot_rows (conjugate gradients; calls without z and A^H y).  A template parameter for the same
// reason as HAS_ATY: with the block sums behind a run-time test the plain call of 20 frames of 192 x 160 took 17.3 us, not 16.4.
template <class P, bool HAS_Z, int FORM, bool HAS_ATY, bool ADJ, bool DOT>
__global__ void __launch_bounds__(FORM == FLAT_SM ? 512 : FORM == FLAT_TAIL ? 128 : 32,
                                  FORM == FLAT_SM ? 1 : WarpFlat<P, HAS_Z, FORM == FLAT_SM>::SINGLE_BLOCKS / (FORM == FLAT_TAIL ? 4 : 1))
warpflat_kernel(const RowArgs a, const int nwhole) {
    grid_dependency_wait();
    constexpr bool SMW = FORM == FLAT_SM, TAIL = FORM == FLAT_TAIL;
    using WF = WarpFlat<P, HAS_Z, SMW>;
    constexpr int N = P::N, R0 = P::R0, RL = P::RL, LW = WF::LW, UPC = WF::UPC, US = WF::USTRIDE, SLOTS = WF::SLOTS;
    // Folded twiddles: plain and normal-equations calls 87 -> 85 and 88 -> 86 us (8 x 16 coils of 640 x 320), 30 -> 28 (8 x 8
    // of 512 x 256); the block of many warps without A^H y measured slower with them (20 frames of 192 x 160, 16.4 -> 16.8),
    // and so did the 23-point image side (4 x 15 of 640 x 368, 78.7 -> 79.0 and 80.1 -> 80.9).
    constexpr bool FOLD = !HAS_Z && (!SMW || HAS_ATY) && R0 != 23;
    constexpr int KCAP = WF::KCAP, KSTRIDE = WF::KSTRIDE, KTILE = WF::KTILE, ZS = WF::ZS, MS = WF::MS;
    extern __shared__ __align__(16) float2 smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cf* wsm = smem + warp * WF::ELEMS;
    cf* sX = wsm + WF::OFF_X;
    cf* sE = wsm + WF::OFF_E;
    float* sM = reinterpret_cast<float*>(wsm + WF::OFF_M2);
    UnitMask* sU = reinterpret_cast<UnitMask*>(wsm + WF::OFF_U);
    cf* sK = wsm + WF::OFF_K;
    long long* sKo = reinterpret_cast<long long*>(wsm + WF::OFF_CNT);      // per line: offset of the z row of coil cbase
    int* sC = reinterpret_cast<int*>(wsm + WF::OFF_CNT + LW);              // per line: sampled entries (none in a line past the end)
    bool split = SMW && warp >= nwhole;                            // one of four warps that share a group
    const int set = split ? (warp - nwhole) >> 2 : 0;
    int q = split ? (warp - nwhole) & 3 : 0;
    int cbase = split ? q * a.C / 4 : 0;                           // first coil and number of coils of this warp
    int nc = split ? (q + 1) * a.C / 4 - cbase : a.C;

    const bool img = WF::LANES == 32 || lane < WF::LANES;
    const int l = img ? lane / RL : LW - 1, j = img ? lane % RL : 0;      // image-side identity: line of the warp, butterfly

    // inter-stage twiddles exp(-2 pi i j k / N) of this lane (fetching them again before the image-side stages of
    // every round, to free registers for the k-space round, was measured slower: 18.7 against 16.4 us per call)
    cf tw0[R0];
#pragma unroll
    for (int k = 0; k < R0; ++k) tw0[k] = unit_root_fwd<N>((j * k) % N);
    const long long ngroups = (a.nrows + LW - 1) / LW;
    // A single round: the next launch may come in.  Not behind single-warp blocks with z: they leave room for the next launch's
    // blocks on some SMs only, and the launches behind it in a chain keep that uneven split (enqueued calls, let in -> not: A^H y
    // and 6 steps of 3 x 9 coils of 384 x 256 136 -> 103 us, 5 prepared steps and VJPs of 2 x 16 of 512 x 384 378 -> 325, of 3 x 12
    // of 384 x 320 252 -> 218; equal elsewhere).
    if (SMW || (!TAIL && !HAS_Z && (long long)gridDim.x >= ngroups)) grid_launch_dependents();
    int total = UPC * nc, rounds = (total + 31) / 32;
    const long long g_first = TAIL ? 4LL * blockIdx.x + warp : !SMW ? (long long)blockIdx.x
                            : split ? (long long)(nwhole + set) * gridDim.x + blockIdx.x : (long long)warp * gridDim.x + blockIdx.x;
    long long g_step = SMW ? ngroups : TAIL ? 4LL * gridDim.x : (long long)gridDim.x;      // SMW: a single round
    const long long g_whole = TAIL ? ngroups / g_step * g_step : ngroups;        // TAIL: groups of the full rounds
    if (SMW && DOT && a.dot_blocks && g_first >= ngroups && lane < 3) reinterpret_cast<double*>(sX)[lane] = 0.0;

    for (long long g = g_first; g < ngroups || (TAIL && !split); g += g_step) {
        if (TAIL && !split && g >= g_whole) {            // from here on the block's four warps share a group
            split = true;
            q = warp; cbase = q * a.C / 4; nc = (q + 1) * a.C / 4 - cbase;
            total = UPC * nc; rounds = (total + 31) / 32;
            g = g_whole + blockIdx.x; g_step = gridDim.x;
            if (g >= ngroups) break;
        }
        const long long row = g * LW + l;
        const bool row_ok = img && row < a.nrows;
        const unsigned rowu = row_ok ? (unsigned)row : 0u;       // host side guarantees nrows < 2^31
        const unsigned bt = rowu / (unsigned)a.RPB;
        const int ri = (int)(rowu - bt * (unsigned)a.RPB);
        const int b = (int)(bt / (unsigned)a.T), t = (int)(bt - (unsigned)b * (unsigned)a.T);
        const long long x_off = ((long long)bt * a.RPB + ri) * N;
        // coil indices below are relative to cbase
        const long long s_off = (((long long)(b * a.C + cbase) * a.Ts + (a.Ts > 1 ? t : 0)) * a.RPB + ri) * N;
        const long long k_off = (((long long)(b * a.C + cbase) * a.T + t) * a.RPB + ri) * N;
        const long long s_stride = (long long)a.Ts * a.RPB * N;
        const long long k_stride = (long long)a.T * a.RPB * N;
        const cf* sp = a.sens + s_off + j;                       // this lane's sensitivities of coil 0

        __syncwarp();   // the previous group's shared-memory reads are complete
        // ---- x rows, scaled mask^2 in raw k order and (with z) the rank of every sampled k ----
#pragma unroll
        for (int ll = 0; ll < LW; ++ll) {
            const bool ok = __shfl_sync(0xffffffffu, (int)row_ok, ll * RL) != 0;
            const long long xo = __shfl_sync(0xffffffffu, x_off, ll * RL);
            const long long bto = __shfl_sync(0xffffffffu, (long long)bt, ll * RL);
            if (!ok) {                                               // no z is read for a line past the end
                if (HAS_Z && lane == 0) sC[ll] = 0;
                if (HAS_Z && lane < R0) sU[ll * R0 + lane] = UnitMask{0u, 0};
                continue;
            }
            if (ADJ) {
            } else if (!a.x_planar) {
                for (int i = lane; i < N / 2; i += 32) cp_async16(sX + ll * N + 2 * i, a.x + xo + 2 * i);
            } else {
                const long long bo = __shfl_sync(0xffffffffu, (long long)b, ll * RL);
                const float* xf = reinterpret_cast<const float*>(a.x) + xo + bo * a.plane;
                float* dst = reinterpret_cast<float*>(sX + ll * N);
                if (N % 4 == 0) {       // staged as two planes of N floats (16-byte copies), read as pairs below
                    for (int i = lane; i < N / 4; i += 32) { cp_async16(dst + 4 * i, xf + 4 * i); cp_async16(dst + N + 4 * i, xf + a.plane + 4 * i); }
                } else {
                    for (int i = lane; i < N; i += 32) { dst[2 * i] = xf[i]; dst[2 * i + 1] = xf[a.plane + i]; }
                }
            }
            if (HAS_Z) {
                const int cnt = line_units<R0, RL>(a.mask + bto * N, true, lane, sU + ll * R0, ADJ ? nullptr : sM + ll * MS);
                if (lane == 0) sC[ll] = cnt;
                if (img && lane == ll * RL) sKo[ll] = k_off;
            } else {
#pragma unroll
                for (int k0 = 0; k0 < N; k0 += 32) {       // a trip count known at compile time: all loads in flight
                    const int k = k0 + lane;
                    const float mv = (k < N) ? a.mask[bto * N + shift_half(k, N)] : 0.f;
                    if (k < N) sM[ll * MS + k] = mv * mv * (1.0f / N);
                }
            }
        }
        __syncwarp();
        // z row of coil c for every line of the warp -> slot c % ZS
        auto issue_z = [&](int c) {
#pragma unroll
            for (int ll = 0; ll < LW; ++ll) {
                const long long ko = sKo[ll];
                const int kc = sC[ll];
                if (kc > KCAP) continue;
                const cf* ks = a.z + ko + c * k_stride;
                for (int i = lane; i < (kc + 1) / 2; i += 32) cp_async16(sK + (c % ZS) * KTILE + ll * KSTRIDE + 2 * i, ks + 2 * i);
            }
        };
        constexpr bool STAGED_Z = HAS_Z && !WF::RING_Z;
        if (STAGED_Z) issue_z(0);
        cp_async_commit();

        const bool x_planes = a.x_planar && (N % 4 == 0);          // x staged as two planes of floats
        const cf* cX = sX + l * N;
        auto x_at = [&](int idx) -> cf {
            if (!x_planes) return cX[idx];
            const float* xf = reinterpret_cast<const float*>(cX);
            return make_float2(xf[idx], xf[N + idx]);
        };
        auto load_sens = [&](cf (&dst)[R0], int c) {
            const cf* p = sp + c * s_stride;
#pragma unroll
            for (int m = 0; m < R0; ++m) dst[m] = row_ok ? p[RL * m] : make_float2(0.f, 0.f);
        };

        cf acc[R0];
#pragma unroll
        for (int m = 0; m < R0; ++m) acc[m] = (HAS_ATY && row_ok && q == 0) ? a.aty[x_off + j + RL * m] : make_float2(0.f, 0.f);
        cf sf[R0];                       // sensitivities of the next forward image-side stage
        if (!ADJ && nc > 0) load_sens(sf, 0);
        int af = 0, ai = 0;              // next coil of the forward / of the inverse image-side stage

        for (int br = 0; br < rounds; ++br) {
            const int upto = min(32 * (br + 1), total);
            const int need = (upto + UPC - 1) / UPC;                     // coils this round draws units from
            const int done = (br == rounds - 1) ? nc : upto / UPC;       // coils complete after this round
            // ---- forward image-side stage: S x, R0-point butterflies, twiddles, into the ring ----
            while (af < need) {
                if (STAGED_Z) { if (af + 1 < nc) issue_z(af + 1); cp_async_commit(); }
                if (af == 0) { cp_async_wait<STAGED_Z ? 1 : 0>(); __syncwarp(); }      // x (and z of coil 0) have landed
                if (ADJ) { ++af; continue; }
                cf v[R0];
#pragma unroll
                for (int m = 0; m < R0; ++m) v[m] = cmul(sf[m], x_at(j + RL * m));
                if (af + 1 < nc) load_sens(sf, af + 1);
                Dft<R0, -1, FOLD>::run(v);
                cf* e = sE + ((af % SLOTS) * UPC + l * R0) * US + j;
                if (img) {
#pragma unroll
                    for (int k = 0; k < R0; ++k) e[k * US] = (k == 0) ? v[0] : cmul(v[k], tw0[k]);
                }
                ++af;
            }
            if (STAGED_Z) cp_async_wait<1>();    // everything but a request for the next coil's z is there
            __syncwarp();
            // ---- k-space round: units 32 br .. 32 br + 31, one per lane ----
            {
                const int u0 = 32 * br + lane;
                const bool live = u0 < total;
                const int uu = live ? u0 : total - 1;
                const int c = uu / UPC, w = uu - c * UPC;
                const int bl = w / R0, jb = w - bl * R0;
                cf* e = sE + ((c % SLOTS) * UPC + w) * US;
                cf u[RL];
                if (!ADJ) {
#pragma unroll
                    for (int m = 0; m < RL; ++m) u[m] = e[m];
                }
                if (HAS_Z && WF::RING_Z) {
                    // every entry at its place, zero where nothing was sampled; a lane reads back only what it requested
                    const UnitMask um = sU[bl * R0 + jb];
                    if (live) {
                        const cf* zs = a.z + sKo[bl] + c * k_stride + um.first;
#pragma unroll
                        for (int k = 0; k < RL; ++k) if (!(um.bits & (1u << k))) e[k] = make_float2(0.f, 0.f);
                        for (unsigned left = um.bits; left != 0; left &= left - 1) cp_async8(e + (__ffs((int)left) - 1), zs++);
                    }
                    cp_async_commit();
                }
                if (!ADJ) Dft<RL, -1, FOLD>::run(u);
                if (!HAS_Z) {
                    const float* mm = sM + bl * MS + jb;
#pragma unroll
                    for (int k = 0; k < RL; ++k) u[k] = cscale(u[k], mm[R0 * k]);
                } else if (WF::RING_Z) {
                    cp_async_wait<0>();
                    const float* mw = sM + bl * MS + jb;
                    const bool few = sC[bl] <= KCAP;         // one rounding or two, as in the other kernels
                    if (ADJ) {
#pragma unroll
                        for (int k = 0; k < RL; ++k) { const cf q = e[k]; u[k] = make_float2(-q.x, -q.y); }
                    } else if (__all_sync(0xffffffffu, few)) {
#pragma unroll
                        for (int k = 0; k < RL; ++k) { const cf q = e[k]; const float w = mw[R0 * k]; u[k] = make_float2(fmaf(w, u[k].x, -q.x), fmaf(w, u[k].y, -q.y)); }
                    } else {
#pragma unroll
                        for (int k = 0; k < RL; ++k) {
                            const cf q = e[k];
                            const float w = mw[R0 * k];
                            const cf one = make_float2(fmaf(w, u[k].x, -q.x), fmaf(w, u[k].y, -q.y));
                            const cf two = make_float2(__fsub_rn(__fmul_rn(w, u[k].x), q.x), __fsub_rn(__fmul_rn(w, u[k].y), q.y));
                            u[k] = few ? one : two;
                        }
                    }
                } else {
                    // z of a line that is staged from shared memory, of others straight from its row
                    const UnitMask um = sU[bl * R0 + jb];
                    const int kc = sC[bl];
                    const float* mw = sM + bl * MS + jb;
                    if (kc <= KCAP) unit_update<R0, RL, ADJ>(u, um.bits, mw, sK + (c % ZS) * KTILE + bl * KSTRIDE + um.first, true);
                    else unit_update<R0, RL, ADJ>(u, um.bits, mw, a.z + sKo[bl] + c * k_stride + um.first, false);
                }
                Dft<RL, +1, FOLD>::run(u);
                if (live) {
#pragma unroll
                    for (int m = 0; m < RL; ++m) e[m] = u[m];
                }
            }
            __syncwarp();
            // ---- inverse image-side stage of the coils that are complete: twiddles, R0-point butterflies, conj(S) sum ----
            while (ai < done) {
                cf si[R0];
                load_sens(si, ai);
                const cf* e = sE + ((ai % SLOTS) * UPC + l * R0) * US + j;
                cf v[R0];
#pragma unroll
                for (int k = 0; k < R0; ++k) {
                    const cf r = e[k * US];
                    v[k] = (k == 0) ? r : cmulc(r, tw0[k]);
                }
                Dft<R0, +1, FOLD>::run(v);
#pragma unroll
                for (int m = 0; m < R0; ++m) {
                    if (HAS_ATY) {      // acc = aty - sum
                        acc[m].x = fmaf(-si[m].x, v[m].x, fmaf(-si[m].y, v[m].y, acc[m].x));
                        acc[m].y = fmaf(-si[m].x, v[m].y, fmaf(si[m].y, v[m].x, acc[m].y));
                    } else {
                        acc[m].x = fmaf(si[m].x, v[m].x, fmaf(si[m].y, v[m].y, acc[m].x));
                        acc[m].y = fmaf(si[m].x, v[m].y, fmaf(-si[m].y, v[m].x, acc[m].y));
                    }
                }
                ++ai;
            }
        }
        cp_async_wait<0>();
        __syncwarp();
        if ((SMW || TAIL) && split) {
            // partial coil sums of the other three warps are added by the first in warp order (the ring is free by now); all four
            // warps of the group get here
            if (q > 0) {
#pragma unroll
                for (int m = 0; m < R0; ++m) sE[m * 32 + lane] = acc[m];
            }
            if (TAIL) __syncthreads();
            else if (set == 0) asm volatile("bar.sync 1, 128;" ::: "memory");
            else asm volatile("bar.sync 2, 128;" ::: "memory");
            if (q == 0) {
                for (int w = 1; w < 4; ++w) {
                    const cf* o = smem + ((TAIL ? 0 : nwhole + 4 * set) + w) * WF::ELEMS + WF::OFF_E;
#pragma unroll
                    for (int m = 0; m < R0; ++m) acc[m] = cadd(acc[m], o[m * 32 + lane]);
                }
            }
            if (TAIL) __syncthreads();          // a warp's ring is free again once its sums have been read
            if (q > 0) continue;
        }
        // ---- out = x - eta * sum, and Re<x, out>, <out, out> per row for the caller's inner products ----
        double dsum = 0.0, nsum = 0.0;
        if (row_ok) {
#pragma unroll
            for (int m = 0; m < R0; ++m) {
                const cf xv = ADJ ? make_float2(0.f, 0.f) : x_at(j + RL * m);
                const cf av = acc[m];
                const float se = HAS_ATY ? a.eta : -a.eta;          // HAS_ATY: acc holds aty - sum
                const cf ov = make_float2(fmaf(se, av.x, xv.x), fmaf(se, av.y, xv.y));
                store_image(a.out, x_off + j + RL * m, ov, a.out_planar, b, a.plane);
                if (DOT) { dsum += (double)xv.x * ov.x + (double)xv.y * ov.y; nsum += (double)ov.x * ov.x + (double)ov.y * ov.y; }
            }
        }
        if (SMW && DOT && a.dot_blocks) {
            for (int o = 16; o > 0; o >>= 1) { dsum += __shfl_down_sync(0xffffffffu, dsum, o); nsum += __shfl_down_sync(0xffffffffu, nsum, o); }
            __syncwarp();                // the image has been read
            if (lane == 0) { double* p = reinterpret_cast<double*>(sX); p[0] = dsum; p[1] = nsum; p[2] = (double)b; }
        } else if (DOT) {
            for (int o = pow2_ceil(RL) / 2; o > 0; o >>= 1) {
                const double d = __shfl_down_sync(0xffffffffu, dsum, o), n = __shfl_down_sync(0xffffffffu, nsum, o);
                if (j + o < RL) { dsum += d; nsum += n; }
            }
            if (j == 0 && row_ok) { a.dot_rows[row] = dsum; a.dot_rows[a.nrows + row] = nsum; }
        }
    }
    if (SMW && DOT && a.dot_blocks) {    // one pair of sums per block and example, in a fixed order
        __syncthreads();
        if (warp == 0) {
            const int warps = blockDim.x >> 5;
            const double* p = reinterpret_cast<const double*>(smem + (lane < warps ? lane : 0) * WF::ELEMS + WF::OFF_X);
            const bool has = lane < nwhole || (lane < warps && ((lane - nwhole) & 3) == 0);
            for (int ex = 0; ex < a.dot_blocks; ++ex) {
                const bool mine = has && p[2] == (double)ex;
                double d = mine ? p[0] : 0.0, n = mine ? p[1] : 0.0;
                for (int o = 8; o > 0; o >>= 1) { d += __shfl_down_sync(0xffffffffu, d, o); n += __shfl_down_sync(0xffffffffu, n, o); }
                if (lane == 0) { double* out = a.dot_rows + (long long)ex * a.T * a.RPB + blockIdx.x; out[0] = d; out[a.nrows] = n; }
            }
        }
    }
}

}  // namespace gleam
