// Per-length launch table: one entry per supported transform length, defined in the translation
// unit that instantiates the kernels of that length.
#pragma once
#include "dc_kernels.cuh"
#include "dc_warpline.cuh"
#include "dc_warpflat.cuh"
#include "dc_coilpar.cuh"

#include <atomic>
#include <type_traits>

namespace gleam {

// Launch state that CUDA keeps per device (function attributes, occupancy, SM count) is cached per
// device ordinal: one process may drive several GPUs, from several host threads.  The cached values
// are idempotent, so two threads that race on a first use both compute and store the same thing.
constexpr int MAX_DEVICES = 64;
struct PerDevice {
    std::atomic<int> v[MAX_DEVICES];         // 0 = not yet known on that device
    std::atomic<int>* slot() {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return nullptr;
        return &v[dev];
    }
};

// Launches the row kernel; with `lets_in` nothing is launched, it tells whether the launch would let the next one in at its start
// (grid_launch_dependents; a single round of blocks).
typedef cudaError_t (*RowLaunch)(const RowArgs& a, cudaStream_t s, bool* lets_in);

struct SizeOps {
    int N, unit_r0;              // unit_r0: units per line of the row kernels that take z (one plan for all of them)
    RowLaunch row;
    cudaError_t (*col_z)(const ColArgs& a, const RowArgs* row, RowLaunch row_launch, cudaStream_t s);
};

// static_bytes: statically declared shared memory of the kernel, which counts against the same
// 48 KB default limit as the dynamic part
template <class K>
inline cudaError_t ensure_smem(K kernel, size_t bytes, PerDevice& done, size_t static_bytes = 0) {
    if (bytes + static_bytes <= 48 * 1024) return cudaSuccess;
    std::atomic<int>* flag = done.slot();               // null: device ordinal outside the cache, set every time
    if (flag && flag->load(std::memory_order_acquire)) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    if (flag) flag->store(1, std::memory_order_release);
    return cudaSuccess;
}

// SM count of the current device, cached per device
inline cudaError_t device_sms(int* out) {
    static PerDevice cache;
    std::atomic<int>* c = cache.slot();
    if (c) { const int v = c->load(std::memory_order_acquire); if (v > 0) { *out = v; return cudaSuccess; } }
    int dev = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(out, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if (c) c->store(*out, std::memory_order_release);
    return cudaSuccess;
}

// resident blocks of `kernel` on the current device (SM count x blocks per SM), cached per device
template <class K>
inline cudaError_t resident_slots(K kernel, int threads, size_t smem, PerDevice& cache, int* out) {
    std::atomic<int>* c = cache.slot();
    if (c) { const int v = c->load(std::memory_order_acquire); if (v > 0) { *out = v; return cudaSuccess; } }
    int sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = device_sms(&sms)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem)) != cudaSuccess) return e;
    *out = sms * (per_sm > 0 ? per_sm : 1);
    if (c) c->store(*out, std::memory_order_release);
    return cudaSuccess;
}

// persistent launch of the warp-resident row kernel: one block per resident slot, warps stride
// over the line groups
template <class P, bool HAS_Z, bool ADJ>
inline cudaError_t launch_warpline_z(const RowArgs& a, cudaStream_t s, bool* lets_in) {
    using WL = WarpLine<P, HAS_Z>;
    constexpr int WARPS = 1;
    constexpr size_t SMEM = sizeof(cf) * WARPS * WL::WARP_ELEMS_ALIGNED;
    static PerDevice attr_done;
    static PerDevice slots_cache;
    cudaError_t e = ensure_smem(warpline_kernel<P, WARPS, HAS_Z, ADJ>, SMEM, attr_done);
    if (e != cudaSuccess) return e;
    int slots = 0;
    if ((e = resident_slots(warpline_kernel<P, WARPS, HAS_Z, ADJ>, WARPS * 32, SMEM, slots_cache, &slots)) != cudaSuccess) return e;
    const long long groups = (a.nrows + WL::LW - 1) / WL::LW;
    long long blocks = (groups + WARPS - 1) / WARPS;
    if (lets_in) { *lets_in = blocks <= slots; return cudaSuccess; }
    if (blocks <= 0) return cudaSuccess;
    if (blocks > slots) blocks = slots;
    return launch_overlapped(true, warpline_kernel<P, WARPS, HAS_Z, ADJ>, dim3((unsigned)blocks),
                             dim3(WARPS * 32), SMEM, s, a);
}

// GLEAM_NO_SPLIT=1 keeps single-warp blocks for every group (tuning aid, read once).
inline bool split_enabled() {
    static int v = -1;
    if (v < 0) { const char* e = getenv("GLEAM_NO_SPLIT"); v = (e && e[0] == '1') ? 0 : 1; }
    return v == 1;
}

// the one-pass kernel with the k-space units numbered across the coils (dc_warpflat.cuh)
template <class P, bool HAS_Z, bool HAS_ATY, bool ADJ, bool DOT>
inline cudaError_t launch_warpflat_zy(const RowArgs& a, cudaStream_t s, bool* lets_in) {
    static_assert(WarpFlat<P, HAS_Z>::ELIGIBLE, "not a plan the coil-numbered kernel takes");
    using WF = WarpFlat<P, HAS_Z, false>;
    static PerDevice attr_done;
    static PerDevice slots_cache;
    cudaError_t e = ensure_smem(warpflat_kernel<P, HAS_Z, FLAT_SINGLE, HAS_ATY, ADJ, DOT>, WF::WARP_BYTES, attr_done);
    if (e != cudaSuccess) return e;
    int slots = 0;
    if ((e = resident_slots(warpflat_kernel<P, HAS_Z, FLAT_SINGLE, HAS_ATY, ADJ, DOT>, 32, WF::WARP_BYTES, slots_cache, &slots)) != cudaSuccess) return e;
    const long long groups = (a.nrows + WF::LW - 1) / WF::LW;
    if (lets_in) *lets_in = !HAS_Z && groups <= slots;       // single-warp blocks; one block per SM: below
    if (groups <= 0) return cudaSuccess;
    // One round of 8 to 16 groups per SM: one block per SM that holds all its warps.  4 k + 1 (or 4 k + 2) groups per
    // SM: the groups beyond 4 k are split by coils over four warps each, one per scheduler.  (Measured on cine-shaped
    // problems, per call: 13 groups per SM 18.7 -> 16.6 us, with z 22.7 -> 21.5 us, 12 per SM 18.7 -> 15.3 us; up to 7 per SM single-warp
    // blocks are faster, 11.3 against 12.7 us.)
    if constexpr (P::RL <= 16 && P::R0 <= 12 && !WF::PRIME) {   // larger butterflies need more registers than 16 warps per SM leave
        using WS = WarpFlat<P, HAS_Z, true>;
        static PerDevice attrs_done;
        int sms = 0;
        if (split_enabled() && groups <= slots && device_sms(&sms) == cudaSuccess && groups > 7LL * sms) {
            const int per = (int)((groups + sms - 1) / sms);
            int nsplit = (a.C >= 4 && (per % 4 == 1 || per % 4 == 2)) ? per % 4 : 0;
            if (per - nsplit + 4 * nsplit > 16) nsplit = 0;
            const int nwhole = per - nsplit, warps = nwhole + 4 * nsplit;
            const size_t bytes = WS::WARP_BYTES * (size_t)warps;
            if (warps <= 16 && bytes <= 227 * 1024) {
                // A sum per block and example, for few examples: the lines of a group belong to one (a line of it decides which).
                // One warp adds an example after another at the end of the block.  Per row -> per block, VJP of 10 steps, 8 coils
                // of 160 points: 1 example of 3840 rows 267 -> 247 us, 2 of 1920 259 -> 252, 3 of 1288 272 -> 269; 4 of 800 still 242 ->
                // 224, but 5 of 640 214 -> 223, 6 of 640 249 -> 259, 8 of 480 251 -> 265.
                const long long rows = (long long)a.T * a.RPB;
                const bool whole = DOT && rows >= sms && rows % WF::LW == 0 && a.nrows <= 3 * rows;
                if (DOT && a.dot_form) *a.dot_form = DotForm{whole ? sms : (int)rows, warps, nsplit > 0};
                if (lets_in) { *lets_in = true; return cudaSuccess; }
                RowArgs b = a;
                b.dot_blocks = whole ? (int)(a.nrows / rows) : 0;
                // the attribute is set once, to what the largest block of this kernel can ask for
                constexpr size_t SMEM_CAP = 227 * 1024;
                if ((e = ensure_smem(warpflat_kernel<P, HAS_Z, FLAT_SM, HAS_ATY, ADJ, DOT>, 16 * WS::WARP_BYTES < SMEM_CAP ? 16 * WS::WARP_BYTES : SMEM_CAP, attrs_done)) != cudaSuccess) return e;
                return launch_overlapped(true, warpflat_kernel<P, HAS_Z, FLAT_SM, HAS_ATY, ADJ, DOT>, dim3((unsigned)sms), dim3(32 * warps), bytes, s, b, nwhole);
            }
        }
    }
    if (lets_in) return cudaSuccess;
    // A nearly empty last round: blocks of four warps that share each group of it, a quarter of the coils each (FLAT_TAIL).  Such a
    // round costs a warp's whole run time however few groups it has: 4 x 15 coils of 640 x 368 are 1280 groups on 1184 warps, VJP
    // 77.6 -> 63.6 us, and 2560 with z, prepared step 92 -> 84.  Two lines, by the warps an SM holds:
    // 8 or fewer (368, 512, 640 points): a last round of at most a quarter of the warps.  6 to 32 coils: VJP behind one full round 1.05-
    // 1.30 times as fast; prepared step behind one to fourteen 1.00-1.33, 368 points 1.02 in the mean at 14 rounds, 640 points 1.05 (with
    // every second line sampled and 6 rounds or more 0.96-1.02).  The warps of a block drift apart over the rounds and wait for
    // one another before the last: with 512 points 1.03 at 5 rounds, 1.01 at 6, 0.99 from 8 on (0.96 at worst), so at most 6.
    // More: the single-warp blocks, which finish one by one, fill the last round themselves (VJP, 7 to 12 coils of 320 and 384 points,
    // 0.82-0.93 times as fast in fours); only prepared steps behind one full round gain, 1.04-1.29 with 12 to 16 coils and at most 15
    // % of the warps in the last round (0.95-0.98 with fewer coils or more groups).
    // Two groups a block: 368 points 1.09, most others slower.  A group of few units is one round whoever shares it.
    // Spilled for it (128 threads, the bound of the single warps): VJP of 368 points 56 B, with A^H y 52; prepared step of 384 points 92
    // (single warps 32), 160 points 48, 320 points 12, 256 points 4 (none).
    constexpr bool FEW_WARPS = WF::SINGLE_BLOCKS <= 8;
    constexpr long long MOST_ROUNDS = P::N == 512 ? 6 : 1LL << 40;
    if constexpr ((FEW_WARPS || HAS_Z) && 4 * WF::WARP_BYTES <= 227 * 1024) {
        if (groups > slots && a.C >= (FEW_WARPS ? 6 : 12) && WF::UPC * a.C > 64) {
            static PerDevice tail_attr_done, tail_cache;
            constexpr size_t BYTES = 4 * WF::WARP_BYTES;
            int resident = 0;
            if ((e = ensure_smem(warpflat_kernel<P, HAS_Z, FLAT_TAIL, HAS_ATY, ADJ, DOT>, BYTES, tail_attr_done)) != cudaSuccess) return e;
            if ((e = resident_slots(warpflat_kernel<P, HAS_Z, FLAT_TAIL, HAS_ATY, ADJ, DOT>, 128, BYTES, tail_cache, &resident)) != cudaSuccess) return e;
            const long long full = groups / (4LL * resident), tail = groups % (4LL * resident);
            if (4 * resident >= slots && tail > 0 && (FEW_WARPS ? tail <= resident : 5 * tail <= 3 * resident) && (full == 1 || (FEW_WARPS && HAS_Z && full <= MOST_ROUNDS)))
                return launch_overlapped(true, warpflat_kernel<P, HAS_Z, FLAT_TAIL, HAS_ATY, ADJ, DOT>, dim3((unsigned)resident), dim3(128), BYTES, s, a, 4);
        }
    }
    long long blocks = groups;
    if (blocks > slots) blocks = slots;
    return launch_overlapped(true, warpflat_kernel<P, HAS_Z, FLAT_SINGLE, HAS_ATY, ADJ, DOT>, dim3((unsigned)blocks), dim3(32), WF::WARP_BYTES, s, a, 1);
}
template <class P, bool HAS_Z>
inline cudaError_t launch_warpflat_z(const RowArgs& a, cudaStream_t s, bool* lets_in) {
    if constexpr (!HAS_Z) { if (a.aty != nullptr) return launch_warpflat_zy<P, false, true, false, false>(a, s, lets_in); }
    else { if (a.x == nullptr) return launch_warpflat_zy<P, true, false, true, false>(a, s, lets_in); }
    if constexpr (!HAS_Z) { if (a.dot_rows != nullptr) return launch_warpflat_zy<P, false, false, false, true>(a, s, lets_in); }
    return launch_warpflat_zy<P, HAS_Z, false, false, false>(a, s, lets_in);
}
// GLEAM_NO_FLAT=1 keeps the plain warp-resident kernel for those lengths (tuning aid, read once).
inline bool flat_enabled() {
    static int v = -1;
    if (v < 0) { const char* e = getenv("GLEAM_NO_FLAT"); v = (e && e[0] == '1') ? 0 : 1; }
    return v == 1;
}

// Stage plans of the one-pass kernel with units numbered across coils, per length: the last radix RL (butterflies of
// the first stage per line) for calls without and with z, 0 where the plain warp-resident kernel with the plan of
// sizes.def is used.  The line lies where the lanes are: a length stays on the plain kernel while that keeps three
// quarters of them busy in both stages.  Measured, VJP / prepared step, 8 x 16 coils x 512 rows, plain -> numbered:
// 46: 100 / 113 -> 23 / 33 us; 92: 107 / 127 -> 36 / 49; 184: 127 / 144 -> 68 / 81; 384: 150 / 217 -> 89 / 125;
// 512: 153 / 252 -> 124 / 157; 640: 391 / 822 -> 155 / 200 (three-stage block kernel before); 64 as 4 x 16 and 32 as
// 4 x 8 for the VJP: 19 -> 16, 23 -> 15 us; but 120: 37 / 44 -> 42 / 56, 240: 60 / 72 -> 69 / 88.  With z, 256 gains where a
// line has more samples than are staged (at 3.2x 156 -> 101 us, at 6x equal), 32 28 -> 24 us.
// With z one plan has to serve every problem of a length, since the ranks of the samples follow it.  Prepared steps, this
// plan against the other: 368 as 16 x 23 against 23 x 16, 19 problems of 320 to 5120 rows and 4 to 16 coils: faster in 15 (8 coils
// of 640 rows 21 against 28 us, 15 of 2560 93 against 106), slower by up to 13 % where 23 x 16 just fills its last round (15 of
// 1920 rows 74 against 65, 16 of 2048 77 against 69).  64 as 8 x 8 against 4 x 16: faster while the coils go side by side (2 x 16
// coils of 512 rows 8.6 against 16.8 us), slower beyond (8 x 16 coils of 512 28.5 against 21.4, 24 x 8 of 128 15.6 against 10.7).
template <int N> struct FlatRL { static constexpr int v = 0, z = 0; };
#define GLEAM_FLAT(N, V, Z) template <> struct FlatRL<N> { static constexpr int v = V, z = Z; };
GLEAM_FLAT(32, 8, 8)
GLEAM_FLAT(46, 23, 23)
GLEAM_FLAT(48, 8, 8)
GLEAM_FLAT(64, 16, 0)
GLEAM_FLAT(80, 16, 16)
GLEAM_FLAT(92, 23, 23)
GLEAM_FLAT(96, 16, 16)
GLEAM_FLAT(128, 16, 16)
GLEAM_FLAT(160, 16, 16)
GLEAM_FLAT(184, 23, 23)
GLEAM_FLAT(192, 0, 32)
GLEAM_FLAT(256, 0, 16)
GLEAM_FLAT(320, 32, 32)
GLEAM_FLAT(368, 16, 23)
GLEAM_FLAT(384, 32, 32)
GLEAM_FLAT(512, 32, 32)
GLEAM_FLAT(640, 32, 32)
#undef GLEAM_FLAT
template <class P, int RL> using FlatPlan = Plan<P::N, P::N / RL, RL>;

// the plan of every row kernel that takes z: the ranks of the sampled positions follow its units
template <class P> using ZPlan = std::conditional_t<FlatRL<P::N>::z != 0, FlatPlan<P, FlatRL<P::N>::z ? FlatRL<P::N>::z : P::RL>, P>;

// Few lines: the coils of a line group side by side (dc_coilpar.cuh), as long as that takes no more than 16 warps per SM
// and so many rounds of resident blocks (shared memory holds one line group per coil, registers 16 warps per SM).
// Measured per call, numbered or plain kernel -> here: one 64 x 64 slice of 8 coils 12.5 -> 4.3 us (prepared step),
// 4.7 -> 3.4 us (VJP); 6 x 8 coils of 46 x 240 18.6 -> 7.3 and 11.7 -> 6.2 us; beyond 16 warps per SM 6 x 4 coils of
// 368 x 80 7.6 -> 11.3 us; with 2 or 3 coils 3.9 -> 4.8 us.  Larger problems first take several coils per warp: prepared
// step of 8 x 16 coils of 128 x 24 24 -> 5.9 us, 4 x 7 coils of 384 x 32 12.7 -> 5.5 us, 6 x 10 coils of 128 x 160 16 -> 11 us;
// not below 8 warps without z (14 x 17 frames of 64 x 128, VJP 11 -> 16 us with 4) and not for last radices beyond 16
// (16 coils of 320 x 320, 19.5 -> 26 us).  *taken: the call was launched here.
//
// Rounds.  A second one costs as much as the first, so it pays only where a coil costs the other kernel much.  Prepared
// step / VJP, other kernel -> two rounds: 16 x 23 points, 12 coils of 184 x 368 23.2 / 26.6 -> 18.0 / 16.6 us, 9 coils of 240
// x 368 18.9 / 20.6 -> 18.2 / 16.5; 256 points, 2 x 16 coils of 512 x 256 35.2 -> 31.5, 12 coils of 640 x 256 27.5 -> 22.5; 240
// points, 14 coils of 320 x 240 24.2 / 18.7 -> 18.1 / 15.2; 160 points, 12 coils of 384 x 160 18.0 / 11.4 -> 11.8 / 9.5.  It does
// not with 32 lanes or few image-side butterflies, where the numbered kernel is at its best: 7 coils of 320 x 320 11.6 / 7.8
// -> 15.2 / 12.6, 7 coils of 320 x 512 14.4 / 10.8 -> 19.9 / 16.4, 12 coils of 192 x 640 25.8 / 19.0 -> 24.5 / 23.4; 12 coils of
// 184 x 184 13.1 / 9.6 -> 14.7 / 12.0, of 192 x 92 8.9 / 7.0 -> 13.1 / 10.6.  With z and last radices up to 16, fewer warps that
// make it one round come first: 12 coils of 384 x 240 15.8 -> 13.9, of 384 x 160 11.8 -> 9.6.
template <class P, bool HAS_Z, bool ADJ>
inline cudaError_t launch_coilpar(const RowArgs& a, cudaStream_t s, bool* taken, bool* lets_in) {
    using CP = CoilPar<P>;
    *taken = false;
    int sms = 0;
    cudaError_t e = device_sms(&sms);
    if (e != cudaSuccess) return e;
    constexpr int WARPS = 16;
    constexpr int ROUNDS = (P::RL == 32 || (P::RL == 23 && P::R0 <= 8)) ? 1 : 2;
    // fewest warps that still pay: each takes several coils then, so that more line groups are resident at once
    constexpr int LEAST = !HAS_Z ? 8 : P::RL <= 16 ? 4 : WARPS;
    int warps = a.C < WARPS ? a.C : WARPS;
    const long long groups = (a.nrows + CP::LW - 1) / CP::LW;
    while (groups * warps > (long long)WARPS * sms && (warps + 1) / 2 >= LEAST) warps = (warps + 1) / 2;
    if (a.C < 4 || groups <= 0 || groups * warps > (long long)WARPS * sms) return cudaSuccess;
    static PerDevice done, by_warps[WARPS + 1];
    if ((e = ensure_smem(coilpar_kernel<P, HAS_Z, ADJ>, CP::LIMIT, done)) != cudaSuccess) return e;
    long long rounds = 0;
    auto count_rounds = [&](int w) -> cudaError_t {
        int slots = 0;                                       // by threads and registers; shared memory depends on the coils
        if ((e = resident_slots(coilpar_kernel<P, HAS_Z, ADJ>, 32 * w, 0, by_warps[w], &slots)) != cudaSuccess) return e;
        const long long by_smem = (long long)sms * (CP::SM_BYTES / (CP::bytes(w, a.C) + CP::BLOCK_BYTES));
        const long long resident = slots < by_smem ? slots : by_smem;
        rounds = resident > 0 ? (groups + resident - 1) / resident : groups;
        return cudaSuccess;
    };
    if ((e = count_rounds(warps)) != cudaSuccess) return e;
    if (HAS_Z && P::RL <= 16 && rounds > 1) {
        const int most = warps;
        const long long with_most = rounds;
        while (rounds > 1 && (warps + 1) / 2 >= LEAST) {
            warps = (warps + 1) / 2;
            if ((e = count_rounds(warps)) != cudaSuccess) return e;
        }
        if (rounds > 1) { warps = most; rounds = with_most; }
    }
    const size_t bytes = CP::bytes(warps, a.C);
    if (bytes > CP::LIMIT || rounds > ROUNDS) return cudaSuccess;
    *taken = true;
    if (lets_in) { *lets_in = rounds <= 1; return cudaSuccess; }
    return launch_overlapped(true, coilpar_kernel<P, HAS_Z, ADJ>, dim3((unsigned)groups), dim3(32 * warps), bytes, s, a);
}

template <class P>
inline cudaError_t launch_warpline(const RowArgs& a, cudaStream_t s, bool* lets_in) {
    bool taken = false;
    const cudaError_t e = a.z == nullptr ? launch_coilpar<ZPlan<P>, false, false>(a, s, &taken, lets_in)
                        : a.x != nullptr ? launch_coilpar<ZPlan<P>, true, false>(a, s, &taken, lets_in) : launch_coilpar<ZPlan<P>, true, true>(a, s, &taken, lets_in);
    if (taken || e != cudaSuccess) return e;
    // the numbering across coils pays once a round of 32 units spans more than one coil
    const bool flat = flat_enabled() && a.C >= 2;
    if constexpr (FlatRL<P::N>::v != 0) if (flat && a.z == nullptr) return launch_warpflat_z<FlatPlan<P, FlatRL<P::N>::v>, false>(a, s, lets_in);
    if constexpr (FlatRL<P::N>::z != 0) if (flat && a.z != nullptr) return launch_warpflat_z<FlatPlan<P, FlatRL<P::N>::z>, true>(a, s, lets_in);
    if (a.z == nullptr) return launch_warpline_z<P, false, false>(a, s, lets_in);
    return a.x != nullptr ? launch_warpline_z<ZPlan<P>, true, false>(a, s, lets_in) : launch_warpline_z<ZPlan<P>, true, true>(a, s, lets_in);
}

// row, row_launch: the row launch of such a call (2-D problems), or null
template <class P, int L>
inline cudaError_t launch_col_z(const ColArgs& a, const RowArgs* row, RowLaunch row_launch, cudaStream_t s) {
    using E = LineFFT<P, L>;
    using CZ = ColZ<P, L>;
    static PerDevice attr_done, slots_cache;
    cudaError_t e = ensure_smem(col_z_kernel<P, L>, CZ::SMEM_BYTES, attr_done, (COLZ_SELF_MAX + COLZ_SELF_MAX / 32) * sizeof(int));
    if (e != cudaSuccess) return e;
    int slots = 0;
    if ((e = resident_slots(col_z_kernel<P, L>, E::THREADS, CZ::SMEM_BYTES, slots_cache, &slots)) != cudaSuccess) return e;
    if (a.images <= 0) return cudaSuccess;
    // The number of sampled ranks is known only on the device.  The blocks of an image share its tiles: one round of
    // blocks, more for volumes (ColZ::TILES).
    ColArgs b = a;
    const long long most = (long long)a.C * ((a.es + L - 1) / L);
    long long bpi = slots / a.images;
    if (a.rank == 3 && CZ::TILES > 0 && bpi < most / cmax(CZ::TILES, 1)) bpi = most / cmax(CZ::TILES, 1);
    b.bpi = (int)(bpi < 1 ? 1 : bpi > most ? most : bpi);
    const long long blocks = (long long)a.images * b.bpi;
    if (blocks > 2147483647LL) return cudaErrorInvalidConfiguration;
    // Scheduled as the launch before it ends, except where that may be a row launch which lets the next launch in at its start
    // (asked of the row launch of such a call, without z and with it): early blocks of the table then crowd the SMs that had
    // room.  Forward and VJP in turn, without -> with the attribute: one round, 2 x 16 coils of 640 x
    // 320 91 -> 116 us, 4 x 8 of 384 x 384 66 -> 85, 3 x 15 of 640 x 368 (the VJP alone is one round) 162 -> 169, 20 frames x
    // 8 of 192 x 160 54 -> 62; several rounds, 24 frames 71.9 -> 69.8, 4 x 15 of 640 x 368 226.5 -> 224.0, 4 x 8 coils x 8 frames
    // of 128 x 92 52.1 -> 50.2 (a launch's latency, hidden; enqueued call by call, equal in a replayed graph).  Where only
    // single-warp blocks with z are one round, which let nothing in, 11 x 6 coils of 320 x 256, two forwards and a VJP 110.9 ->
    // 106.2.  Grids of a few blocks gain, too.
    bool overlap = true;
    if (row != nullptr && blocks > 64) {
        RowArgs plain = *row;
        plain.z = nullptr; plain.aty = nullptr;
        bool lets_in = false;
        if ((e = row_launch(plain, s, &lets_in)) != cudaSuccess) return e;
        if (!lets_in && (e = row_launch(*row, s, &lets_in)) != cudaSuccess) return e;
        overlap = !lets_in;
    }
    return launch_overlapped(overlap, col_z_kernel<P, L>, dim3((unsigned)blocks), dim3(E::THREADS), CZ::SMEM_BYTES, s, b);
}

template <class P, class PC, int LC>
struct SizeImpl {
    static_assert(WarpLine<P>::ELIGIBLE, "row plans have at most two stages of at most 32 butterflies");
    static cudaError_t row(const RowArgs& a, cudaStream_t s, bool* lets_in) { return launch_warpline<P>(a, s, lets_in); }
    static cudaError_t col_z(const ColArgs& a, const RowArgs* row, RowLaunch row_launch, cudaStream_t s) { return launch_col_z<PC, LC>(a, row, row_launch, s); }
};

}  // namespace gleam
