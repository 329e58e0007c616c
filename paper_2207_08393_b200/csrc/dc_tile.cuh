// Row-tile kernels: the phase-encode plane (ky, kz) of the 3-D path, or the whole slice (n1, n2) of a 2-D problem
// with an arbitrary mask, is transformed so that every pass over the coil workspace is contiguous in memory.
//
// ky has the split N1 = RY * BY, kz the one- or two-stage plan PZ.  With ky = j + BY m (m < RY) on the image side
// and ky = k0 + RY k1 (k1 < BY) on the k-space side:
//   pass 1  tile_fwd : block (b,t,i0,j) takes the RY rows ky = j + BY m, multiplies by S_c, transforms the rows
//                      against each other (radix RY, one thread per kz), then each row along kz, and stores
//                      V[unit][i0][k0][j][kz].
//   pass 2  mid      : block (unit,i0,k0) reads the BY rows V[..][k0][0..BY)[kz], applies the ky twiddles
//                      w_N1^(j k0), radix-BY transform over j (-> k1), the k-space work of the call at the raw
//                      position (k0 + RY k1, kz), and the mirror image back, in place.
//   pass 3  tile_inv : mirror of pass 1 with the conjugate-sensitivity coil sum and the update of Eq. 3.
//
// All stages of passes 1 and 3 are distributed over the whole block (a stage of N butterflies keeps N lanes busy
// whatever the radices are; with one warp per row, as before, a 23-point stage of 184 = 8 x 23 used 8 of every 32
// lanes).  The radix-RY stage comes first because it reads the staged sensitivities column by column as they lie in
// memory; the ky twiddles belong to the middle pass, which is bound by memory and has issue slots to spare.
#pragma once
#include "size_ops.cuh"

namespace gleam {

struct TileArgs {
    const cf* x; const cf* sens; cf* out;     // image side; x may be null in pass 3 (a zero image)
    cf* V;                                    // workspace
    long long v_unit, v_slab, v_k0, v_j;      // its strides (elements); kz is contiguous
    float eta;
    int C, T, Ts, n0, G, i0_start, BY;
    int csplit;                               // the coils of one tile are dealt to this many blocks (pass 3: a cluster)
    int x_planar, out_planar; long long plane; // two-real-channel layout of x / out (see RowArgs)
    const cf* aty;                            // A^H y image of the normal-equations form, or null (see RowArgs)
};

// LOOSE: of kernels that are built in two forms, the one with more registers and fewer blocks on an SM (TWO_FWD, TWO_INV).
template <class PZ, int RY, bool LOOSE = false>
struct Tile {
    static constexpr int NZ = PZ::N, R0 = PZ::R0, RL = PZ::RL, S = PZ::S;
    static constexpr int BF0 = PZ::BF0;                      // butterflies per row of the first kz stage
    static constexpr int LS1 = PZ::LS1;                      // odd run length: the second stage reads without bank conflicts
    static constexpr int TH = ((NZ + 31) / 32) * 32;         // one thread per kz column
    static constexpr int RMAX = cmax(RY, cmax(R0, RL));
    static constexpr bool PRIME = RMAX > 4 && RMAX % 2 == 1 && smallest_odd_factor(RMAX) == RMAX;
    // The outputs of a prime radix are stored as they are formed on long rows (8 coils of 96 x 240 x 368 807 -> 804 us, 12 of 96 x
    // 240 x 184 493 -> 488; but 128 x 92 x 92 125 -> 129).  A bound without room for them spills all the same (up to 80 B); more
    // blocks outweigh that where few image rows are kept and blocks are large: VJP of 8 coils, us, 128 x 92 x 184 283 -> 234,
    // 128 x 92 x 368 602 -> 485, 256 x 46 x 184 361 -> 325, 4 slices of 92 x 184 23.6 -> 18.9; not with 16 rows (up to 244 B; 128 x
    // 256 x 92 239 -> 264, 128 x 96 x 184 193 -> 202) nor on short rows (24 x 92 x 92, 4 coils, 17.8 -> 18.8).  Only where they save a
    // round of blocks (LOOSE otherwise, TileImpl).
    static constexpr bool EARLY = NZ >= 184, SHORT = PRIME && RY <= 4 && EARLY, TIGHT = SHORT && !LOOSE;
    // Threads per row in the first kz stage.  Half warps of 23 butterflies a row met on one bank where they cross to the next row, in
    // every read and write of the stage; with a thread left out per row, and rows congruent to 24 modulo 16, they do not.  VJP of
    // 12 coils of 96 x 240 x 184 490 -> 476 us, of 8 of 96 x 240 x 368 804 -> 781.
    static constexpr int BFP = RL == 23 && R0 >= 8 ? 24 : BF0;
    // A thread whose butterflies all have one place in their rows keeps their twiddles: 476 -> 458 and 781 -> 772 us, 4 slices of
    // 320 x 384 77 -> 74, 8 coils of 128 x 160 x 64 90 -> 87.  Where registers admit it: not 10- and 12-point stages next to short
    // ones (64 x 96 rows of 96 46.9 -> 51.1, 128 x 240 of 160 347 -> 357), nor 512 points (320 x 512 94 -> 95), nor SHORT tiles.
    static constexpr bool OWN_TW = S == 2 && TH % BFP == 0 && (R0 <= 8 || (RL >= 23 && NZ <= 384)) && !SHORT;
    // In pass 3 not where they spill (20 rows of 64, 47 x 11 coils of 640 x 64 80 -> 91 us a pass), nor for 16 rows of 368, one block per
    // SM with them or without (13 coils of 24 x 256 x 368 158 -> 163).  With 8 rows of 24 points they cost blocks on an SM (89
    // registers -> 99, 20 blocks -> 16: 9 coils of 368 x 64 x 24 24.8 -> 28.6), so only where that takes no further round (LOOSE).
    static constexpr bool FEWER_BLOCKS = RY == 8 && NZ == 24;
    static constexpr bool OWN_TW_INV = OWN_TW && (LOOSE || !FEWER_BLOCKS) && !(RY == 20 && NZ == 64) && !(RY == 16 && NZ == 368);
    static constexpr bool TWO_FWD = SHORT, TWO_INV = SHORT || FEWER_BLOCKS;      // kernels in two forms, chosen by rounds (TileImpl)
    // Slots of a row in the exchange tile.  Congruent to BFP modulo 16: threads take the butterflies of the first kz stage row
    // after row, and each then has the bank of its thread number.  With rows of R0 runs (odd, packed) two rows of a half warp
    // met on the same banks in its reads and writes.  Packed -> congruent, VJP call, us: 8 coils of 64 x 128 x 128 79.9 -> 73.2,
    // 96 x 96 x 96 76.7 -> 72.0, 64 x 240 x 192 226 -> 217, 48 x 320 x 240 281 -> 272, 48 x 320 x 320 386 -> 375.
    // Not for short rows and first radices below 8, where the second stage crosses rows more often than that
    // gains: 64 x 92 x 92 62.7 -> 63.9, 80 x 64 x 46 40.8 -> 41.8, 64 x 96 x 40 30.1 -> 30.2.  (Rows of 23-point
    // stages congruent to 23 were slower, too: forward of 15 coils of 128 x 160 x 184 746 -> 793.)
    static constexpr int PACKED = R0 * LS1;
    static constexpr int ROW = S != 2 ? NZ : (R0 < 8 || NZ < 64) ? PACKED : PACKED + ((BFP - PACKED) % 16 + 16) % 16;
    static constexpr int T_ELEMS = (RY * ROW + 1) / 2 * 2, STAGE = RY * NZ, TW = (S == 2 && !OWN_TW) ? NZ : 0, TW_INV = (S == 2 && !OWN_TW_INV) ? NZ : 0;
    static constexpr int slot(int kz) { return (S == 2) ? (kz / BF0) * LS1 + kz % BF0 : kz; }
    static constexpr size_t LIMIT = 227 * 1024;
    static constexpr size_t FWD_BYTES = sizeof(cf) * (T_ELEMS + STAGE + TW);
    // Pass 3 stages a tile of the workspace and one of the sensitivities.  Where both and the exchange tile take more
    // than a third of the SM they take turns in one buffer: a third block per SM hides more latency than the longer
    // reach of two buffers (8 slices of 320 x 256, 8 coils: 84.7 -> 76.7 us per VJP call).
    static constexpr bool ONE_STAGE = sizeof(cf) * (T_ELEMS + 2 * STAGE + TW_INV) > LIMIT / 3;
    static constexpr size_t INV_BYTES = sizeof(cf) * (T_ELEMS + (ONE_STAGE ? 1 : 2) * STAGE + TW_INV);
    // The register bound lets the blocks that shared memory admits be resident.  RY values of the image or of the coil
    // sum are kept over the coil loop next to a butterfly (a prime radix also holds its sums and differences).
    // The twiddles of OWN_TW are not counted: under bounds that leave room for them pass 1 of 64-point rows would not spill (up to 68 B),
    // but with fewer blocks; with the spills it is 1.00-1.07 times as fast as with twiddles in shared memory.
    // A block has a thread per column, so 640-point rows have at most 96 registers and spill up to 180 B whatever the bound.
    static constexpr int REGS = 2 * RY + (PRIME && !TIGHT ? 4 : 2) * RMAX + (TIGHT ? 24 : 16);
    // Pass 1 with 4 rows of 92 points takes 104 registers where 96 do, 4 warps per scheduler instead of 5 (4 x 2 x 4 coils of 120 x 92 x 92,
    // VJP, 468 -> 451 us).
    static constexpr int REGS_FWD = RY == 4 && NZ == 92 ? 104 : REGS;
    static constexpr int blocks(size_t bytes, int regs) {
        const int n = cmin(16, cmin((int)(LIMIT / (bytes + 1024)), 65536 / (TH * ((regs + 7) / 8 * 8))));
        return cmax(1, cmin(n, 2048 / TH));
    }
};

constexpr int MAX_CSPLIT = 8;                // blocks that may share the coils of a tile
__device__ __forceinline__ void cluster_arrive_wait() {
    asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}
// value of another block's shared memory at the same address as `p` in this block
__device__ __forceinline__ cf cluster_load(const cf* p, unsigned rank) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    unsigned r; cf v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(r));
    return v;
}

// which tile and which coils a block has
struct TileId {
    int b, t, i0, j, c0, c1;
    unsigned bt, gi, part;
    __device__ __forceinline__ explicit TileId(const TileArgs& a) {
        part = blockIdx.x % (unsigned)a.csplit;
        const unsigned blk = blockIdx.x / (unsigned)a.csplit;
        j = (int)(blk % (unsigned)a.BY);
        gi = (blk / (unsigned)a.BY) % (unsigned)a.G;
        bt = blk / ((unsigned)a.BY * (unsigned)a.G);
        b = (int)(bt / (unsigned)a.T); t = (int)(bt - (unsigned)b * a.T);
        i0 = a.i0_start + (int)gi;
        c0 = (int)part * a.C / a.csplit; c1 = ((int)part + 1) * a.C / a.csplit;
    }
};

// RY rows of NZ values, `row_stride` apart in global memory, to a dense tile in shared memory
template <int NZ, int RY>
__device__ __forceinline__ void stage_rows(cf* dst, const cf* src, long long row_stride) {
    if ((int)threadIdx.x < NZ) {
        const int h = (int)threadIdx.x / (NZ / 2), p = (int)threadIdx.x - h * (NZ / 2);
        const cf* s = src + h * row_stride + 2 * p;
        cf* d = dst + h * NZ + 2 * p;
#pragma unroll
        for (int m = 0; m < RY / 2; ++m) { cp_async16(d + 2 * m * NZ, s); s += 2 * row_stride; }
        if (RY % 2 == 1 && h == 0) cp_async16(d + (RY - 1) * NZ, s);
    }
    cp_async_commit();
}

template <class PZ, int RY, bool LOOSE = false>
__global__ void __launch_bounds__(Tile<PZ, RY>::TH, Tile<PZ, RY, LOOSE>::blocks(Tile<PZ, RY, LOOSE>::FWD_BYTES, Tile<PZ, RY, LOOSE>::REGS_FWD))
tile_fwd_kernel(const TileArgs a) {
    grid_dependency_wait();
    using TL = Tile<PZ, RY, LOOSE>;
    constexpr int NZ = PZ::N, R0 = PZ::R0, RL = PZ::RL, BF0 = TL::BF0, BFP = TL::BFP, LS1 = TL::LS1, ROW = TL::ROW, TH = TL::TH;
    extern __shared__ __align__(16) float2 smem[];
    cf* sT = smem;
    cf* sS = smem + TL::T_ELEMS;
    cf* sTw = sS + TL::STAGE;                                 // kz twiddles, [k][j]
    const TileId id(a);
    const int tid = threadIdx.x;
    const bool col = tid < NZ;
    const long long N1NZ = (long long)RY * a.BY * NZ, V3 = a.n0 * N1NZ;
    const long long row_elems = id.i0 * N1NZ + (long long)id.j * NZ, row_stride = (long long)a.BY * NZ;
    const cf* sp = a.sens + ((long long)(id.b * a.C) * a.Ts + (a.Ts > 1 ? id.t : 0)) * V3 + row_elems;
    const long long s_stride = (long long)a.Ts * V3;
    if (id.c0 < id.c1) stage_rows<NZ, RY>(sS, sp + id.c0 * s_stride, row_stride);
    if (TL::S == 2 && !TL::OWN_TW) for (int i = tid; i < NZ; i += TH) sTw[i] = unit_root_fwd<NZ>(((i / BF0) * (i % BF0)) % NZ);
    cf tw[TL::OWN_TW ? R0 : 1];
    if (TL::OWN_TW) {
#pragma unroll
        for (int k = 1; k < (TL::OWN_TW ? R0 : 1); ++k) tw[k] = unit_root_fwd<NZ>((k * (tid % BFP)) % NZ);
    }
    auto twiddle = [&](int k, int j) -> cf { return TL::OWN_TW ? tw[TL::OWN_TW ? k : 0] : sTw[k * BF0 + j]; };
    cf xv[RY];
#pragma unroll
    for (int m = 0; m < RY; ++m)
        xv[m] = col ? load_image(a.x, id.bt * V3 + row_elems + m * row_stride + tid, a.x_planar, id.b, a.plane) : make_float2(0.f, 0.f);

    for (int c = id.c0; c < id.c1; ++c) {
        cp_async_wait<0>();
        __syncthreads();                 // the sensitivities are visible, every thread has left the tile
        if (col) {
            cf v[RY];
#pragma unroll
            for (int m = 0; m < RY; ++m) v[m] = cmul(sS[m * NZ + tid], xv[m]);
            Dft<RY, -1, true>::run(v);
#pragma unroll
            for (int k = 0; k < RY; ++k) sT[k * ROW + TL::slot(tid)] = v[k];
        }
        __syncthreads();
        if (c + 1 < id.c1) stage_rows<NZ, RY>(sS, sp + (c + 1) * s_stride, row_stride);
        const long long unit = ((long long)(id.b * a.C + c)) * a.T + id.t;
        cf* Vp = a.V + unit * a.v_unit + id.gi * a.v_slab + id.j * a.v_j;
        // first kz stage, in place: butterfly j of a row reads and writes the slots {k * LS1 + j}
#pragma unroll 1
        for (int t = tid; t < RY * BFP; t += TH) {
            const int row = t / BFP, j = t - row * BFP;
            if (BFP != BF0 && j >= BF0) continue;
            cf* e = sT + row * ROW + j;
            cf v[R0];
#pragma unroll
            for (int m = 0; m < R0; ++m) v[m] = e[m * LS1];
            Dft<R0, -1, true>::run(v);
            if (TL::S == 2) {
#pragma unroll
                for (int k = 0; k < R0; ++k) e[k * LS1] = (k == 0) ? v[0] : cmul(v[k], twiddle(k, j));
            } else {
                cf* o = Vp + row * a.v_k0;
#pragma unroll
                for (int k = 0; k < R0; ++k) o[k] = v[k];
            }
        }
        if (TL::S == 2) {
            __syncthreads();
            // second kz stage: butterfly j reads the run j * LS1 .. + RL
#pragma unroll 1
            for (int t = tid; t < RY * R0; t += TH) {
                const int row = t / R0, j = t - row * R0;
                const cf* e = sT + row * ROW + j * LS1;
                cf u[RL];
#pragma unroll
                for (int m = 0; m < RL; ++m) u[m] = e[m];
                cf* o = Vp + row * a.v_k0 + j;
                dft_emit<RL, -1, true, TL::EARLY>(u, [&](int k, cf x) { o[R0 * k] = x; });
            }
        }
    }
    cp_async_wait<0>();
}

template <class PZ, int RY, bool LOOSE = false>
__global__ void __launch_bounds__(Tile<PZ, RY>::TH, Tile<PZ, RY, LOOSE>::blocks(Tile<PZ, RY, LOOSE>::INV_BYTES, Tile<PZ, RY, LOOSE>::REGS))
tile_inv_kernel(const TileArgs a) {
    grid_dependency_wait();
    using TL = Tile<PZ, RY, LOOSE>;
    constexpr int NZ = PZ::N, R0 = PZ::R0, RL = PZ::RL, BF0 = TL::BF0, BFP = TL::BFP, LS1 = TL::LS1, ROW = TL::ROW, TH = TL::TH;
    extern __shared__ __align__(16) float2 smem[];
    cf* sT = smem;
    cf* sV = smem + TL::T_ELEMS;
    cf* sS = sV + (TL::ONE_STAGE ? 0 : TL::STAGE);
    cf* sTw = sS + TL::STAGE;
    const TileId id(a);
    const int tid = threadIdx.x;
    const bool col = tid < NZ;
    const long long N1NZ = (long long)RY * a.BY * NZ, V3 = a.n0 * N1NZ;
    const long long row_elems = id.i0 * N1NZ + (long long)id.j * NZ, row_stride = (long long)a.BY * NZ;
    const cf* sp = a.sens + ((long long)(id.b * a.C) * a.Ts + (a.Ts > 1 ? id.t : 0)) * V3 + row_elems;
    const long long s_stride = (long long)a.Ts * V3, x_off = id.bt * V3 + row_elems + tid;
    auto v_ptr = [&](int c) { return a.V + (((long long)(id.b * a.C + c)) * a.T + id.t) * a.v_unit + id.gi * a.v_slab + id.j * a.v_j; };
    if (id.c0 < id.c1) stage_rows<NZ, RY>(sV, v_ptr(id.c0), a.v_k0);
    if (TL::S == 2 && !TL::OWN_TW_INV) for (int i = tid; i < NZ; i += TH) sTw[i] = unit_root_fwd<NZ>(((i / BF0) * (i % BF0)) % NZ);
    cf tw[TL::OWN_TW_INV ? R0 : 1];
    if (TL::OWN_TW_INV) {
#pragma unroll
        for (int k = 1; k < (TL::OWN_TW_INV ? R0 : 1); ++k) tw[k] = unit_root_fwd<NZ>((k * (tid % BFP)) % NZ);
    }
    auto twiddle = [&](int k, int j) -> cf { return TL::OWN_TW_INV ? tw[TL::OWN_TW_INV ? k : 0] : sTw[k * BF0 + j]; };
    cf acc[RY];
#pragma unroll
    for (int m = 0; m < RY; ++m)
        acc[m] = (col && id.part == 0) ? coil_sum_start(a.aty, x_off + m * row_stride) : make_float2(0.f, 0.f);

    for (int c = id.c0; c < id.c1; ++c) {
        cp_async_wait<0>();
        __syncthreads();                 // the workspace tile is visible, every thread has left the other tiles
        if (!TL::ONE_STAGE) stage_rows<NZ, RY>(sS, sp + c * s_stride, row_stride);
        if (TL::S == 2) {
#pragma unroll 1
            for (int t = tid; t < RY * R0; t += TH) {
                const int row = t / R0, j = t - row * R0;
                const cf* o = sV + row * NZ + j;
                cf* e = sT + row * ROW + j * LS1;
                cf u[RL];
#pragma unroll
                for (int k = 0; k < RL; ++k) u[k] = o[R0 * k];
                dft_emit<RL, +1, true, TL::EARLY>(u, [&](int m, cf x) { e[m] = x; });
            }
            __syncthreads();
            if (TL::ONE_STAGE) stage_rows<NZ, RY>(sS, sp + c * s_stride, row_stride);
            else if (c + 1 < id.c1) stage_rows<NZ, RY>(sV, v_ptr(c + 1), a.v_k0);
            else cp_async_commit();
#pragma unroll 1
            for (int t = tid; t < RY * BFP; t += TH) {
                const int row = t / BFP, j = t - row * BFP;
                if (BFP != BF0 && j >= BF0) continue;
                cf* e = sT + row * ROW + j;
                cf v[R0];
#pragma unroll
                for (int k = 0; k < R0; ++k) { const cf r = e[k * LS1]; v[k] = (k == 0) ? r : cmulc(r, twiddle(k, j)); }
                Dft<R0, +1, true>::run(v);
#pragma unroll
                for (int m = 0; m < R0; ++m) e[m * LS1] = v[m];
            }
        } else {
            for (int t = tid; t < RY; t += TH) {
                cf v[R0];
#pragma unroll
                for (int k = 0; k < R0; ++k) v[k] = sV[t * NZ + k];
                Dft<R0, +1, true>::run(v);
#pragma unroll
                for (int m = 0; m < R0; ++m) sT[t * NZ + m] = v[m];
            }
            __syncthreads();
            if (c + 1 < id.c1) stage_rows<NZ, RY>(sV, v_ptr(c + 1), a.v_k0);
            else cp_async_commit();
        }
        cp_async_wait<TL::ONE_STAGE ? 0 : 1>();
        __syncthreads();                 // the sensitivities and the row transforms are visible
        if (col) {
            cf v[RY];
#pragma unroll
            for (int k = 0; k < RY; ++k) v[k] = sT[k * ROW + TL::slot(tid)];
            Dft<RY, +1, true>::run(v);
#pragma unroll
            for (int m = 0; m < RY; ++m) {
                const cf s = sS[m * NZ + tid];
                acc[m].x = fmaf(s.x, v[m].x, fmaf(s.y, v[m].y, acc[m].x));
                acc[m].y = fmaf(s.x, v[m].y, fmaf(-s.y, v[m].x, acc[m].y));
            }
        }
        if (TL::ONE_STAGE) {
            __syncthreads();
            if (c + 1 < id.c1) stage_rows<NZ, RY>(sV, v_ptr(c + 1), a.v_k0);
        }
    }
    cp_async_wait<0>();
    auto finish = [&](int m, cf sum) {       // out = x - eta * sum of row m
        const long long e = x_off + m * row_stride;
        const cf xv = a.x ? load_image(a.x, e, a.x_planar, id.b, a.plane) : make_float2(0.f, 0.f);
        store_image(a.out, e, make_float2(fmaf(-a.eta, sum.x, xv.x), fmaf(-a.eta, sum.y, xv.y)), a.out_planar, id.b, a.plane);
    };
    if (a.csplit > 1) {
        // The partial coil sums of the cluster's blocks, added in block order; the blocks share the rows.  All loads of a
        // row are requested before the first is used (one after another they took 10 us).
        __syncthreads();
        if (col) {
#pragma unroll
            for (int m = 0; m < RY; ++m) sT[m * NZ + tid] = acc[m];
        }
        cluster_arrive_wait();
        if (col) {
#pragma unroll 2
            for (int m = (int)id.part; m < RY; m += a.csplit) {
                cf t[MAX_CSPLIT];
#pragma unroll
                for (int p = 0; p < MAX_CSPLIT; ++p) t[p] = (p < a.csplit) ? cluster_load(sT + m * NZ + tid, (unsigned)p) : make_float2(0.f, 0.f);
                cf sum = t[0];
#pragma unroll
                for (int p = 1; p < MAX_CSPLIT; ++p) sum = cadd(sum, t[p]);
                finish(m, sum);
            }
        }
        cluster_arrive_wait();           // no block leaves while its sums are being read
        return;
    }
    if (!col) return;
    cf xv[RY];
#pragma unroll
    for (int m = 0; m < RY; ++m) xv[m] = a.x ? load_image(a.x, x_off + m * row_stride, a.x_planar, id.b, a.plane) : make_float2(0.f, 0.f);
#pragma unroll
    for (int m = 0; m < RY; ++m)
        store_image(a.out, x_off + m * row_stride, make_float2(fmaf(-a.eta, acc[m].x, xv[m].x), fmaf(-a.eta, acc[m].y, xv[m].y)), a.out_planar, id.b, a.plane);
}

}  // namespace gleam
