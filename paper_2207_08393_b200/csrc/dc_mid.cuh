// Pass 2 of the row-tile scheme (dc_tile.cuh): radix-BY transform over the rows j of one k0 group, the k-space work
// of the call, and the mirror image back, in place on the workspace.  One thread per kz column, the BY values in
// registers, no exchange through shared memory.  Bound by HBM: 16 bytes per element, 10 log2 BY + 12 flop.
#pragma once
#include "dc_tile.cuh"

namespace gleam {

enum MidMode {
    MID_SEP = 0,     // no measurements (VJP, normal-equations form): readout-invariant mask, or 2-D problem with an arbitrary one
    MID_SEP_Z = 1,   // readout-invariant mask and the table z of the measurements
    MID_ADJ_Z = 2,   // A^H y: minus the table z alone, nothing is read from the workspace
    MID_FULL = 3,    // 2-D problem with an arbitrary mask and measurements
    MID_ADJ_FULL = 4,
    MID_FWD = 5,     // forward half alone (arbitrary 3-D masks: the readout axis follows)
    MID_INV = 6,     // inverse half alone
    MID_GRADY = 7    // forward half and the mask, written to k-space: last step of the forward operator A, 2-D
};

struct MidArgs {
    cf* V; long long v_unit, v_slab, v_k0, v_j;
    const float* mask;                        // MID_SEP*: (B,T,N1,NZ); MID_FULL*, MID_GRADY: (B,T,N1,NZ) or (B,T,NZ)
    int mask_row;                             // MID_GRADY: the mask has one row per (b,t)
    const cf* zin; const int* zidx;           // compact z table; ranks inside the k0 group, -1 where nothing was sampled
    const float* m2c; const int* zstart;      // squared mask weights by rank, times scale2; (B,T,33) first rank of each k0 group
    const cf* y; cf* ky_out;
    float scale, scale2;                      // g / sqrt(N1 NZ) (times eta: MID_GRADY), 1 / (N1 NZ)
    int C, T, n0, G, i0_start, NZ, zcap;
    long long nunits;                         // B*C*T
};

// The kernel streams: what matters is how many columns are in flight, so the register bound leaves little beyond the
// column itself (a prime radix also holds its sums and differences) and everything else the k-space work needs is
// fetched late or staged in shared memory.  Without the bound the compiler keeps mask weights and addresses of the
// whole column: 100 registers, 2 blocks per SM, 907 us for the middle pass of a 320 x 320 x 256 volume with 8 coils
// instead of 510 us.
template <int BY> constexpr int mid_blocks() {
    constexpr bool prime = BY > 4 && smallest_odd_factor(BY) == BY && BY % 2 == 1;
    constexpr int regs = ((prime ? 4 : 2) * BY + 24 + 7) / 8 * 8;
    return cmin(8, cmax(1, 65536 / (256 * regs)));
}

template <int RY, int BY, int MODE>
__global__ void __launch_bounds__(256, mid_blocks<BY>())
mid_kernel(const MidArgs a) {
    grid_dependency_wait();
    constexpr int N1 = RY * BY;
    constexpr bool FORWARD = MODE != MID_INV && MODE != MID_ADJ_Z && MODE != MID_ADJ_FULL;
    constexpr bool INVERSE = MODE != MID_FWD && MODE != MID_GRADY;
    constexpr bool Z = MODE == MID_SEP_Z || MODE == MID_ADJ_Z;
    constexpr bool FULL = MODE == MID_FULL || MODE == MID_ADJ_FULL;
    const int NZ = a.NZ;
    const int kz = blockIdx.y * blockDim.x + threadIdx.x;          // gridDim.y covers NZ
    const bool col_ok = kz < NZ;
    const unsigned blk = blockIdx.x;                               // (unit, gi, k0)
    const int k0 = (int)(blk % RY);
    const unsigned gi = (blk / RY) % (unsigned)a.G;
    const unsigned unit = blk / (RY * (unsigned)a.G);
    const unsigned bc = unit / (unsigned)a.T;
    const int t = (int)(unit - bc * (unsigned)a.T);
    const int b = (int)(bc / (unsigned)a.C);
    const long long bt = (long long)b * a.T + t;
    const long long pe = (long long)N1 * NZ;
    cf* Vp = a.V + unit * a.v_unit + gi * a.v_slab + k0 * a.v_k0 + kz;
    __shared__ cf s_tw[BY];                                        // w_N1^(j k0)
    if ((int)threadIdx.x < BY) s_tw[threadIdx.x] = unit_root_fwd<N1>(((int)threadIdx.x * k0) % N1);
    // Each half of the kernel reads the twiddles for itself (volatile: a value kept from the first half to the second
    // would cost 2 BY registers).
    const unsigned tw_addr = (unsigned)__cvta_generic_to_shared(s_tw);
    auto twiddle = [&](int j) -> cf {
        cf w;
        asm volatile("ld.volatile.shared.v2.f32 {%0, %1}, [%2];" : "=f"(w.x), "=f"(w.y) : "r"(tw_addr + 8u * j));
        return w;
    };

    // The z values of this block's ky group are contiguous in the compact table (ranks zstart[k0] .. zstart[k0+1]);
    // they are staged in shared memory while the transform runs, with their mask weights.  The slots before the first hold
    // zeros for the unsampled entries (rank -1), which keeps the update free of branches and of index arithmetic.  Ranks inside
    // the group and weights that are scaled already, against ranks of the whole plane: prepared step of 8 coils of 160 x 320 x 256
    // 927 -> 901 us, of 96 x 160 x 128 at 4x 162 -> 157; value and weight in one 16-byte slot 984 (a wavefront more per entry).
    // The test for a staged group lies outside the loop over the entries (6 coils of 64 x 368 x 320 at 3x, whose groups are
    // larger than the staging area: 732 -> 498).
    extern __shared__ __align__(16) float2 mid_smem[];
    cf* s_z = reinterpret_cast<cf*>(reinterpret_cast<float*>(mid_smem) + BY * blockDim.x) + 1;      // behind the slots of the threads
    float* s_w = reinterpret_cast<float*>(s_z + a.zcap) + 1;
    int z_first = 0;
    bool z_staged = false;
    if (Z) {
        z_first = a.zstart[bt * 33 + k0];
        const int nz = a.zstart[bt * 33 + k0 + 1] - z_first;
        z_staged = nz <= a.zcap;
        if (z_staged) {
            const cf* zsrc = a.zin + ((long long)unit * a.n0 + a.i0_start + (int)gi) * pe + z_first;
            const float* wsrc = a.m2c + bt * pe + z_first;
            for (int e = threadIdx.x; e < nz; e += blockDim.x) {
                cp_async8(&s_z[e], zsrc + e);
                if (MODE == MID_SEP_Z) cp_async4(&s_w[e], wsrc + e);
            }
            cp_async_commit();
            if (threadIdx.x == 0) { s_z[-1] = make_float2(0.f, 0.f); s_w[-1] = 0.f; }
        }
    }
    // What the k-space work of this column needs is copied to shared memory while the transform runs, into slots of the
    // thread's own: mask weights (MID_SEP), ranks among the sampled positions (with z), weights and measurements
    // (arbitrary mask; measurements at unsampled positions are not read, they may hold anything).
    const int s2 = shift_half(kz, NZ);
    const int TH = blockDim.x;
    float* s_m = reinterpret_cast<float*>(mid_smem) + threadIdx.x;
    cf* s_y = reinterpret_cast<cf*>(reinterpret_cast<float*>(mid_smem) + BY * TH) + threadIdx.x;
    // centred ky of the raw index k0 + RY k1; an even BY turns the half shift into a rotation of k1
    auto centred = [&](int k1) { return BY % 2 == 0 ? k0 + RY * ((k1 + BY / 2) % BY) : shift_half(k0 + RY * k1, N1); };
    if (MODE == MID_SEP && col_ok) {
        const float* mk = a.mask + bt * pe + s2;
#pragma unroll
        for (int k1 = 0; k1 < BY; ++k1) cp_async4(s_m + k1 * TH, mk + centred(k1) * NZ);
        cp_async_commit();
    }
    if (Z && col_ok) {
        const int* zi = a.zidx + bt * pe + (long long)k0 * NZ + kz;
#pragma unroll
        for (int k1 = 0; k1 < BY; ++k1) cp_async4(s_m + k1 * TH, zi + RY * k1 * NZ);
        cp_async_commit();
    }
    cf c[BY];
    if (col_ok && (FORWARD || MODE == MID_INV)) {
        const cf* p = Vp;
#pragma unroll
        for (int j = 0; j < BY; ++j) { c[j] = *p; p += a.v_j; }
    }
    if (FULL && col_ok) {
        const float* mk = a.mask + bt * pe + s2;
        const cf* yy = a.y + (long long)unit * pe + s2;
#pragma unroll
        for (int k1 = 0; k1 < BY; ++k1) {
            const int off = centred(k1) * NZ;
            const float m = mk[off];
            s_m[k1 * TH] = m;
            if (m != 0.f) cp_async8(s_y + k1 * TH, yy + off);
        }
        cp_async_commit();
    }
    cp_async_wait<0>();
    __syncthreads();
    if (!col_ok) return;
    if (FORWARD) {
        if (RY > 1) {
#pragma unroll
            for (int j = 1; j < BY; ++j) c[j] = cmul(c[j], twiddle(j));
        }
        Dft<BY, -1, true>::run(c);
    }
    if (MODE == MID_SEP) {
#pragma unroll
        for (int k1 = 0; k1 < BY; ++k1) { const float m = s_m[k1 * TH]; c[k1] = cscale(c[k1], m * m * a.scale2); }
    } else if (Z) {
        const int* zi = reinterpret_cast<const int*>(s_m);
        const cf* zz = a.zin + ((long long)unit * a.n0 + a.i0_start + (int)gi) * pe + z_first;
        const float* m2 = a.m2c + bt * pe + z_first;
        auto update = [&](int k1, float zx, float zy, float w) {
            if (MODE == MID_SEP_Z) c[k1] = make_float2(fmaf(w, c[k1].x, -zx), fmaf(w, c[k1].y, -zy));
            else c[k1] = make_float2(-zx, -zy);
        };
        if (z_staged) {
#pragma unroll
            for (int k1 = 0; k1 < BY; ++k1) {
                const int r = zi[k1 * TH];
                const cf zv = s_z[r];
                update(k1, zv.x, zv.y, MODE == MID_SEP_Z ? s_w[r] : 0.f);
            }
        } else {                                                    // more sampled entries than the staging area holds
#pragma unroll
            for (int k1 = 0; k1 < BY; ++k1) {
                const int r = zi[k1 * TH];
                const cf zv = (r >= 0) ? zz[r] : make_float2(0.f, 0.f);
                update(k1, zv.x, zv.y, (MODE == MID_SEP_Z && r >= 0) ? m2[r] : 0.f);
            }
        }
    } else if (FULL) {
#pragma unroll
        for (int k1 = 0; k1 < BY; ++k1) {
            const float m = s_m[k1 * TH], w = m * m * a.scale2;
            const cf yv = (m != 0.f) ? s_y[k1 * TH] : make_float2(0.f, 0.f);
            const float f = (((centred(k1) + s2) & 1) ? -a.scale : a.scale) * m;
            if (MODE == MID_FULL) c[k1] = make_float2(fmaf(w, c[k1].x, -f * yv.x), fmaf(w, c[k1].y, -f * yv.y));
            else c[k1] = make_float2(-f * yv.x, -f * yv.y);
        }
    } else if (MODE == MID_GRADY) {
        const float* mk = a.mask + bt * (a.mask_row ? NZ : pe) + s2;
        cf* dst = a.ky_out + (long long)unit * pe + s2;
#pragma unroll
        for (int k1 = 0; k1 < BY; ++k1) {
            const int s1 = centred(k1);
            dst[s1 * NZ] = cscale(c[k1], (((s1 + s2) & 1) ? -a.scale : a.scale) * mk[a.mask_row ? 0 : s1 * NZ]);
        }
        return;
    }
    if (INVERSE) {
        Dft<BY, +1, true>::run(c);
        if (RY > 1) {
#pragma unroll
            for (int j = 1; j < BY; ++j) c[j] = cmulc(c[j], twiddle(j));
        }
    }
    cf* p = Vp;
#pragma unroll
    for (int j = 0; j < BY; ++j) { *p = c[j]; p += a.v_j; }
}

// ---------------------------------------------------------------------------------------------
// launch tables: passes 1 and 3 per (RY, kz plan), pass 2 per ky length
// ---------------------------------------------------------------------------------------------
struct TileOps {
    int ry, n2;
    // images: B*T; tiles: tiles of the whole problem (they decide how the coils are split, so that a volume gives the
    // same bits whatever part of it one launch covers)
    cudaError_t (*fwd)(const TileArgs&, long long images, long long tiles, cudaStream_t);
    cudaError_t (*inv)(const TileArgs&, long long images, long long tiles, cudaStream_t);
};
struct MidOps {
    int n1, ry, by;
    cudaError_t (*launch)(int mode, const MidArgs&, cudaStream_t);
};

// Blocks that share the coils of a tile: doubled while that leaves no more than 640 threads per SM.  Splitting only
// fills SMs that would be idle (a 160 x 160 slice with 16 coils, 16 tiles: 47 us per VJP call unsplit, 33 / 25 / 21 us
// for 2 / 4 / 8 blocks a tile); beyond that the start-up of the additional blocks costs more than the finer grain gains
// (limits of 512 / 640 / 768 / 1024 threads: 2 x 16 coils of 640 x 320 109 / 94 / 94 / 94 us, 5 coils of 24 x 128 x 128
// 37 / 37 / 43 / 43 us, 9 coils of 320 x 48 x 24 49 / 49 / 49 / 64 us).
inline int coil_split(long long tiles, int threads, int sms, int C) {
    int cs = 1;
    while (cs < MAX_CSPLIT && 2 * cs <= C && 2 * cs * tiles * threads <= 640LL * sms) cs *= 2;
    return cs;
}

template <class PZ, int RY>
struct TileImpl {
    using TL = Tile<PZ, RY>;
    using LL = Tile<PZ, RY, true>;
    static cudaError_t fwd(const TileArgs& a, long long images, long long tiles, cudaStream_t s) {
        if constexpr (TL::TWO_FWD) return launch_either<tile_fwd_kernel<PZ, RY>, tile_fwd_kernel<PZ, RY, true>>(TL::FWD_BYTES, LL::FWD_BYTES, false, a, images, tiles, s);
        else return launch<tile_fwd_kernel<PZ, RY>>(TL::FWD_BYTES, false, a, images, tiles, s);
    }
    static cudaError_t inv(const TileArgs& a, long long images, long long tiles, cudaStream_t s) {
        if constexpr (TL::TWO_INV) return launch_either<tile_inv_kernel<PZ, RY>, tile_inv_kernel<PZ, RY, true>>(TL::INV_BYTES, LL::INV_BYTES, true, a, images, tiles, s);
        else return launch<tile_inv_kernel<PZ, RY>>(TL::INV_BYTES, true, a, images, tiles, s);
    }

private:
    static cudaError_t count_blocks(const TileArgs& a, long long images, long long tiles, int* csplit, long long* blocks) {
        int sms = 0;
        const cudaError_t e = device_sms(&sms);
        if (e != cudaSuccess) return e;
        *csplit = coil_split(tiles, TL::TH, sms, a.C);
        *blocks = images * a.G * a.BY * *csplit;
        return cudaSuccess;
    }
    template <auto KERNEL> static cudaError_t resident(size_t bytes, int* slots) {
        static PerDevice done, cache;
        const cudaError_t e = ensure_smem(KERNEL, bytes, done);
        return e != cudaSuccess ? e : resident_slots(KERNEL, TL::TH, bytes, cache, slots);
    }
    // The form with more blocks on an SM pays for its spills, or its twiddles in shared memory, where it saves a round of blocks.  VJP, us,
    // loose / dense: 5 coils of 32 x 46 x 184 (736 blocks, two rounds of either) 32.6 / 36.0, 12 of 12 slices of 92 x 184 (276 blocks,
    // one round) 37.0 / 41.4; 8 coils of 128 x 92 x 184 283 / 234.
    template <auto DENSE, auto LOOSE>
    static cudaError_t launch_either(size_t dense_bytes, size_t loose_bytes, bool cluster, const TileArgs& a, long long images, long long tiles, cudaStream_t s) {
        int csplit = 1, dense = 1, loose = 1;
        long long blocks = 0;
        cudaError_t e;
        if ((e = count_blocks(a, images, tiles, &csplit, &blocks)) != cudaSuccess) return e;
        if ((e = resident<DENSE>(dense_bytes, &dense)) != cudaSuccess || (e = resident<LOOSE>(loose_bytes, &loose)) != cudaSuccess) return e;
        if ((blocks + dense - 1) / dense < (blocks + loose - 1) / loose) return launch<DENSE>(dense_bytes, cluster, a, images, tiles, s);
        return launch<LOOSE>(loose_bytes, cluster, a, images, tiles, s);
    }
    // cluster: the blocks that share a tile form one
    template <auto KERNEL>
    static cudaError_t launch(size_t bytes, bool cluster, const TileArgs& a0, long long images, long long tiles, cudaStream_t s) {
        static PerDevice done;
        cudaError_t e = ensure_smem(KERNEL, bytes, done);
        if (e != cudaSuccess) return e;
        TileArgs a = a0;
        long long blocks = 0;
        if ((e = count_blocks(a, images, tiles, &a.csplit, &blocks)) != cudaSuccess) return e;
        if (blocks <= 0) return cudaSuccess;
        if (blocks > 2147483647LL) return cudaErrorInvalidConfiguration;
        if (cluster) return launch_overlapped_cluster((unsigned)a.csplit, KERNEL, dim3((unsigned)blocks), dim3(TL::TH), bytes, s, a);
        return launch_overlapped(true, KERNEL, dim3((unsigned)blocks), dim3(TL::TH), bytes, s, a);
    }
};

template <int RY, int BY>
struct MidImpl {
    static constexpr int ZCAP = 2048;          // z values of one k0 group that are staged
    template <int MODE> static cudaError_t go(const MidArgs& a0, cudaStream_t s) {
        MidArgs a = a0;
        const int parts = (a.NZ + 255) / 256, threads = ((a.NZ + parts - 1) / parts + 31) / 32 * 32;   // equal shares of a row
        const long long blocks = a.nunits * a.G * RY;
        if (blocks <= 0) return cudaSuccess;
        if (blocks > 2147483647LL) return cudaErrorInvalidConfiguration;
        // shared memory: a weight or rank per element, and the measurements (arbitrary mask) or the z values and
        // weights of one k0 group
        constexpr bool Z = MODE == MID_SEP_Z || MODE == MID_ADJ_Z, FULL = MODE == MID_FULL || MODE == MID_ADJ_FULL;
        size_t bytes = (Z || FULL || MODE == MID_SEP) ? (size_t)BY * threads * sizeof(float) : 0;
        if (FULL) {
            static PerDevice done;
            cudaError_t e = ensure_smem(mid_kernel<RY, BY, MODE>, BY * 256 * (sizeof(cf) + sizeof(float)), done, BY * sizeof(cf));
            if (e != cudaSuccess) return e;
            bytes += (size_t)BY * threads * sizeof(cf);
        }
        if (Z) {
            a.zcap = BY * a.NZ < ZCAP ? BY * a.NZ : ZCAP;
            bytes += (size_t)(a.zcap + 1) * (sizeof(cf) + sizeof(float));
        }
        if (Z) {
            static PerDevice done;
            cudaError_t e = ensure_smem(mid_kernel<RY, BY, MODE>, BY * 256 * sizeof(float) + (ZCAP + 1) * 12, done, BY * sizeof(cf));
            if (e != cudaSuccess) return e;
        }
        return launch_overlapped(true, mid_kernel<RY, BY, MODE>, dim3((unsigned)blocks, (unsigned)parts), dim3(threads), bytes, s, a);
    }
    static cudaError_t launch(int mode, const MidArgs& a, cudaStream_t s) {
        switch (mode) {
            case MID_SEP: return go<MID_SEP>(a, s);
            case MID_SEP_Z: return go<MID_SEP_Z>(a, s);
            case MID_ADJ_Z: return go<MID_ADJ_Z>(a, s);
            case MID_FULL: return go<MID_FULL>(a, s);
            case MID_ADJ_FULL: return go<MID_ADJ_FULL>(a, s);
            case MID_FWD: return go<MID_FWD>(a, s);
            case MID_INV: return go<MID_INV>(a, s);
            case MID_GRADY: return go<MID_GRADY>(a, s);
        }
        return cudaErrorInvalidValue;
    }
};

}  // namespace gleam
