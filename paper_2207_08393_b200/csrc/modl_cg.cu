// MoDL data-consistency step (Eq. 7, second line):  out = (A^H A + mu I)^{-1} (A^H y + mu z)
// by a fixed number of conjugate-gradient steps, and its vector-Jacobian product with respect to z.
//
// The normal operator is the data-consistency VJP path of this library with eta = -1/mu:
//     q = p + (1/mu) A^H A p = H p / mu,          H = A^H A + mu I,
// so the factor mu moves into the scalars (alpha = <r,r> / (mu <p,q>),  r -= alpha mu q) and no
// operator kernel changes.  What remains are image-sized vector updates with inner products per batch example:
//
//     cg_init : b = A^H y + mu z  (VJP: b = mu g);  r = p = b;  x = 0;  partial sums of <b,b>
//     cg_dot  : partial sums of Re <p,q> and <q,q>
//     cg_step : alpha = rr / (mu pq);  x += alpha p;  r -= alpha mu q;  beta = rr' / rr;  p = r + beta p;
//               partial sums of <r,r>;  the last step only updates x
//
// Where the operator is a one-pass 2-D kernel, that kernel also stores Re<p_row, q_row> and <q_row, q_row> of every
// image row it writes (it holds both in registers at its update step) and cg_dot is not launched.
//
// One launch per step: the norm of the new residual follows from sums that are known before it exists,
//     rr' = <r,r> - 2 alpha mu <r,q> + (alpha mu)^2 <q,q>,        <r,q> = <p,q> - beta_old <p_old,q>,
// and the direction is updated in the pass that forms the residual.  <p_old,q> is zero for exactly conjugate directions, but
// not for steps that were rounded to 32 bits (beta first of all).  H is Hermitian, so it is
//     <q_old,p> = <q_old,r> + beta_old <q_old,p_old>,
// and the same identity for the step before, now with the norm that was summed, gives <q_old,r> = (rr_old - (alpha mu)^2
// <q_old,q_old> - rr) / (2 alpha mu): four scalars of the step before (CgCarry) and no further sum.  Without that term the
// error of beta grows with the condition number (against 64 bits, 10 steps: 20 frames of 192 x 160 with mu = 1e-3 9.5e-7,
// with it 1.9e-7, as with a norm that is summed first).  Only beta takes this value: alpha is built from the sum <r,r> of
// the residual itself, so every step minimises along its direction whatever rounding does to beta.  Bound by launches and
// L2: 20 frames of 192 x 160, solve and VJP with 10 steps: 664 -> 567 us (40 vector launches -> 22, started while the
// operator drains).
//
// Inner products: every thread accumulates in double precision, a block reduces in a fixed order
// and stores one partial sum; the kernel that needs the scalar adds the partial sums of its example
// in a fixed order at its start (every block the same sum).  Producer and consumer are different
// launches on one stream: no atomics, no fences, no block waits for another one, and the result
// does not depend on the order in which blocks run.  <r,r> and the carried scalars alternate between two
// arrays (step parity): cg_step reads one and writes the other.
#include "dc_entry.h"
#include "launch_overlap.cuh"

#include <cmath>
#include <cstdint>
#include <type_traits>

namespace gleam {

constexpr int CG_THREADS = 256;
constexpr int CG_MAX_BLOCKS = 592;          // partial sums per example (4 blocks per SM on 148 SMs)

// What a step leaves for the next one's <p_old,q>: rr - (alpha mu)^2 <q,q>, 1 / (2 alpha mu), beta, <p,q>
// (alpha mu as the residual took it).
struct CgCarry { double u, v, beta, pq; };

struct CgArgs {
    const float4* z;         // z (forward) or grad_out (VJP), two complex values per element
    const float4* q;         // A^H y at cg_init, H p / mu afterwards
    float4* r; float4* p; float4* x;
    double* part_rr;         // (2, B, CG_MAX_BLOCKS): <r,r> partial sums of even / odd steps
    CgCarry* carry;          // (2, B), even / odd steps
    double* part_pq;         // (B, CG_MAX_BLOCKS) twice: <p,q> and <q,q> partial sums written by cg_dot
    const double* dot_rows;  // (B, rows_per_example) twice: Re<p,q> and <q,q> per image row or block from the operator, or null
    int rows_per_example, dot_count;         // dot_count of them are in use
    long long ne2;           // float4 elements per example
    float mu;
    double inv_mu;
    int parity;              // step k & 1: part_rr[parity] holds <r_k, r_k>
};

// Sums of three values over the block in a fixed order, in the threads of the first warp.  64-bit arithmetic runs at a
// fraction of the 32-bit rate, so what is the same for all threads is left to one warp (20 frames of 192 x 160, solve and
// VJP with 10 steps: 584 -> 567 us).
struct Sums { double a, b, c; };
__device__ __forceinline__ Sums block_sums(Sums v) {
    __shared__ Sums warp_sum[CG_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        v.a += __shfl_down_sync(0xffffffffu, v.a, o); v.b += __shfl_down_sync(0xffffffffu, v.b, o); v.c += __shfl_down_sync(0xffffffffu, v.c, o);
    }
    __syncthreads();                                    // earlier readers of warp_sum are done
    if (lane == 0) warp_sum[warp] = v;
    __syncthreads();
    Sums t{0.0, 0.0, 0.0};
    if (warp == 0) {
#pragma unroll
        for (int w = 0; w < CG_THREADS / 32; ++w) { t.a += warp_sum[w].a; t.b += warp_sum[w].b; t.c += warp_sum[w].c; }
    }
    return t;
}

// This thread's share of the sum of n values written by an earlier launch, in a fixed order, as thread `first` of `threads`;
// v is 16-byte aligned.  Eight pairs are requested at a time: 20 frames of 192 rows are one round of loads of a block.
__device__ __forceinline__ double array_share(const double* v, int n, int first, int threads) {
    double t = 0.0;
    const int pairs = n / 2;
    for (int i0 = first; i0 < pairs; i0 += 8 * threads) {
        double2 w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) w[e] = (i0 + e * threads < pairs) ? __ldcg(reinterpret_cast<const double2*>(v) + i0 + e * threads) : make_double2(0.0, 0.0);
#pragma unroll
        for (int e = 0; e < 8; ++e) t += w[e].x + w[e].y;
    }
    if (n % 2 && first == 0) t += __ldcg(v + n - 1);
    return t;
}
// Sums of the arrays a (na values), b and c (nb values each; c may be null), valid in the first thread.  Short arrays are
// dealt to the warps, so that a warp has one value to add across its lanes (6 coils of 320 x 320, 10 steps: 117 -> 110 us);
// long ones take every thread (10 frames of 192 rows: 306 -> 298).
constexpr int CG_DEALT = 768;
__device__ __forceinline__ Sums array_sums(const double* a, int na, const double* b, const double* c, int nb) {
    constexpr int W = CG_THREADS / 32, WA = 2, WB = (W - WA) / 2;           // warps of a, of b and of c
    __shared__ double warp_sum[W];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int which = warp < WA ? 0 : warp < WA + WB ? 1 : 2, first = which == 0 ? 0 : which == 1 ? WA : WA + WB;
    const double* v = which == 0 ? a : which == 1 ? b : c;
    double t = v == nullptr ? 0.0 : array_share(v, which == 0 ? na : nb, (warp - first) * 32 + lane, (which == 0 ? WA : WB) * 32);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) warp_sum[warp] = t;
    __syncthreads();
    Sums s{0.0, 0.0, 0.0};
    if (threadIdx.x == 0) {
        for (int w = 0; w < WA; ++w) s.a += warp_sum[w];
        for (int w = WA; w < WA + WB; ++w) s.b += warp_sum[w];
        for (int w = WA + WB; w < W; ++w) s.c += warp_sum[w];
    }
    return s;
}

__device__ __forceinline__ double* rr_slot(const CgArgs& a, int which) {
    return a.part_rr + ((size_t)which * gridDim.y + blockIdx.y) * CG_MAX_BLOCKS;
}

__device__ __forceinline__ double norm2(float4 v) {
    return (double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z + (double)v.w * v.w;
}
__device__ __forceinline__ double dot4(float4 p, float4 q) {
    return (double)p.x * q.x + (double)p.y * q.y + (double)p.z * q.z + (double)p.w * q.w;
}
// y + c * x
__device__ __forceinline__ float4 axpy4(float c, float4 x, float4 y) {
    return make_float4(fmaf(c, x.x, y.x), fmaf(c, x.y, y.y), fmaf(c, x.z, y.z), fmaf(c, x.w, y.w));
}

template <bool HAS_Q>
__global__ void __launch_bounds__(CG_THREADS) cg_init_kernel(const CgArgs a) {
    grid_dependency_wait();
    const long long base = (long long)blockIdx.y * a.ne2;
    double acc = 0.0;
    for (long long i = (long long)blockIdx.x * CG_THREADS + threadIdx.x; i < a.ne2; i += (long long)gridDim.x * CG_THREADS) {
        const float4 zv = a.z[base + i];
        float4 b = make_float4(a.mu * zv.x, a.mu * zv.y, a.mu * zv.z, a.mu * zv.w);
        if (HAS_Q) b = axpy4(a.mu, zv, a.q[base + i]);
        a.r[base + i] = b;
        a.p[base + i] = b;
        a.x[base + i] = make_float4(0.f, 0.f, 0.f, 0.f);
        acc += norm2(b);
    }
    const Sums t = block_sums(Sums{acc, 0.0, 0.0});
    if (threadIdx.x == 0) rr_slot(a, 0)[blockIdx.x] = t.a;
    if (threadIdx.x == 0 && blockIdx.x == 0) a.carry[blockIdx.y] = CgCarry{0.0, 0.0, 0.0, 0.0};      // p = r
}

__global__ void __launch_bounds__(CG_THREADS) cg_dot_kernel(const CgArgs a) {
    grid_dependency_wait();
    const long long base = (long long)blockIdx.y * a.ne2;
    Sums acc{0.0, 0.0, 0.0};
    for (long long i = (long long)blockIdx.x * CG_THREADS + threadIdx.x; i < a.ne2; i += (long long)gridDim.x * CG_THREADS) {
        const float4 pv = a.p[base + i], qv = a.q[base + i];
        acc.a += dot4(pv, qv);
        acc.b += norm2(qv);
    }
    acc = block_sums(acc);
    if (threadIdx.x == 0) {
        double* part = a.part_pq + (size_t)blockIdx.y * CG_MAX_BLOCKS + blockIdx.x;
        part[0] = acc.a;
        part[(size_t)gridDim.y * CG_MAX_BLOCKS] = acc.b;
    }
}

// BATCH elements of every vector are requested before the sums are formed, so that their latency covers that of the sums.
// The bounds (four, three and two blocks on an SM) make the forms that are not the last step and request two or three elements spill 32 to
// 96 B, two with sums per row also in the last step (8 B); four elements fit their 128 registers.
template <bool FROM_ROWS, bool DEALT, bool LAST, int BATCH>
__global__ void __launch_bounds__(CG_THREADS, BATCH == 2 ? 4 : BATCH == 3 ? 3 : 2) cg_step_kernel(const CgArgs a) {
    grid_dependency_wait();
    const long long base = (long long)blockIdx.y * a.ne2, stride = (long long)gridDim.x * CG_THREADS;
    long long i = (long long)blockIdx.x * CG_THREADS + threadIdx.x;
    float4 pv[BATCH], xv[BATCH], qv[LAST ? 1 : BATCH], rv[LAST ? 1 : BATCH];
    auto fetch = [&]() {
#pragma unroll
        for (int e = 0; e < BATCH; ++e) {
            const long long at = base + i + e * stride;
            if (i + e * stride >= a.ne2) break;
            pv[e] = a.p[at]; xv[e] = a.x[at];
            if (!LAST) { qv[e] = a.q[at]; rv[e] = a.r[at]; }
        }
    };
    fetch();
    __shared__ double carry[4];              // CgCarry of the step before
    if (!LAST && threadIdx.x < 4) carry[threadIdx.x] = __ldcg(reinterpret_cast<const double*>(a.carry + (size_t)a.parity * gridDim.y + blockIdx.y) + threadIdx.x);
    const double* pq = FROM_ROWS ? a.dot_rows + (size_t)blockIdx.y * a.rows_per_example : a.part_pq + (size_t)blockIdx.y * CG_MAX_BLOCKS;
    const int npq = FROM_ROWS ? a.dot_count : (int)gridDim.x;
    const double* qq = pq + (size_t)gridDim.y * (FROM_ROWS ? a.rows_per_example : CG_MAX_BLOCKS);
    Sums s;
    if (DEALT) {
        s = array_sums(rr_slot(a, a.parity), (int)gridDim.x, pq, LAST ? nullptr : qq, npq);
    } else {
        s.a = array_share(rr_slot(a, a.parity), (int)gridDim.x, threadIdx.x, CG_THREADS);
        s.b = array_share(pq, npq, threadIdx.x, CG_THREADS);
        s.c = LAST ? 0.0 : array_share(qq, npq, threadIdx.x, CG_THREADS);
        s = block_sums(s);
    }
    __shared__ float scalars[3];
    if (threadIdx.x == 0) {
        // an example whose residual is exactly zero stays as it is; one division on the way to the vectors
        const bool live = s.a > 0.0 && s.b > 0.0;
        const double inv = 1.0 / s.b, amu = live ? s.a * inv : 0.0;
        const float cf_ = (float)-amu;
        float beta = 0.f;
        if (!LAST) {
            const CgCarry c{carry[0], carry[1], carry[2], carry[3]};
            const double old = c.beta * ((c.u - s.a) * c.v + c.beta * c.pq);        // beta_old <p_old,q>
            const double ratio = amu * s.c * inv - 1.0 + 2.0 * old * inv;           // rr' / rr
            if (live && ratio > 0.0) beta = (float)ratio;
        }
        scalars[0] = (float)(amu * a.inv_mu); scalars[1] = cf_; scalars[2] = beta;
    }
    __syncthreads();
    const float af = scalars[0], cf_ = scalars[1], beta = scalars[2];
    double acc = 0.0;
    while (i < a.ne2) {
#pragma unroll
        for (int e = 0; e < BATCH; ++e) {
            const long long at = base + i + e * stride;
            if (i + e * stride >= a.ne2) break;
            a.x[at] = axpy4(af, pv[e], xv[e]);
            if (!LAST) {
                const float4 r = axpy4(cf_, qv[e], rv[e]);
                a.r[at] = r;
                a.p[at] = axpy4(beta, pv[e], r);
                acc += norm2(r);
            }
        }
        i += BATCH * stride;
        fetch();
    }
    if (LAST) return;
    const Sums t = block_sums(Sums{acc, 0.0, 0.0});
    if (threadIdx.x == 0) rr_slot(a, a.parity ^ 1)[blockIdx.x] = t.a;
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        const double amu = -(double)cf_;
        a.carry[(size_t)(a.parity ^ 1) * gridDim.y + blockIdx.y] = CgCarry{s.a - amu * amu * s.c, amu > 0.0 ? 0.5 / amu : 0.0, (double)beta, s.b};
    }
}

static inline uint64_t up256(uint64_t v) { return (v + 255) / 256 * 256; }

struct CgLayout {
    uint64_t dc_bytes, img_bytes, off_q, off_r, off_p, off_rr, off_carry, off_pq, off_rows, total;
    long long ne2;
    int B;
};

static int cg_layout(const gleam_dims* d, CgLayout* L) {
    if (!d) return GLEAM_ERR_NULL_POINTER;
    uint64_t dc = 0;
    const int rc = gleam_dc_workspace_size(d, &dc);          // validates dims; sized for the forward call
    if (rc != GLEAM_OK) return rc;
    const long long V = (long long)d->n[0] * d->n[1] * d->n[2];
    const long long ne = (long long)d->frames * V;            // complex values per example (even: V is even)
    L->B = d->batch;
    L->ne2 = ne / 2;
    L->dc_bytes = up256(dc);
    L->img_bytes = (uint64_t)d->batch * (uint64_t)ne * 8u;
    uint64_t off = L->dc_bytes;
    L->off_q = off; off = up256(off + L->img_bytes);
    L->off_r = off; off = up256(off + L->img_bytes);
    L->off_p = off; off = up256(off + L->img_bytes);
    L->off_rr = off; off = up256(off + 2u * (uint64_t)d->batch * CG_MAX_BLOCKS * sizeof(double));
    L->off_carry = off; off = up256(off + 2u * (uint64_t)d->batch * sizeof(CgCarry));
    L->off_pq = off; off = up256(off + 2u * (uint64_t)d->batch * CG_MAX_BLOCKS * sizeof(double));
    L->off_rows = off; off = up256(off + 2u * (uint64_t)d->batch * d->frames * d->n[1] * sizeof(double));
    L->total = off;
    return GLEAM_OK;
}

static bool overlap(const void* a, uint64_t na, const void* b, uint64_t nb) {
    const uintptr_t a0 = (uintptr_t)a, b0 = (uintptr_t)b;
    return a0 < b0 + nb && b0 < a0 + na;
}

#define CGCK(call) do { cudaError_t e_ = (call); if (e_ != cudaSuccess) return GLEAM_ERR_CUDA; } while (0)
#define CGRUN(call) do { const int rc_ = (call); if (rc_ != GLEAM_OK) return rc_; } while (0)

// z: image (forward) or cotangent (VJP, y == nullptr)
static int modl_cg(const void* z, const void* y, const void* sens, const float* mask, float mu, int n_iter,
                   void* out, const gleam_dims* d) {
    if (!d || !z || !sens || !mask || !out) return GLEAM_ERR_NULL_POINTER;
    if (!(mu > 0.f) || !std::isfinite(mu) || n_iter < 0 || n_iter > 1000) return GLEAM_ERR_BAD_DIMS;
    CgLayout L;
    CGRUN(cg_layout(d, &L));
    if (!d->workspace) return GLEAM_ERR_NULL_POINTER;
    if (d->workspace_bytes < L.total) return GLEAM_ERR_WORKSPACE_TOO_SMALL;
    if (((uintptr_t)d->workspace & 255) != 0) return GLEAM_ERR_BAD_DIMS;
    if ((((uintptr_t)z) & 15) != 0 || (((uintptr_t)out) & 15) != 0) return GLEAM_ERR_BAD_DIMS;
    CGRUN(check_device_ptr(z));
    CGRUN(check_device_ptr(out));
    CGRUN(check_device_ptr(d->workspace));
    // out may be z itself; nothing else may overlap the output or the workspace
    if (out != z && overlap(out, L.img_bytes, z, L.img_bytes)) return GLEAM_ERR_ALIAS;
    const uint64_t V = (uint64_t)d->n[0] * d->n[1] * d->n[2];
    const uint64_t ksp_bytes = L.img_bytes * (uint64_t)d->coils;
    const uint64_t sens_bytes = (uint64_t)d->batch * d->coils * (d->sens_has_frames ? d->frames : 1) * V * 8u;
    const uint64_t pe = (d->fft_rank == 2) ? (uint64_t)d->n[2] : (uint64_t)d->n[1] * d->n[2];
    const uint64_t mask_bytes = (uint64_t)d->batch * d->frames * (d->mask_kind == GLEAM_MASK_FULL ? V : pe) * 4u;
    if (overlap(d->workspace, L.total, z, L.img_bytes) || overlap(d->workspace, L.total, out, L.img_bytes) ||
        overlap(d->workspace, L.total, sens, sens_bytes) || overlap(d->workspace, L.total, mask, mask_bytes) ||
        (y && overlap(d->workspace, L.total, y, ksp_bytes)))
        return GLEAM_ERR_ALIAS;
    if (overlap(out, L.img_bytes, sens, sens_bytes) || overlap(out, L.img_bytes, mask, mask_bytes) ||
        (y && overlap(out, L.img_bytes, y, ksp_bytes)))
        return GLEAM_ERR_ALIAS;

    cudaStream_t s = (cudaStream_t)d->stream;
    char* ws = (char*)d->workspace;
    gleam_dims dd = *d;
    dd.workspace_bytes = L.dc_bytes;
    CgArgs a{};
    a.z = (const float4*)z; a.q = (const float4*)(ws + L.off_q);
    a.r = (float4*)(ws + L.off_r); a.p = (float4*)(ws + L.off_p); a.x = (float4*)out;
    a.part_rr = (double*)(ws + L.off_rr); a.part_pq = (double*)(ws + L.off_pq);
    a.carry = (CgCarry*)(ws + L.off_carry);
    a.ne2 = L.ne2; a.mu = mu; a.inv_mu = 1.0 / (double)mu; a.parity = 0;
    // the one-pass 2-D operator kernel delivers <p,q> per image row
    const bool from_rows = dot_rows_supported(d);
    double* dot_rows = from_rows ? (double*)(ws + L.off_rows) : nullptr;
    a.dot_rows = dot_rows; a.rows_per_example = d->frames * d->n[1];

    // the operator's own argument checks (y, sens, mask) before anything is enqueued
    DotForm op{};
    CGRUN(run(ws + L.off_r, y, sens, mask, 1.0f, ws + L.off_q, &dd, RUN_ALL, dot_rows, true, 0, nullptr, &op));
    a.dot_count = op.sums;
    // Elements a thread of the vector launches, and how many of them a step requests at once.  All of them where that is one
    // round of resident blocks: a thread that comes back for a few more waits for memory once more after the sums (20 frames of
    // 192 x 160: 4096 of 307,200 elements were left over by 592 blocks of two a thread; 10 steps 240 -> 227 us with three).  Two
    // while the blocks are one per SM, then four (two blocks per SM), three (three) and, beyond that, four in two rounds.
    // Measured against two and four elements in rounds of two, 10 steps: 5 coils of 384 x 640 251 -> 219, of 640 x 320 129 -> 119,
    // 6 x 18 of 384 x 80 220 -> 203, 3 x 5 of 320 x 256 135 -> 125, 8 x 24 x 3 of 64 x 128 203 -> 199; 4 x 4 of 92 x 640 equal (210).
    // Some problems of short vectors lose: 10 x 2 x 7 of 46 x 120 111 -> 114, 32 x 2 x 6 of 32 x 46 174 -> 179.
    // No more than a block per SM: what counts is how the blocks spread over the SMs that an operator of one block per SM gives free (us
    // of 10 steps, two at once / four).  Behind 13 to 16 warps of it nothing fits before they end, and then blocks of 64 registers a
    // thread crowd by fours on the first SMs, of 128 by twos: 36 x 5 coils of 128 x 64 154 / 122, 10 coils x 7 of 512 x 80 195 / 165.
    // Next to 11 or 12 warps one block of 64 registers fits, none of 128, and comes in while the operator drains: 24 x 4 x 8 of 32 x 48
    // 116 / 122, 48 x 6 of 64 x 64 107 / 115, 3 x 5 x 8 of 128 x 96 119 / 128; next to 8 warps two would: 6 coils x 28 of 80 x 128
    // 125 / 119.  Where 12 warps share groups by fours the sums tell: per block two at once (4 coils x 10 of 256 x 80 102 / 111), per
    // row four (38 x 6 of 64 x 96 120 / 115).  12 warps of 32 points take four as well (3 x 4 x 24 of 96 x 32 139 / 112).
    auto blocks_of = [&](int each) { const long long n = (L.ne2 + (long long)CG_THREADS * each - 1) / ((long long)CG_THREADS * each); return n < 1 ? 1 : n; };
    const long long one = CG_MAX_BLOCKS / 4;                 // a block per SM
    const bool sums_per_block = op.sums != a.rows_per_example;
    const bool beside = op.warps == 11 || (op.warps == 12 && d->n[2] >= 48 && (!op.shared || sums_per_block));
    int each = 4, batch = 2;
    if (blocks_of(2) * L.B <= one) each = batch = 2;
    else if (blocks_of(4) * L.B <= 2 * one) batch = (beside && blocks_of(4) * L.B <= one) ? 2 : 4;
    else if (blocks_of(3) * L.B <= 3 * one) each = batch = 3;
    const dim3 grid((unsigned)(blocks_of(each) < CG_MAX_BLOCKS ? blocks_of(each) : CG_MAX_BLOCKS), (unsigned)L.B);
    if (y) {
        CGRUN(run(nullptr, y, sens, mask, 1.0f, ws + L.off_q, &dd, RUN_ADJOINT));
        CGCK(prof_mark(GLEAM_K_CG_VEC, s));
        CGCK(launch_overlapped(true, cg_init_kernel<true>, grid, dim3(CG_THREADS), 0, s, a));
    } else {
        CGCK(prof_mark(GLEAM_K_CG_VEC, s));
        CGCK(launch_overlapped(true, cg_init_kernel<false>, grid, dim3(CG_THREADS), 0, s, a));
    }
    for (int k = 0; k < n_iter; ++k) {
        a.parity = k & 1;
        CGRUN(run(a.p, nullptr, sens, mask, -1.0f / mu, ws + L.off_q, &dd, RUN_ALL, dot_rows));     // q = H p / mu
        const bool last = k + 1 == n_iter;
        if (!from_rows) {
            CGCK(prof_mark(GLEAM_K_CG_VEC, s));
            CGCK(launch_overlapped(true, cg_dot_kernel, grid, dim3(CG_THREADS), 0, s, a));
        }
        CGCK(prof_mark(GLEAM_K_CG_VEC, s));
        auto pick = [&](auto n) {
            constexpr int N = decltype(n)::value;
            return !from_rows ? (last ? cg_step_kernel<false, true, true, N> : cg_step_kernel<false, true, false, N>)
                 : a.dot_count <= CG_DEALT ? (last ? cg_step_kernel<true, true, true, N> : cg_step_kernel<true, true, false, N>)
                                           : (last ? cg_step_kernel<true, false, true, N> : cg_step_kernel<true, false, false, N>);
        };
        auto step = batch == 4 ? pick(std::integral_constant<int, 4>{}) : batch == 3 ? pick(std::integral_constant<int, 3>{}) : pick(std::integral_constant<int, 2>{});
        CGCK(launch_overlapped(true, step, grid, dim3(CG_THREADS), 0, s, a));
        CGCK(cudaGetLastError());
    }
    CGCK(prof_mark(-1, s));
    return GLEAM_OK;
}

}  // namespace gleam

extern "C" {

GLEAM_API int gleam_modl_cg_forward(const void* z, const void* y, const void* sens, const float* mask, float mu,
                                    int32_t n_iter, void* out, const gleam_dims* dims) {
    if (!y) return GLEAM_ERR_NULL_POINTER;
    return gleam::modl_cg(z, y, sens, mask, mu, n_iter, out, dims);
}

GLEAM_API int gleam_modl_cg_vjp(const void* grad_out, const void* sens, const float* mask, float mu,
                                int32_t n_iter, void* grad_z, const gleam_dims* dims) {
    return gleam::modl_cg(grad_out, nullptr, sens, mask, mu, n_iter, grad_z, dims);
}

GLEAM_API int gleam_modl_cg_workspace_size(const gleam_dims* dims, uint64_t* bytes) {
    if (!dims || !bytes) return GLEAM_ERR_NULL_POINTER;
    gleam::CgLayout L;
    const int rc = gleam::cg_layout(dims, &L);
    if (rc != GLEAM_OK) return rc;
    *bytes = L.total;
    return GLEAM_OK;
}

}  // extern "C"
