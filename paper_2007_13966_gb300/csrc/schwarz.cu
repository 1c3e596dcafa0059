// One-level restricted additive Schwarz (Section 3.1) on sm_103a.
//
// The paper's subdomains (one per MPI rank on Tianhe-2) become one CTA each. Inside a
// subdomain the natural-order ILU(0) triangular solves run as a wavefront with the
// working vector in shared memory: over blocks of 2 x 2 cells with FP32 / BF16
// factors, over single cells with FP64 factors (whose arithmetic, not the wavefront's
// latency, bounds them). Factor records are stored in the order of the sweep, so that
// each staged chunk of consecutive levels is one contiguous range, streamed into a
// shared-memory ring with cp.async ahead of the sweep that consumes it.
#include "schwarz.cuh"

#include "recip.cuh"

#include <algorithm>
#include <cstdlib>
#include <map>
#include <tuple>

namespace ras {

// ---------------------------------------------------------------------------
// factor record types
// ---------------------------------------------------------------------------

struct RecF64 { double a, b, c, d; };
struct __align__(16) RecF32 { float a, b, c, d; };
struct __align__(8) RecB16 { __nv_bfloat16 a, b, c, d; };

template <int PREC> struct RecT;
template <> struct RecT<64> { using T = RecF64; using Acc = double; };
template <> struct RecT<32> { using T = RecF32; using Acc = float; };
template <> struct RecT<16> { using T = RecB16; using Acc = float; };

template <int PREC>
__device__ __forceinline__ void store_rec(void *base, long long idx, double a, double b, double c,
                                          double d) {
    if constexpr (PREC == 64) {
        reinterpret_cast<RecF64 *>(base)[idx] = RecF64{a, b, c, d};
    } else if constexpr (PREC == 32) {
        reinterpret_cast<RecF32 *>(base)[idx] = RecF32{(float)a, (float)b, (float)c, (float)d};
    } else {
        // FP64 -> FP32 -> BF16, each round to nearest even
        RecB16 r;
        r.a = __float2bfloat16_rn((float)a);
        r.b = __float2bfloat16_rn((float)b);
        r.c = __float2bfloat16_rn((float)c);
        r.d = __float2bfloat16_rn((float)d);
        reinterpret_cast<RecB16 *>(base)[idx] = r;
    }
}

template <typename Acc, typename R>
__device__ __forceinline__ void load_rec(const unsigned char *p, Acc &a, Acc &b, Acc &c, Acc &d) {
    if constexpr (sizeof(R) == 32) {
        const double2 *q = reinterpret_cast<const double2 *>(p);
        const double2 u = q[0], v = q[1];
        a = u.x; b = u.y; c = v.x; d = v.y;
    } else if constexpr (sizeof(R) == 16) {
        const float4 u = *reinterpret_cast<const float4 *>(p);
        a = u.x; b = u.y; c = u.z; d = u.w;
    } else {
        const RecB16 u = *reinterpret_cast<const RecB16 *>(p);
        a = __bfloat162float(u.a); b = __bfloat162float(u.b);
        c = __bfloat162float(u.c); d = __bfloat162float(u.d);
    }
}

// Multiply-adds of the triangular sweeps, fused explicitly so that every kernel
// that runs them rounds identically: fmsub(a, b, s) = s - a b, fmadd(a, b, s) = s + a b.
__device__ __forceinline__ float fmsub(float a, float b, float s) { return __fmaf_rn(-a, b, s); }
__device__ __forceinline__ double fmsub(double a, double b, double s) { return __fma_rn(-a, b, s); }
__device__ __forceinline__ float fmadd(float a, float b, float s) { return __fmaf_rn(a, b, s); }
__device__ __forceinline__ double fmadd(double a, double b, double s) { return __fma_rn(a, b, s); }

// ---------------------------------------------------------------------------
// cp.async staging
// ---------------------------------------------------------------------------

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// copy the 16-byte-aligned window around global bytes [b0, b1) of `base`
// into `dst`; the data of byte b0 lands at dst + (b0 & 15)
__device__ __forceinline__ void stage_bytes(unsigned char *dst, const unsigned char *base,
                                            long long b0, long long b1) {
    const long long a0 = b0 & ~15LL;
    const long long a1 = (b1 + 15) & ~15LL;
    for (long long o = a0 + 16LL * threadIdx.x; o < a1; o += 16LL * blockDim.x)
        cp_async16(dst + (o - a0), base + o);
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------

// q / d for 0 <= q < 2^16 and 1 <= d <= 256 as a multiply-high by ceil(2^32 / d)
// (exact in that range: q (ceil(2^32/d) d - 2^32) < 2^32 since the excess is < d)
__host__ __device__ __forceinline__ unsigned magic_div(int d) {
    return d == 1 ? 0u : (unsigned)((0x100000000ull + (unsigned)d - 1) / (unsigned)d);
}
__device__ __forceinline__ int fast_div(int q, int d, unsigned m) {
    return d == 1 ? q : (int)__umulhi((unsigned)q, m);
}



// A read-only load that stays where it is written (a batch of loads before their uses)
__device__ __forceinline__ double load_now(const double *p) {
    double v;
    asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}

// One subdomain solve (one CTA), cell by cell: box `box` of the handle described by P,
// input r, output z (whole-grid vectors of that handle).
template <int PREC, int NBUF>
__device__ __forceinline__ void ras_apply_cells(const ApplyParams &P, int box, const double *r, double *z,
                                              int accumulate) {
    using R = typename RecT<PREC>::T;
    using Acc = typename RecT<PREC>::Acc;
    constexpr int RB = (int)sizeof(R);
    extern __shared__ __align__(16) unsigned char smem[];
    // [zero guard: gcap][Y: ycap][zero guard: gcap][level starts][ring]
    Acc *Y = reinterpret_cast<Acc *>(smem) + P.gcap;
    const size_t ybytes = ((size_t)P.ycap + 2 * (size_t)P.gcap) * sizeof(Acc);
    int *lvl_s = reinterpret_cast<int *>(smem + ybytes);
    unsigned char *ring = smem + ybytes + (size_t)P.lcap * sizeof(int);
    const int rcap = ((P.chunk_cells * RB + 32) + 15) & ~15;
    const int ccap = ((P.chunk_cells * 4 + 32) + 15) & ~15;
    unsigned char *ring_rec = ring;
    unsigned char *ring_cell = ring + (size_t)NBUF * rcap;

    const SubInfo si = P.subs[box];
    const ShapeInfo sh = P.shapes[si.shape];
    const int *chunk_lev = P.chunk + sh.chunk_off;
    for (int t = threadIdx.x; t <= sh.nlev; t += blockDim.x) lvl_s[t] = P.lvl[sh.lvl_off + t];
    for (int t = threadIdx.x; t < sh.bx * sh.by; t += blockDim.x) {
        Y[-1 - t] = (Acc)0;
        Y[sh.ncell + t] = (Acc)0;
    }
    __syncthreads();

    const int nstage = 2 * sh.nchunk;
    const bool one = (int)blockDim.x >= sh.maxw;   // one cell per thread per level
    auto issue = [&](int t) {
        if (t < nstage) {
            const bool fw = t < sh.nchunk;
            const int c = fw ? t : nstage - 1 - t;
            const int qa = lvl_s[chunk_lev[c]], qb = lvl_s[chunk_lev[c + 1]];
            const int slot = t % NBUF;
            stage_bytes(ring_rec + (size_t)slot * rcap, fw ? P.fwd : P.bwd,
                        (si.foff + qa) * (long long)RB, (si.foff + qb) * (long long)RB);
            stage_bytes(ring_cell + (size_t)slot * ccap,
                        reinterpret_cast<const unsigned char *>(P.cidx),
                        (sh.cell_off + (long long)qa) * 4, (sh.cell_off + (long long)qb) * 4);
        }
        cp_async_commit();
    };
#pragma unroll
    for (int t = 0; t < NBUF - 1; ++t) issue(t);

    // gather R_i^delta r into shared memory, flat over the box's cells with GB
    // loads in flight per thread before any is consumed (the gather is bound by
    // the bytes in flight per SM, not by bandwidth)
    constexpr int GB = 10;   // a batch that stays in 64 registers with the direct z stores
    const int bx = sh.bx, by = sh.by, bxy = sh.bx * sh.by;
    const int nx = P.nx, nxy = P.nx * P.ny;
    const long long g0 = si.e0x + (long long)nx * (si.e0y + (long long)P.ny * si.e0z);
    const double *rg = r + g0;
    const unsigned mbx = magic_div(bx), mby = magic_div(by);
    for (int q0 = threadIdx.x; q0 < sh.ncell; q0 += GB * blockDim.x) {
        double v[GB];
#pragma unroll
        for (int m = 0; m < GB; ++m) {
            const int q = q0 + m * (int)blockDim.x;
            if (q < sh.ncell) {
                const int row = fast_div(q, bx, mbx), k = fast_div(row, by, mby);
                v[m] = load_now(rg + (q - row * bx) + nx * (row - k * by) + nxy * k);
            }
        }
#pragma unroll
        for (int m = 0; m < GB; ++m) {
            const int q = q0 + m * (int)blockDim.x;
            if (q < sh.ncell) {
                bool own = true;
                if (P.kind == 2) {   // right-RAS: R_i^0 on the input (cells of other boxes read as 0)
                    const int row = fast_div(q, bx, mbx), k = fast_div(row, by, mby);
                    const int i = q - row * bx, j = row - k * by;
                    own = i >= si.ox0 && i < si.ox1 && j >= si.oy0 && j < si.oy1 && k >= si.oz0 &&
                          k < si.oz1;
                }
                Y[q] = own ? (Acc)v[m] : (Acc)0;
            }
        }
    }

    // Left-RAS writes each owned cell's z as soon as the backward sweep has it
    // ((R_i^0)^T: one owner per cell, so an add when accumulating is a plain update)
    const bool direct = P.kind == 1;
    double *zg = z + g0;
    auto put = [&](int n, Acc y) {
        const int row = fast_div(n, bx, mbx), k = fast_div(row, by, mby);
        const int i = n - row * bx, j = row - k * by;
        if (i >= si.ox0 && i < si.ox1 && j >= si.oy0 && j < si.oy1 && k >= si.oz0 && k < si.oz1) {
            double *zp = zg + (i + nx * j + nxy * k);
            if (accumulate) atomicAdd(zp, (double)y);
            else *zp = (double)y;
        }
    };

    // Sweeps, level by level. A neighbour outside the box has a zero factor value and
    // reads a finite value (a cell of the box or the zero guard band on either side
    // of Y), so no cell needs a flag test.
    for (int t = 0; t < nstage; ++t) {
        cp_async_wait<NBUF - 2>();
        __syncthreads();
        issue(t + NBUF - 1);
        const bool fw = t < sh.nchunk;
        const int c = fw ? t : nstage - 1 - t;
        const int l0 = chunk_lev[c], l1 = chunk_lev[c + 1];
        const int qa = lvl_s[l0];
        const int slot = t % NBUF;
        const unsigned char *rec = ring_rec + (size_t)slot * rcap +
                                   (int)(((si.foff + qa) * (long long)RB) & 15);
        const int *cel = reinterpret_cast<const int *>(
            ring_cell + (size_t)slot * ccap + (int)(((sh.cell_off + (long long)qa) * 4) & 15));
        // When the block covers the widest level, a level is one guarded pass (no loop
        // back-edge before the barrier) with addresses from per-chunk bases.
        const int tid = threadIdx.x;
        const int *cel_t = cel - qa + tid;                       // cel_t[lo]: cell lo + tid
        const unsigned char *rec_t = rec + (long long)RB * (tid - qa);
        if (one) {
            if (fw) {
#pragma unroll 2
                for (int l = l0; l < l1; ++l) {
                    const int lo = lvl_s[l];
                    if (lo + tid < lvl_s[l + 1]) {
                        const int n = cel_t[lo];
                        Acc ax, ay, az, dinv;
                        load_rec<Acc, R>(rec_t + (size_t)RB * lo, ax, ay, az, dinv);
                        Acc *yn = Y + n;
                        Acc s = yn[0];
                        s = fmsub(az, yn[-bxy], s);
                        s = fmsub(ay, yn[-bx], s);
                        s = fmsub(ax, yn[-1], s);
                        yn[0] = s * dinv;
                    }
                    __syncthreads();
                }
            } else {
#pragma unroll 2
                for (int l = l1 - 1; l >= l0; --l) {
                    const int lo = lvl_s[l];
                    if (lo + tid < lvl_s[l + 1]) {
                        const int n = cel_t[lo];
                        Acc ax, ay, az, dinv;
                        load_rec<Acc, R>(rec_t + (size_t)RB * lo, ax, ay, az, dinv);
                        Acc *yn = Y + n;
                        Acc s = ax * yn[1];
                        s = fmadd(ay, yn[bx], s);
                        s = fmadd(az, yn[bxy], s);
                        const Acc y = fmsub(dinv, s, yn[0]);
                        yn[0] = y;
                        if (direct) put(n, y);
                    }
                    __syncthreads();
                }
            }
            continue;
        }
        if (fw) {
            // forward: w_n = (r_n - sum_{m<n} a_nm w_m) / d_n, w = D^{-1} L^{-1} r
            for (int l = l0; l < l1; ++l) {
                const int q1 = lvl_s[l + 1];
                for (int q = lvl_s[l] + threadIdx.x; q < q1; q += blockDim.x) {
                    const int n = cel[q - qa];
                    Acc ax, ay, az, dinv;
                    load_rec<Acc, R>(rec + (size_t)RB * (q - qa), ax, ay, az, dinv);
                    Acc s = Y[n];
                    s = fmsub(az, Y[n - bxy], s);
                    s = fmsub(ay, Y[n - bx], s);
                    s = fmsub(ax, Y[n - 1], s);
                    Y[n] = s * dinv;
                }
                __syncthreads();
            }
        } else {
            // backward: z_n = w_n - d_n^{-1} sum_{m>n} a_nm z_m
            for (int l = l1 - 1; l >= l0; --l) {
                const int q1 = lvl_s[l + 1];
                for (int q = lvl_s[l] + threadIdx.x; q < q1; q += blockDim.x) {
                    const int n = cel[q - qa];
                    Acc ax, ay, az, dinv;
                    load_rec<Acc, R>(rec + (size_t)RB * (q - qa), ax, ay, az, dinv);
                    Acc s = ax * Y[n + 1];
                    s = fmadd(ay, Y[n + bx], s);
                    s = fmadd(az, Y[n + bxy], s);
                    const Acc y = fmsub(dinv, s, Y[n]);
                    Y[n] = y;
                    if (direct) put(n, y);
                }
                __syncthreads();
            }
        }
    }
    cp_async_wait<0>();

    if (P.kind != 1) {   // AS / right-RAS: the whole box solution, summed per cell later
        double *dst = P.zbuf + si.foff;
        for (int q = threadIdx.x; q < sh.ncell; q += blockDim.x) dst[q] = (double)Y[q];
        return;
    }
}

// ---- mbarriers of the sweeps in blocks (one phase per box; waits are bounded) ----
constexpr int APPLY_TIMEOUT = 7;                // error word of a wait that ran out
constexpr int APPLY_POLLS = 1 << 22;
// what a wait needs: the handle's error word, the CTA's flag of a wait that ran out (the
// others then give up too: the box is lost, and every role still runs to its end; the steps
// copied follow it), and the launch's poll limit (0: the default)
struct Waits {
    int *err;
    volatile int *failed;
    int polls;
};
__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mb_init(unsigned long long *b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mb_inval(unsigned long long *b) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void mb_arrive(unsigned long long *b) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
}
// one poll (the hardware suspends it for a while), or a test without a wait
__device__ __forceinline__ bool mb_poll(unsigned long long *b) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred pp;\n"
        "mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 pp, [%1], 0;\n"
        "selp.u32 %0, 1, 0, pp;\n}\n"
        : "=r"(ok) : "r"(smem_addr(b)) : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mb_test(unsigned long long *b) {
    unsigned ok;
    asm volatile(
        "{\n.reg .pred pp;\n"
        "mbarrier.test_wait.parity.acquire.cta.shared::cta.b64 pp, [%1], 0;\n"
        "selp.u32 %0, 1, 0, pp;\n}\n"
        : "=r"(ok) : "r"(smem_addr(b)) : "memory");
    return ok != 0;
}
template <bool LIMIT>
__device__ __forceinline__ bool mb_wait(unsigned long long *b, const Waits &w) {
    for (int it = 0; it < (LIMIT ? w.polls : APPLY_POLLS); ++it) {
        if (LIMIT ? mb_test(b) : mb_poll(b)) return true;
        if (*w.failed) return false;
    }
    *w.failed = 1;
    atomicMax(w.err, APPLY_TIMEOUT);
    return false;
}
// `bytes` of global memory into shared memory by the bulk copy engine, completing on b
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, unsigned long long *b) {
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;"
                 ::"r"(smem_addr(b)), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(b)) : "memory");
}
__device__ __forceinline__ void cta_barrier() { asm volatile("bar.sync 0;" ::: "memory"); }   // (from any warp role)

// One subdomain solve (one CTA) in blocks of 2 x 2 cells of a plane, FP32 / BF16 factors.
//
// Cell by cell the sweeps are chains of bx + by + bz - 2 levels (58 for 20^3), each a CTA
// barrier, a table look-up, shared-memory reads and one cell's arithmetic: ~0.2 us per
// level whatever the bytes, 23 of the kernel's 45 us. Over blocks of 2 x 2 cells a sweep has
// bx / 2 + by / 2 + bz - 2 levels (38) of at most 100 blocks, one thread per block: a thread
// reads its 4 records (ahead of the barrier) and 4 + 8 values, runs the block's cells in
// registers in natural order and writes 4 values. Every cell's arithmetic and its order
// are those of the cell-by-cell sweep, so the values are the same bit for bit.
// 45.5 -> 34.8 us per launch on 128 x 128 x 64 cells (256 boxes of up to 20^3, FP32, 69 MB:
// 1.97 TB/s). What bounds it is the length of the warps' instruction streams, about 18
// cycles per instruction and warp with ~5 warps per scheduler (ncu): a level of the sweep
// is ~80 instructions, ~400 cycles. Blocks of 2 x 2 x 2 cells have 28 levels of ~620 cycles:
// the same time, and more padding on flat boxes. With half as many helpers (four cells of a
// plane each) the gather takes 43 us.
//
// Warp roles, so that the sweeping warps wait for nothing but one another:
//   - sweepers (as many as the widest level takes) meet at a barrier of their own per
//     level;
//   - one thread streams the records, level by level, into a ring with bulk copies, as far
//     ahead as the ring holds (a host table gives each step's place and how far to run);
//   - one warp waits for them and for r, and joins the sweepers' barrier when both are in;
//   - the helpers gather r plane by plane ahead of the forward sweep (every thread the same
//     cells of each plane: index arithmetic per cell took longer than the loads), and write the owned cells of every
//     four levels that the backward sweep has finished.
// All warps meeting at one barrier per level took 43 us: the level then takes as long as
// its slowest role.
//
// The vector is held as float4 per block (elements di + 2 dj), with a plane stride that
// makes the threads of a level (J + 1, k - 1 from one lane to the next) step by an odd
// number of 16-byte units: no bank conflicts. A neighbour outside the box has a zero
// factor value and reads a finite value (a block of the box or the zero guard on either
// side); cells that pad an odd edge are zero throughout (zero records).
constexpr int PUT_LEVELS = 4;
template <int PREC, bool LIMIT>
__device__ __forceinline__ void ras_apply_blocks(const ApplyParams &P, int box, const double *r, double *z,
                                                 int accumulate, int polls) {
    using R = typename RecT<PREC>::T;
    constexpr int RB = (int)sizeof(R);
    extern __shared__ __align__(16) unsigned char smem[];
    const BoxInfo bi = P.boxes[box];
    const SubInfo &si = bi.sub;
    const ShapeInfo &sh = bi.shape;
    const int bx = sh.bx, by = sh.by, bz = sh.bz, mx = sh.mx, mp = sh.mp, nlev = sh.nlev, nstep = 2 * nlev;
    const int yoff = sh.my > 1 ? mx : 0, zoff = bz > 1 ? mp : 0, guard = sh.guard;
    // [values with guards][steps][block table][mbarriers: records of a step in / read, plane of r, put of levels][ring]
    float4 *Y = reinterpret_cast<float4 *>(smem) + P.gcap;
    int4 *st = reinterpret_cast<int4 *>(Y + P.ycap + P.gcap);
    unsigned *bt = reinterpret_cast<unsigned *>(st + 2 * P.lcap);           // I | J << 8 | k << 16, level order
    unsigned long long *mb_rec = reinterpret_cast<unsigned long long *>(bt + P.ycap);
    unsigned long long *mb_free = mb_rec + 2 * P.lcap, *mb_pl = mb_free + 2 * P.lcap, *mb_put = mb_pl + P.lcap;
    unsigned char *ring = reinterpret_cast<unsigned char *>(mb_put + P.lcap);
    // (the last of mb_free's places is beyond the last step)
    const Waits wt{P.err, reinterpret_cast<volatile int *>(mb_free + 2 * P.lcap - 1), polls};
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    // warps: sweepers, helpers (one at least, see the launch), a waiter and an issuer
    const int nsw = (sh.maxw + 31) & ~31, nh = nt - nsw - 64;
    const bool sweeper = tid < nsw, waiter = tid >= nt - 64 && tid < nt - 32, issuer = tid >= nt - 32;
    const bool helper = !sweeper && tid < nt - 64;
    const int ht = tid - nsw;                                               // helper's number
    const int nput = (nlev + PUT_LEVELS - 1) / PUT_LEVELS;

    const int nx = P.nx, nxy = P.nx * P.ny, bxy = bx * by;
    const long long g0 = si.e0x + (long long)nx * (si.e0y + (long long)P.ny * si.e0z);
    const unsigned mbx = magic_div(bx), mby = magic_div(by);
    auto element = [&](int i, int j, int k) { return 4 * ((i >> 1) + mx * (j >> 1) + mp * k) + (i & 1) + 2 * (j & 1); };
    // right-RAS: R_i^0 on the input (cells of other boxes read as 0)
    auto in_xy = [&](int i, int j) {
        return P.kind != 2 || (i >= si.ox0 && i < si.ox1 && j >= si.oy0 && j < si.oy1);
    };
    auto in_z = [&](int k) { return P.kind != 2 || (k >= si.oz0 && k < si.oz1); };
    // helpers: R_i^delta r. A thread takes the same GC cells of every plane, so their places
    // are computed once, and holds GD planes' loads in flight.
    constexpr int GC = 2, GD = 4;
    double v[GD][GC];
    int off[GC], elem[GC];
    const bool planes = GC * nh >= bxy;          // (else: cell by cell, long thin boxes)
    auto fetch = [&](int k, double (&d)[GC]) {
#pragma unroll
        for (int c = 0; c < GC; ++c)
            if (k < bz && off[c] >= 0) d[c] = load_now(r + g0 + off[c] + (long long)nxy * k);
    };
    if (helper && planes) {
#pragma unroll
        for (int c = 0; c < GC; ++c) {
            const int q = ht + c * nh, j = fast_div(q, bx, mbx), i = q - j * bx;
            off[c] = q < bxy && in_xy(i, j) ? i + nx * j : -1;
            elem[c] = element(i, j, 0);
        }
#pragma unroll
        for (int d = 0; d < GD; ++d) fetch(d, v[d]);
    }
    const int4 *steps = P.steps + sh.chunk_off;  // [nstep + 1]: {first block, blocks, ring place / 16, issue limit}
    {
        const int nall = mp * bz;
        const bool pad = ((bx | by) & 1) != 0 || mp != mx * sh.my;
        for (int t = tid; t <= nstep; t += nt) st[t] = steps[t];
        for (int t = tid; t < sh.nblk; t += nt) bt[t] = (unsigned)P.cidx[sh.cell_off + t];
        for (int t = tid; t < nstep; t += nt) {
            mb_init(mb_rec + t, 1);
            mb_init(mb_free + t, 1);
        }
        for (int t = tid; t < bz; t += nt) mb_init(mb_pl + t, nh >> 5);
        for (int t = tid; t < nput; t += nt) mb_init(mb_put + t, nsw >> 5);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        // a batch's boxes of other handles have their vectors and tables where this one has
        // its ring: their ordinary writes come before the bulk copies
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int t = tid; t < guard; t += nt) Y[-1 - t] = Y[nall + t] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tid == 0) *wt.failed = 0;
        if (pad || P.kind == 2)
            for (int t = tid; t < nall; t += nt) Y[t] = make_float4(0.f, 0.f, 0.f, 0.f);
        cta_barrier();
    }
    // helpers: (R_i^0)^T of the blocks [b0, b1) of the table, a row of two cells per item
    double *zg = z + g0;
    auto put = [&](int b0, int b1) {
        for (int e = 2 * b0 + ht; e < 2 * b1; e += nh) {
            const unsigned b = bt[e >> 1];
            const int I = b & 255u, J = (b >> 8) & 255u, k = b >> 16, c = e & 1;
            const int i = 2 * I, j = 2 * J + c;
            if (j < si.oy0 || j >= si.oy1 || k < si.oz0 || k >= si.oz1) continue;
            const float2 y = reinterpret_cast<const float2 *>(Y + (I + mx * J + mp * k))[c];
            double *zp = zg + (i + nx * j + nxy * k);
            if (i >= si.ox0 && i < si.ox1) {
                if (accumulate) atomicAdd(zp, (double)y.x);   // one owner per cell
                else zp[0] = (double)y.x;
            }
            if (i + 1 >= si.ox0 && i + 1 < si.ox1) {
                if (accumulate) atomicAdd(zp + 1, (double)y.y);
                else zp[1] = (double)y.y;
            }
        }
    };

    float ax[4] = {}, ay[4] = {}, az[4] = {}, di[4] = {};
    int m = 0;                                   // this thread's block of the coming step
    bool on = false;
    auto fcell = [&](int c, float s, float zv, float yv, float xv) {   // w_n = (r_n - sum_{m<n} a_nm w_m) / d_n
        s = fmsub(az[c], zv, s);
        s = fmsub(ay[c], yv, s);
        return fmsub(ax[c], xv, s) * di[c];
    };
    auto forward = [&]() {
        float4 a = Y[m];
        const float4 zm = Y[m - zoff], xm = Y[m - 1];
        const float2 ym = reinterpret_cast<const float2 *>(Y + (m - yoff))[1];
        a.x = fcell(0, a.x, zm.x, ym.x, xm.y);
        a.y = fcell(1, a.y, zm.y, ym.y, a.x);
        a.z = fcell(2, a.z, zm.z, a.x, xm.w);
        a.w = fcell(3, a.w, zm.w, a.y, a.z);
        Y[m] = a;
    };
    auto bcell = [&](int c, float w, float xv, float yv, float zv) {   // z_n = w_n - d_n^{-1} sum_{m>n} a_nm z_m
        float s = ax[c] * xv;
        s = fmadd(ay[c], yv, s);
        s = fmadd(az[c], zv, s);
        return fmsub(di[c], s, w);
    };
    auto backward = [&]() {
        float4 a = Y[m];
        const float4 zp = Y[m + zoff], xp = Y[m + 1];
        const float2 yp = reinterpret_cast<const float2 *>(Y + (m + yoff))[0];
        a.w = bcell(3, a.w, xp.z, yp.y, zp.w);
        a.z = bcell(2, a.z, a.w, yp.x, zp.z);
        a.y = bcell(1, a.y, xp.x, a.w, zp.y);
        a.x = bcell(0, a.x, a.y, a.z, zp.x);
        Y[m] = a;
    };
    // step n: forward level n, then backward level 2 nlev - 1 - n
    auto step_barrier = [&]() { asm volatile("bar.sync 1, %0;" ::"r"(nsw + 32) : "memory"); };
    if (sweeper) {
        // the coming step's table entries are read two steps ahead, its records one
        int4 s = st[0], s1 = st[1];
        unsigned b = tid < s.y ? bt[s.x + tid] : 0u;
        auto load = [&](int n) {                 // the records of step n, w blocks apart
            on = tid < s.y;
            if (on) {
                m = (int)(b & 255u) + mx * (int)((b >> 8) & 255u) + mp * (int)(b >> 16);
                const unsigned char *rec = ring + 16 * s.z + RB * tid;
#pragma unroll
                for (int c = 0; c < 4; ++c) load_rec<float, R>(rec + RB * c * s.y, ax[c], ay[c], az[c], di[c]);
            }
            s = s1;
            b = tid < s.y ? bt[s.x + tid] : 0u;
        };
        step_barrier();                          // the first records
        load(0);
        for (int n = 0; n < nlev; ++n) {
            step_barrier();
            s1 = st[min(n + 2, nstep - 1)];
            if (on) forward();
            load(n + 1);
        }
        for (int n = nlev; n < nstep; ++n) {
            step_barrier();
            s1 = st[min(n + 2, nstep - 1)];
            if (on) backward();
            const int done = n - nlev + 1;
            if (done % PUT_LEVELS == 0 || n + 1 == nstep) {
                __syncwarp();
                if (lane == 0) mb_arrive(mb_put + (done - 1) / PUT_LEVELS);
            }
            if (n + 1 < nstep) load(n + 1);
        }
    } else if (waiter) {
        // joins the barrier of step n when the plane of r that it reads and the records of
        // step n + 1 are in (the sweepers wait for nothing else); after it step n's records
        // are in registers and their place in the ring is free
        mb_wait<LIMIT>(mb_rec, wt);
        step_barrier();
        for (int n = 0; n < nstep; ++n) {
            if (n < bz) mb_wait<LIMIT>(mb_pl + n, wt);
            if (n + 1 < nstep) mb_wait<LIMIT>(mb_rec + n + 1, wt);
            step_barrier();
            if (lane == 0) mb_arrive(mb_free + n);
        }
    } else if (issuer) {
        if (lane == 0) {
            int next = 0;
            for (int n = -1; n < nstep; ++n) {
                if (n >= 0 && !mb_wait<LIMIT>(mb_free + n, wt)) break;
                const int lim = st[n < 0 ? nstep : n].w;
                for (; next <= lim; ++next) {
                    const int4 s = st[next];
                    const unsigned char *src = (next < nlev ? P.fwd : P.bwd) + (si.foff + 4LL * s.x) * RB;
                    bulk_load(ring + 16 * s.z, src, 4u * s.y * RB, mb_rec + next);
                }
                if (next == nstep) break;
            }
            wt.failed[1] = next;                 // steps whose copies were started
        }
    } else {
        float *Yf = reinterpret_cast<float *>(Y);
        auto arrive = [&](int k) {
            __syncwarp();
            if (lane == 0) mb_arrive(mb_pl + k);
        };
        if (planes) {
            for (int k0 = 0; k0 < bz; k0 += GD) {
#pragma unroll
                for (int d = 0; d < GD; ++d) {
                    const int k = k0 + d;
                    if (k >= bz) continue;
#pragma unroll
                    for (int c = 0; c < GC; ++c)
                        if (off[c] >= 0 && in_z(k)) Yf[elem[c] + 4 * mp * k] = (float)v[d][c];
                    fetch(k + GD, v[d]);
                    arrive(k);
                }
            }
        } else {
            for (int k = 0; k < bz; ++k) {
                for (int q = ht; q < bxy; q += nh) {
                    const int j = fast_div(q, bx, mbx), i = q - j * bx;
                    if (in_xy(i, j) && in_z(k))
                        Yf[element(i, j, k)] = (float)__ldg(r + g0 + i + nx * j + (long long)nxy * k);
                }
                arrive(k);
            }
        }
        if (P.kind == 1)
            for (int e = 0; e < nput; ++e) {     // levels nlev - 1 - PUT_LEVELS e downwards
                mb_wait<LIMIT>(mb_put + e, wt);
                const int l1 = nlev - PUT_LEVELS * e, l0 = max(0, l1 - PUT_LEVELS);
                put(st[l0].x, st[l1 - 1].x + st[l1 - 1].y);
            }
    }
    cta_barrier();
    if (*wt.failed) {                            // the box is lost: its last copies land before the CTA goes on
        for (int t = tid; t < wt.failed[1]; t += nt)
            for (int it = 0; !mb_poll(mb_rec + t) && it < APPLY_POLLS; ++it) {}
        cta_barrier();
    }
    for (int t = tid; t < nstep; t += nt) {
        mb_inval(mb_rec + t);
        mb_inval(mb_free + t);
    }
    for (int t = tid; t < bz; t += nt) mb_inval(mb_pl + t);
    for (int t = tid; t < nput; t += nt) mb_inval(mb_put + t);
    if (P.kind != 1) {   // AS / right-RAS: the whole box solution, summed per cell later
        double *dst = P.zbuf + si.foff;
        for (int q = tid; q < sh.ncell; q += nt) {
            const int row = fast_div(q, bx, mbx), k = fast_div(row, by, mby);
            dst[q] = (double)reinterpret_cast<const float *>(Y)[element(q - row * bx, row - k * by, k)];
        }
    }
}

template <int PREC, bool LIMIT>
__device__ __forceinline__ void ras_apply_box(const ApplyParams &P, int box, const double *r, double *z,
                                              int accumulate, int polls) {
    if constexpr (PREC == 64) ras_apply_cells<PREC, 3>(P, box, r, z, accumulate);
    else ras_apply_blocks<PREC, LIMIT>(P, box, r, z, accumulate, polls);
}

// 64 registers for 2 CTAs of 512 threads per SM with FP64 factors, 72 for two of 448 with
// reduced ones. LIMIT: the waits take the launch's poll limit.
template <int PREC, bool LIMIT>
__global__ void __maxnreg__(PREC == 64 ? 64 : 72) k_ras_apply(ApplyParams P) {
    ras_apply_box<PREC, LIMIT>(P, blockIdx.x, P.r, P.z, P.accumulate, P.polls);
}

// Left-RAS of many handles in one persistent launch: every CTA takes the next
// item of a work queue (an atomic counter over the table of (handle, box), sorted
// largest box first) until the queue is empty, and solves box box_local[item] of
// handle box_inst[item] (items of inactive handles are skipped); r and z are the
// handles' vectors concatenated at off[handle]. No CTA waits on another.
template <int PREC, bool LIMIT>
__global__ void __maxnreg__(PREC == 64 ? 64 : 72) k_ras_apply_batch(BatchApply B) {
    __shared__ int s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(B.qcount, 1);
        __syncthreads();
        const int it = s_item;
        __syncthreads();   // every thread holds the item, and the last box's shared memory is free
        if (it >= B.nitems) return;
        const int h = B.box_inst[it];
        if (!B.active[h]) continue;
        ras_apply_box<PREC, LIMIT>(B.inst[h], B.box_local[it], B.r + B.off[h], B.z + B.off[h], B.accumulate, B.polls);
    }
}

// z (+)= sum over the overlapped boxes covering each cell of their solution
// ((R_i^delta)^T), boxes in ascending index order (deterministic)
struct SumParams {
    const SubInfo *subs;
    const ShapeInfo *shapes;
    const int *clo[3], *chi[3];   // per axis and coordinate: parts whose boxes cover it
    int parts[3];
    int nx, ny, nz;
    const double *zbuf;
    double *z;
    int accumulate;
};

__global__ void __launch_bounds__(256) k_ras_sum(SumParams P) {
    const long long N = (long long)P.nx * P.ny * P.nz;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        const int c[3] = {(int)(n % P.nx), (int)((n / P.nx) % P.ny), (int)(n / ((long long)P.nx * P.ny))};
        double acc = 0.0;
        for (int pz = P.clo[2][c[2]]; pz <= P.chi[2][c[2]]; ++pz) {
            for (int py = P.clo[1][c[1]]; py <= P.chi[1][c[1]]; ++py) {
                for (int px = P.clo[0][c[0]]; px <= P.chi[0][c[0]]; ++px) {
                    const SubInfo si = P.subs[px + P.parts[0] * (py + P.parts[1] * pz)];
                    const ShapeInfo &sh = P.shapes[si.shape];
                    const int q = (c[0] - si.e0x) + sh.bx * ((c[1] - si.e0y) + sh.by * (c[2] - si.e0z));
                    acc += P.zbuf[si.foff + q];
                }
            }
        }
        P.z[n] = P.accumulate ? P.z[n] + acc : acc;
    }
}


// ---------------------------------------------------------------------------
// ILU(0) factorisation
// ---------------------------------------------------------------------------

// (u, v) pairs of an nu x nv grid with u + v < d: those of the quarter plane less those
// past either edge
__host__ __device__ __forceinline__ int tri(int x) { return x > 0 ? x * (x + 1) / 2 : 0; }
__host__ __device__ __forceinline__ int diag_base(int d, int nu, int nv) {
    return tri(d) - tri(d - nu) - tri(d - nv) + tri(d - nu - nv);
}
// position of (u, v) in the order by diagonal u + v, then u
__host__ __device__ __forceinline__ int diag_pos(int u, int v, int nu, int nv) {
    return diag_base(u + v, nu, nv) + u - max(0, u + v - (nv - 1));
}

// axis along which the factorisation's pencils run: x unless that leaves too many
// pencils for one CTA, then the longest axis (at most 16384^(2/3) = 645 pencils)
constexpr int FAC_MAXPEN = 1024;
__host__ __device__ __forceinline__ int pencil_axis(int bx, int by, int bz) {
    if (by * bz <= FAC_MAXPEN) return 0;
    return bx >= by && bx >= bz ? 0 : (by >= bz ? 1 : 2);
}
__host__ __device__ __forceinline__ int pencil_count(int bx, int by, int bz) {
    const int a = pencil_axis(bx, by, bz);
    return a == 0 ? by * bz : (a == 1 ? bx * bz : bx * by);
}

// ILU(0) of A_i in natural order: only the diagonal changes,
// d_n = a_nn - sum_{m<n neighbour} a_nm (a_mn / d_m)   (m: -z, -y, -x).
// One CTA per box (box `box` of the handle described by P), one thread per pencil of
// cells; a pencil handles one cell per wavefront level, so a_mn / d_m of its own previous
// cell is in a register and those of the two neighbouring pencils, finished at the
// previous level, in a shared slot per pencil (by parity of the level). Every operator
// value is read once, consecutive along the pencil, a level ahead of its use, and both
// factor records are written at once. Pencils are numbered by diagonal, so that a warp's
// pencils are active together.
//
// Bound: FP64 (2 FMA per cycle and SM): 3 FMA, a reciprocal (3 FMA, where a division takes
// about ten operations) and 3 multiplications per cell. Three divisions per cell, the
// operator read cell by cell in level order and a second pass for the records took 1.8
// times as long: factors and a first use, 60 x 220 x 85 cells in FP64, 585 -> 323 us.
template <int PREC, int pa>
__device__ __forceinline__ void ras_factor_pencils(const FactorParams &P, const SubInfo &si, const ShapeInfo &sh) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr int ua = pa == 0 ? 1 : 0, va = pa == 2 ? 1 : 2;
    auto stride = [&](int a) { return a == 0 ? 1LL : (a == 1 ? (long long)P.nx : (long long)P.nx * P.ny); };
    const int nm = pa == 0 ? sh.bx : (pa == 1 ? sh.by : sh.bz), nu = ua ? sh.by : sh.bx, nv = va == 1 ? sh.by : sh.bz;
    const int npen = nu * nv, S = nm + nu + nv - 2;
    double *su = reinterpret_cast<double *>(smem), *sv = su + 2 * npen;   // [2][npen]: a_mn / d_m towards +u, +v
    int *lstart = reinterpret_cast<int *>(sv + 2 * npen);                 // [nlev]: first record less its first number
    int *lw = lstart + sh.nlev;                                           // [nlev]: records between a block's cells
    for (int l = threadIdx.x; l < sh.nlev; l += blockDim.x) {
        const int a = P.lvl[sh.lvl_off + l], b = P.lvl[sh.lvl_off + l + 1];
        if constexpr (PREC == 64) lstart[l] = a - diag_base(max(0, l - sh.bx + 1), sh.by, sh.bz);
        else lstart[l] = 4 * a - diag_base(max(0, l - sh.mx + 1), sh.my, sh.bz);
        lw[l] = b - a;
    }
    // this thread's pencil
    const int pen = threadIdx.x;
    const bool live = pen < npen;
    int u = 0, v = 0;
    if (live) {
        int d = 0;
        while (diag_base(d + 1, nu, nv) <= pen) ++d;
        u = max(0, d - (nv - 1)) + pen - diag_base(d, nu, nv);
        v = d - u;
    }
    const int qu = live && u > 0 ? diag_pos(u - 1, v, nu, nv) : pen, qv = live && v > 0 ? diag_pos(u, v - 1, nu, nv) : pen;
    const bool mu = u > 0, mv = v > 0, pu = u < nu - 1, pv = v < nv - 1;
    const long long g0 = si.e0x + P.nx * (si.e0y + (long long)P.ny * si.e0z) + u * stride(ua) + v * stride(va);
    const long long gm = stride(pa);
    const double *Ac = P.A.c[0] + g0, *Amm = P.A.c[1 + 2 * pa] + g0, *Apm = P.A.c[2 + 2 * pa] + g0;
    const double *Amu = P.A.c[1 + 2 * ua] + g0, *Apu = P.A.c[2 + 2 * ua] + g0;
    const double *Amv = P.A.c[1 + 2 * va] + g0, *Apv = P.A.c[2 + 2 * va] + g0;
    double nc = 0, nmm = 0, npm = 0, nmu = 0, npu = 0, nmv = 0, npv = 0;   // the coming cell's row
    auto fetch = [&](int m) {
        if (!live || (unsigned)m >= (unsigned)nm) return;
        const long long o = m * gm;
        nc = __ldg(Ac + o);
        nmm = m > 0 ? __ldg(Amm + o) : 0.0;
        npm = m < nm - 1 ? __ldg(Apm + o) : 0.0;
        nmu = mu ? __ldg(Amu + o) : 0.0;
        npu = pu ? __ldg(Apu + o) : 0.0;
        nmv = mv ? __ldg(Amv + o) : 0.0;
        npv = pv ? __ldg(Apv + o) : 0.0;
    };
    fetch(0);
    __syncthreads();
    double um = 0.0;                       // a_mn / d_m of the pencil's previous cell
    bool bad = false;
    for (int l = 0; l < S; ++l) {
        const int m = l - u - v, par = l & 1;
        if (live && (unsigned)m < (unsigned)nm) {
            const double c = nc, mm = nmm, pm = npm, m1 = nmu, p1 = npu, m2 = nmv, p2 = npv;
            fetch(m + 1);
            double d = c;
            if (mv) d = fma(-m2, sv[(par ^ 1) * npen + qv], d);
            if (mu) d = fma(-m1, su[(par ^ 1) * npen + qu], d);
            d = fma(-mm, um, d);
            if (!(d != 0.0) || !isfinite(d)) bad = true;
            const double di = recip64(d);
            um = pm * di;
            su[par * npen + pen] = p1 * di;
            sv[par * npen + pen] = p2 * di;
            // the cell and its two records
            const int i = pa == 0 ? m : u, j = pa == 1 ? m : (pa == 0 ? u : v), k = pa == 2 ? m : v;
            long long at;
            if constexpr (PREC == 64) {
                at = si.foff + lstart[i + j + k] + diag_pos(j, k, sh.by, sh.bz);
            } else {
                const int J = j >> 1, L = (i >> 1) + J + k;
                at = si.foff + lstart[L] + lw[L] * ((i & 1) + 2 * (j & 1)) + diag_pos(J, k, sh.my, sh.bz);
            }
            const double mx = pa == 0 ? mm : m1, my = pa == 1 ? mm : (pa == 0 ? m1 : m2), mz = pa == 2 ? mm : m2;
            const double px = pa == 0 ? pm : p1, py = pa == 1 ? pm : (pa == 0 ? p1 : p2), pz = pa == 2 ? pm : p2;
            store_rec<PREC>(P.fwd, at, mx, my, mz, di);
            store_rec<PREC>(P.bwd, at, px, py, pz, di);
        }
        __syncthreads();
    }
    if (bad) atomicMax(P.err, 1);
}
template <int PREC>
__device__ __forceinline__ void ras_factor_box(const FactorParams &P, int box) {
    const SubInfo si = P.subs[box];
    const ShapeInfo sh = P.shapes[si.shape];
    const int a = pencil_axis(sh.bx, sh.by, sh.bz);
    if (a == 0) ras_factor_pencils<PREC, 0>(P, si, sh);
    else if (a == 1) ras_factor_pencils<PREC, 1>(P, si, sh);
    else ras_factor_pencils<PREC, 2>(P, si, sh);
}

template <int PREC>
__global__ void __launch_bounds__(FAC_MAXPEN, 1) k_ras_factor(FactorParams P) {
    ras_factor_box<PREC>(P, blockIdx.x);
}

// The subdomain ILU(0) factorisations of several handles in one launch: CTA b
// factors box box_local[b] of handle box_inst[b] (CTAs of inactive handles return).
template <int PREC>
__global__ void __launch_bounds__(FAC_MAXPEN, 1) k_ras_factor_batch(const FactorParams *__restrict__ inst,
                                                          const int *__restrict__ box_inst,
                                                          const int *__restrict__ box_local,
                                                          const unsigned char *__restrict__ active) {
    const int h = box_inst[blockIdx.x];
    if (!active[h]) return;
    ras_factor_box<PREC>(inst[h], box_local[blockIdx.x]);
}

// ---------------------------------------------------------------------------
// host set-up
// ---------------------------------------------------------------------------

static std::vector<int> split_axis(int n, int parts) {
    std::vector<int> s(parts + 1);
    const int q = n / parts, r = n % parts;
    for (int p = 0; p <= parts; ++p) s[p] = p * q + std::min(p, r);
    return s;
}

// The opt-in limit is raised to the per-CTA maximum once: a later set-up with
// a smaller need must not lower it under a handle that needs more.
constexpr int SMEM_OPTIN = 227 * 1024;
template <int PREC, bool LIMIT>
static int set_apply_attr() {
    RAS_CK(cudaFuncSetAttribute(k_ras_apply<PREC, LIMIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_OPTIN));
    cudaFuncAttributes fa{};   // the persistent batch kernel has a little static shared memory
    RAS_CK(cudaFuncGetAttributes(&fa, k_ras_apply_batch<PREC, LIMIT>));
    RAS_CK(cudaFuncSetAttribute(k_ras_apply_batch<PREC, LIMIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                SMEM_OPTIN - (int)fa.sharedSizeBytes));
    return RAS_OK;
}
template <int PREC>
static int set_factor_attr() {
    RAS_CK(cudaFuncSetAttribute(k_ras_factor<PREC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                SMEM_OPTIN));
    RAS_CK(cudaFuncSetAttribute(k_ras_factor_batch<PREC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                SMEM_OPTIN));
    return RAS_OK;
}

// Level schedule of the subdomain solves: chunks of consecutive levels with at most
// chunk_cells cells (staged into the shared-memory ring together) and threads per
// box. 0 takes the default (chunk 1024 cells, 384 in FP64; threads: the widest
// level rounded up to a warp), or the RAS_APPLY_CHUNK / RAS_APPLY_THREADS tuning
// knobs. Fills the shapes' chunk offsets, chunk_tab, block and smem_apply.
static int schedule_tables(Ras1 &R, int chunk_cells, int threads, std::vector<int> &chunk_tab) {
    int base_chunk = R.prec == 64 ? 384 : 1024;
    if (const char *e = getenv("RAS_APPLY_CHUNK")) {     // tuning knob
        const int v = atoi(e);
        if (v >= 64 && v <= 8192) base_chunk = v;
    }
    if (chunk_cells > 0) base_chunk = chunk_cells;
    int cc = std::max(base_chunk, R.maxw);
    int block = std::min(512, std::max(64, ((R.maxw + 31) / 32) * 32));
    if (const char *e = getenv("RAS_APPLY_THREADS")) {   // tuning knob
        const int v = atoi(e);
        if (v >= 32 && v <= 512 && v % 32 == 0) block = v;
    }
    if (threads > 0) {
        if (threads > 512 || threads % 32) return RAS_EINVAL;
        block = threads;
    }
    // what a schedule may ask for: the shared memory of the sweeps cell by cell (the sweeps in
    // blocks cut their ring to the room there is, and would take any chunk)
    const size_t acc = R.prec == 64 ? 8 : 4;
    const size_t rcap = ((cc * R.rec_bytes + 32) + 15) & ~15;
    const size_t ccap = ((cc * 4 + 32) + 15) & ~15;
    size_t smem = (R.ycap_cells + 2 * (size_t)R.gcap_cells) * acc + R.lcap_cells * sizeof(int) + 3 * (rcap + ccap);
    if (smem > 227 * 1024) return RAS_EINVAL;
    int launch = block;
    chunk_tab.clear();
    if (R.prec == 64) {
        for (auto &sh : R.shapes) {
            sh.chunk_off = (int)chunk_tab.size();
            const int *lv = &R.h_lvl[sh.lvl_off];
            int l = 0;
            chunk_tab.push_back(0);
            int nch = 0;
            while (l < sh.nlev) {
                int l1 = l + 1;
                while (l1 < sh.nlev && lv[l1 + 1] - lv[l] <= cc) ++l1;
                chunk_tab.push_back(l1);
                ++nch;
                l = l1;
            }
            sh.nchunk = nch;
        }
    } else {
        // blocks of 2 x 2 cells: a ring of three chunks of at least the widest level (less
        // where the box vector leaves less room). The sweeps read step n only when step
        // n + 1 is in, and free its place after that, so the two must lie side by side: with
        // three widest levels they do whichever of them wraps (step n then starts past the
        // first of the three, and n + 1 fits into that); a smaller ring is checked below.
        cc = std::max(cc, 4 * R.maxwb);
        const size_t fixed = ((size_t)R.ycap + 2 * R.gcap) * 16 + (size_t)R.ycap * 4 + R.lcap * (2 * 16 + 6 * 8);
        const size_t room = fixed > 227 * 1024 ? 0 : 227 * 1024 - fixed;
        const size_t ring = std::min(3 * (size_t)cc * R.rec_bytes, room) & ~(size_t)15;
        if (ring < 4 * (size_t)R.maxwb * R.rec_bytes) return RAS_EINVAL;
        smem = fixed + ring;
        R.ring_bytes = ring;
        // sweepers, a waiter, an issuer and helpers enough for a box plane at two cells each
        // (up to 448 threads: two CTAs per SM), one warp at least
        const int own = ((R.maxwb + 31) & ~31) + 64, help = std::max(32, ((R.bxy + 1) / 2 + 31) & ~31);
        launch = std::max(std::max(block, own + 32), std::min(own + help, 448));
        // per shape and step (levels up, then down): first block, blocks, place in the ring
        // (in order, from the start again where the end is too near) and the last step whose
        // place is free once the step's records have been read; a last entry with the limit
        // before the first step
        for (auto &sh : R.shapes) {
            const int *lv = &R.h_lvl[sh.lvl_off];
            const int ns = 2 * sh.nlev;
            sh.chunk_off = (int)chunk_tab.size() / 4;
            std::vector<size_t> a(ns), b(ns);
            size_t at = 0;
            for (int n = 0; n < ns; ++n) {
                const int l = n < sh.nlev ? n : ns - 1 - n;
                const size_t bytes = 4 * (size_t)(lv[l + 1] - lv[l]) * R.rec_bytes;
                if (at + bytes > ring) at = 0;
                a[n] = at;
                b[n] = at += bytes;
            }
            auto limit = [&](int n) {        // steps n + 1 .. s are in the ring together
                int q = n;
                while (q + 1 < ns) {
                    bool ok = true;
                    for (int t = n + 1; t <= q && ok; ++t) ok = b[t] <= a[q + 1] || b[q + 1] <= a[t];
                    if (!ok) break;
                    ++q;
                }
                return q;
            };
            const int first = limit(-1);     // before any step has been read
            for (int n = 0; n < ns; ++n) {
                const int l = n < sh.nlev ? n : ns - 1 - n, lim = limit(n);
                if (lim < std::min(n + 2, ns - 1)) return RAS_EINVAL;
                chunk_tab.insert(chunk_tab.end(), {lv[l], lv[l + 1] - lv[l], (int)(a[n] / 16), lim});
            }
            if (first < std::min(1, ns - 1)) return RAS_EINVAL;
            chunk_tab.insert(chunk_tab.end(), {0, 0, 0, first});
            sh.nchunk = ns;
        }
    }
    R.chunk_cells = cc;
    R.launch = launch;
    R.block = block;
    R.smem_apply = smem;
    return RAS_OK;
}

static int upload_boxes(const Ras1 &R) {
    std::vector<BoxInfo> b;
    for (const SubInfo &s : R.subs) b.push_back(BoxInfo{s, R.shapes[s.shape]});
    RAS_CK(cudaMemcpy(R.d_boxes, b.data(), b.size() * sizeof(BoxInfo), cudaMemcpyHostToDevice));
    return RAS_OK;
}

int ras1_set_schedule(Ras1 &R, int chunk_cells, int threads) {
    if (chunk_cells < 0 || threads < 0) return RAS_EINVAL;
    Ras1 T = R;                 // the tables only change if the new schedule is valid
    std::vector<int> chunk_tab;
    RAS_TRY(schedule_tables(T, chunk_cells, threads, chunk_tab));
    int *d = nullptr;
    RAS_TRY(dalloc(&d, chunk_tab.size()));
    if (cudaMemcpy(d, chunk_tab.data(), chunk_tab.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
        cudaMemcpy(R.d_shapes, T.shapes.data(), T.shapes.size() * sizeof(ShapeInfo), cudaMemcpyHostToDevice) !=
            cudaSuccess || upload_boxes(T) != RAS_OK) {
        dfree(d);
        return RAS_ECUDA;
    }
    dfree(R.d_chunk);
    R.d_chunk = d;
    R.shapes = T.shapes;
    ++R.sched;
    R.chunk_cells = T.chunk_cells;
    R.launch = T.launch;
    R.block = T.block;
    R.smem_apply = T.smem_apply;
    return RAS_OK;
}

// The host side of the set-up: boxes, their shapes and the shapes' level tables (no CUDA
// call). cuts: the owned parts along each axis; cidx_tab: level order, local index of each
// cell (block).
static int ras1_geometry(Ras1 &R, int nx, int ny, int nz, int px, int py, int pz, int overlap, int prec, int kind,
                         std::vector<int> (&cuts)[3], std::vector<int> &cidx_tab) {
    if (px < 1 || py < 1 || pz < 1 || overlap < 0) return RAS_EINVAL;
    if (kind < 0 || kind > 2) return RAS_EINVAL;
    R.kind = kind;
    if (px > nx || py > ny || pz > nz) return RAS_EINVAL;
    if (prec != 64 && prec != 32 && prec != 16) return RAS_EINVAL;
    R.nx = nx; R.ny = ny; R.nz = nz; R.N = nx * ny * nz;
    R.prec = prec;
    R.rec_bytes = prec == 64 ? 32 : (prec == 32 ? 16 : 8);
    const int dims[3] = {nx, ny, nz};
    const int parts[3] = {px, py, pz};
    for (int a = 0; a < 3; ++a) cuts[a] = split_axis(dims[a], parts[a]);

    std::map<std::tuple<int, int, int>, int> shape_id;
    std::vector<int> lvl_tab;
    int bxy_all = 1;
    R.subs.clear();
    R.shapes.clear();
    long long foff = 0;
    int maxw_all = 0, ycap = 0, lcap = 0, gcap = 0;      // cell by cell
    int maxwb = 0, ycapb = 0, lcapb = 0, gcapb = 0;      // blocks of 2 x 2 cells
    int npen_all = 1;
    size_t fac_smem = 0;
    for (int kz = 0; kz < pz; ++kz)
        for (int jy = 0; jy < py; ++jy)
            for (int ix = 0; ix < px; ++ix) {
                const int p[3] = {ix, jy, kz};
                int o0[3], o1[3], e0[3], e1[3];
                for (int a = 0; a < 3; ++a) {
                    o0[a] = cuts[a][p[a]];
                    o1[a] = cuts[a][p[a] + 1];
                    e0[a] = dims[a] > 1 ? std::max(o0[a] - overlap, 0) : 0;
                    e1[a] = dims[a] > 1 ? std::min(o1[a] + overlap, dims[a]) : 1;
                }
                const int bx = e1[0] - e0[0], by = e1[1] - e0[1], bz = e1[2] - e0[2];
                if (bx > 256 || by > 256 || bz > 256) return RAS_EINVAL;
                const int ncell = bx * by * bz;
                if (ncell > 16384) return RAS_EINVAL;  // shared-memory pivots in the factor
                auto key = std::make_tuple(bx, by, bz);
                auto it = shape_id.find(key);
                int sid = it == shape_id.end() ? -1 : it->second;
                if (sid < 0) {
                    sid = (int)R.shapes.size();
                    shape_id[key] = sid;
                    ShapeInfo sh{};
                    sh.bx = bx; sh.by = by; sh.bz = bz; sh.ncell = ncell;
                    // level schedule: cells (FP64 factors) or blocks of 2 x 2 cells, by
                    // I + J + k, inside a level by J + k, then J (the factorisation and the
                    // sweeps compute positions from this order)
                    const bool cells = prec == 64;
                    sh.mx = (bx + 1) / 2; sh.my = (by + 1) / 2;
                    sh.nblk = sh.mx * sh.my * bz;
                    // odd step between a level's neighbouring blocks (J + 1, k - 1)
                    sh.mp = sh.mx * sh.my;
                    if ((sh.mx - sh.mp) % 2 == 0) ++sh.mp;
                    sh.guard = std::max(1, std::max(sh.my > 1 ? sh.mx : 0, bz > 1 ? sh.mp : 0));
                    const int dx = cells ? bx : sh.mx, dy = cells ? by : sh.my, dz = bz;
                    sh.nlev = dx + dy + dz - 2;
                    while (cidx_tab.size() % 4) cidx_tab.push_back(0);
                    sh.cell_off = (int)cidx_tab.size();
                    sh.lvl_off = (int)lvl_tab.size();
                    int pos = 0, maxw = 0, maxc = 0;
                    for (int l = 0; l < sh.nlev; ++l) {
                        lvl_tab.push_back(pos);
                        const int p0 = pos;
                        for (int d = std::max(0, l - dx + 1); d <= std::min(l, dy + dz - 2); ++d)
                            for (int j = std::max(0, d - dz + 1); j <= std::min(d, dy - 1); ++j, ++pos)
                                cidx_tab.push_back(cells ? l - d + dx * (j + dy * (d - j)) : (l - d) | j << 8 | (d - j) << 16);
                        maxw = std::max(maxw, pos - p0);
                    }
                    lvl_tab.push_back(pos);
                    sh.maxw = maxw;
                    for (int l = 0; l < bx + by + bz - 2; ++l) {     // widest level of cells
                        int w = 0;
                        for (int d = std::max(0, l - bx + 1); d <= std::min(l, by + bz - 2); ++d)
                            w += std::min(d, by - 1) - std::max(0, d - bz + 1) + 1;
                        maxc = std::max(maxc, w);
                    }
                    maxw_all = std::max(maxw_all, maxc);
                    ycap = std::max(ycap, ncell);
                    gcap = std::max(gcap, bx * by);
                    lcap = std::max(lcap, bx + by + bz - 1);
                    maxwb = std::max(maxwb, maxw);
                    ycapb = std::max(ycapb, sh.mp * bz);
                    bxy_all = std::max(bxy_all, bx * by);
                    lcapb = std::max(lcapb, sh.nlev + 1);
                    gcapb = std::max(gcapb, sh.guard);
                    const int npen = pencil_count(bx, by, bz);
                    npen_all = std::max(npen_all, npen);
                    fac_smem = std::max(fac_smem, 4 * (size_t)npen * sizeof(double) + 2 * (size_t)sh.nlev * sizeof(int));
                    R.shapes.push_back(sh);
                    sid = (int)R.shapes.size() - 1;
                }
                SubInfo si{};
                si.e0x = e0[0]; si.e0y = e0[1]; si.e0z = e0[2];
                si.shape = sid;
                si.ox0 = o0[0] - e0[0]; si.oy0 = o0[1] - e0[1]; si.oz0 = o0[2] - e0[2];
                si.ox1 = o1[0] - e0[0]; si.oy1 = o1[1] - e0[1]; si.oz1 = o1[2] - e0[2];
                si.foff = foff;
                foff += prec == 64 ? (ncell + 3) & ~3 : 4 * (long long)R.shapes[sid].nblk;
                R.ncell_total += ncell;
                R.nown += (long long)(o1[0] - o0[0]) * (o1[1] - o0[1]) * (o1[2] - o0[2]);
                R.subs.push_back(si);
            }
    R.nsub = (int)R.subs.size();
    R.nshape = (int)R.shapes.size();
    // every overlapped box must lie inside the grid and match its shape
    for (const SubInfo &si : R.subs) {
        if (si.shape < 0 || si.shape >= R.nshape) return RAS_EINVAL;
        const ShapeInfo &sh = R.shapes[si.shape];
        if (si.e0x < 0 || si.e0y < 0 || si.e0z < 0 || si.e0x + sh.bx > nx ||
            si.e0y + sh.by > ny || si.e0z + sh.bz > nz)
            return RAS_EINVAL;
        if (si.ox0 < 0 || si.oy0 < 0 || si.oz0 < 0 || si.ox1 > sh.bx || si.oy1 > sh.by ||
            si.oz1 > sh.bz)
            return RAS_EINVAL;
    }
    R.nrec = foff;
    R.ycap_cells = (ycap + 3) & ~3;
    R.gcap_cells = (gcap + 3) & ~3;
    R.lcap_cells = (lcap + 3) & ~3;
    const bool cells = prec == 64;
    R.ycap = cells ? R.ycap_cells : (ycapb + 3) & ~3;
    R.gcap = cells ? R.gcap_cells : gcapb;
    R.lcap = cells ? R.lcap_cells : (lcapb + 3) & ~3;
    R.maxw = maxw_all;
    R.maxwb = maxwb;
    R.bxy = bxy_all;
    R.h_lvl = lvl_tab;
    R.smem_factor = fac_smem;
    R.fac_block = (npen_all + 31) & ~31;
    return RAS_OK;
}

int ras1_setup(Ras1 &R, int nx, int ny, int nz, int px, int py, int pz, int overlap, int prec,
               int kind) {
    const int dims[3] = {nx, ny, nz}, parts[3] = {px, py, pz};
    std::vector<int> cuts[3], cidx_tab, chunk_tab;
    RAS_TRY(ras1_geometry(R, nx, ny, nz, px, py, pz, overlap, prec, kind, cuts, cidx_tab));
    RAS_TRY(schedule_tables(R, 0, 0, chunk_tab));
    const std::vector<int> &lvl_tab = R.h_lvl;
    if (R.smem_apply > 227 * 1024 || R.smem_factor > 227 * 1024) return RAS_EINVAL;
    RAS_TRY(dalloc(&R.d_boxes, R.subs.size()));
    RAS_TRY(dalloc(&R.d_subs, R.subs.size()));
    RAS_TRY(dalloc(&R.d_shapes, R.shapes.size()));
    RAS_TRY(dalloc(&R.d_lvl, lvl_tab.size()));
    RAS_TRY(dalloc(&R.d_chunk, chunk_tab.size()));
    RAS_TRY(dalloc(&R.d_cidx, cidx_tab.size() + 16));
    RAS_TRY(dalloc(&R.d_err, 2));
    unsigned char *fw = nullptr, *bw = nullptr;
    RAS_TRY(dalloc(&fw, (size_t)R.nrec * R.rec_bytes + 64));
    RAS_TRY(dalloc(&bw, (size_t)R.nrec * R.rec_bytes + 64));
    R.d_fwd = fw; R.d_bwd = bw;
    RAS_CK(cudaMemcpy(R.d_subs, R.subs.data(), R.subs.size() * sizeof(SubInfo), cudaMemcpyHostToDevice));
    RAS_CK(cudaMemcpy(R.d_shapes, R.shapes.data(), R.shapes.size() * sizeof(ShapeInfo),
                      cudaMemcpyHostToDevice));
    RAS_TRY(upload_boxes(R));
    RAS_CK(cudaMemcpy(R.d_lvl, lvl_tab.data(), lvl_tab.size() * sizeof(int), cudaMemcpyHostToDevice));
    RAS_CK(cudaMemcpy(R.d_chunk, chunk_tab.data(), chunk_tab.size() * sizeof(int),
                      cudaMemcpyHostToDevice));
    RAS_CK(cudaMemset(R.d_cidx, 0, (cidx_tab.size() + 16) * sizeof(int)));
    RAS_CK(cudaMemcpy(R.d_cidx, cidx_tab.data(), cidx_tab.size() * sizeof(int), cudaMemcpyHostToDevice));
    RAS_CK(cudaMemset(R.d_err, 0, 2 * sizeof(int)));
    RAS_CK(cudaMemset(R.d_fwd, 0, (size_t)R.nrec * R.rec_bytes + 64));
    RAS_CK(cudaMemset(R.d_bwd, 0, (size_t)R.nrec * R.rec_bytes + 64));
    if (prec == 64) { RAS_TRY((set_apply_attr<64, false>())); RAS_TRY(set_factor_attr<64>()); }
    if (prec == 32) { RAS_TRY((set_apply_attr<32, false>())); RAS_TRY(set_factor_attr<32>()); }
    if (prec == 16) { RAS_TRY((set_apply_attr<16, false>())); RAS_TRY(set_factor_attr<16>()); }
    if (kind != 1) {
        // per axis and coordinate, the (contiguous) range of parts whose overlapped
        // boxes cover it; box solutions are kept per record offset
        R.parts[0] = px; R.parts[1] = py; R.parts[2] = pz;
        for (int a = 0; a < 3; ++a) {
            std::vector<int> lo(dims[a], parts[a]), hi(dims[a], -1);
            for (int q = 0; q < parts[a]; ++q) {
                const int e0 = std::max(cuts[a][q] - overlap, 0);
                const int e1 = std::min(cuts[a][q + 1] + overlap, dims[a]);
                for (int i = e0; i < e1; ++i) { lo[i] = std::min(lo[i], q); hi[i] = std::max(hi[i], q); }
            }
            RAS_TRY(dalloc(&R.d_clo[a], lo.size()));
            RAS_TRY(dalloc(&R.d_chi[a], hi.size()));
            RAS_CK(cudaMemcpy(R.d_clo[a], lo.data(), lo.size() * sizeof(int), cudaMemcpyHostToDevice));
            RAS_CK(cudaMemcpy(R.d_chi[a], hi.data(), hi.size() * sizeof(int), cudaMemcpyHostToDevice));
        }
        RAS_TRY(dalloc(&R.zbuf, (size_t)R.nrec));
        RAS_CK(cudaMemset(R.zbuf, 0, (size_t)R.nrec * sizeof(double)));
    }
    return RAS_OK;
}

void ras1_free(Ras1 &R) {
    dfree(R.d_subs); dfree(R.d_boxes); dfree(R.d_shapes); dfree(R.d_lvl); dfree(R.d_chunk);
    dfree(R.d_cidx); dfree(R.d_err);
    if (R.d_fwd) cudaFree(R.d_fwd);
    if (R.d_bwd) cudaFree(R.d_bwd);
    R.d_fwd = R.d_bwd = nullptr;
    dfree(R.zbuf);
    for (int a = 0; a < 3; ++a) { dfree(R.d_clo[a]); dfree(R.d_chi[a]); }
}

int ras1_factor(Ras1 &R, const Stencil7 &A, cudaStream_t st) {
    FactorParams P;
    ras1_factor_params(R, A, P);
    if (R.prec == 64) k_ras_factor<64><<<R.nsub, R.fac_block, R.smem_factor, st>>>(P);
    else if (R.prec == 32) k_ras_factor<32><<<R.nsub, R.fac_block, R.smem_factor, st>>>(P);
    else k_ras_factor<16><<<R.nsub, R.fac_block, R.smem_factor, st>>>(P);
    RAS_LAUNCHED();
    return RAS_OK;
}

void ras1_factor_params(const Ras1 &R, const Stencil7 &A, FactorParams &P) {
    P.subs = R.d_subs; P.shapes = R.d_shapes; P.lvl = R.d_lvl;
    P.A = A; P.fwd = R.d_fwd; P.bwd = R.d_bwd;
    P.nx = R.nx; P.ny = R.ny; P.nz = R.nz; P.err = R.d_err;
}

int ras1_factor_batch(const FactorParams *d_inst, const int *d_box_inst, const int *d_box_local,
                      const unsigned char *d_active, int nbox, int prec, int block, size_t smem, cudaStream_t st) {
    if (nbox <= 0) return RAS_OK;
    if (prec == 64) k_ras_factor_batch<64><<<nbox, block, smem, st>>>(d_inst, d_box_inst, d_box_local, d_active);
    else if (prec == 32) k_ras_factor_batch<32><<<nbox, block, smem, st>>>(d_inst, d_box_inst, d_box_local, d_active);
    else k_ras_factor_batch<16><<<nbox, block, smem, st>>>(d_inst, d_box_inst, d_box_local, d_active);
    RAS_LAUNCHED();
    return RAS_OK;
}

int ras1_status(int word) { return word == 0 ? RAS_OK : (word == APPLY_TIMEOUT ? RAS_ETIMEOUT : RAS_EZEROPIVOT); }

int ras1_set_kernel(Ras1 &R, int kernel) {
    if (kernel != 0 && kernel != 1) return RAS_EINVAL;
    if (kernel == 1) {
        if (R.kind != 1 || R.prec == 64) return RAS_EINVAL;
        for (const ShapeInfo &sh : R.shapes)
            if (sh.by * sh.bz > 1024) return RAS_EINVAL;
    }
    R.kernel = kernel;
    return RAS_OK;
}


int ras1_limit_ready(int prec) {
    return prec == 64 ? RAS_OK : (prec == 32 ? set_apply_attr<32, true>() : set_apply_attr<16, true>());
}

int ras1_polls() { return (int)std::min<long long>(barrier_polls(), APPLY_POLLS); }

void ras1_apply_params(const Ras1 &R, ApplyParams &P) {
    P = ApplyParams{};
    P.subs = R.d_subs; P.shapes = R.d_shapes; P.boxes = R.d_boxes; P.lvl = R.d_lvl; P.chunk = R.d_chunk;
    P.cidx = R.d_cidx;
    P.fwd = (const unsigned char *)R.d_fwd; P.bwd = (const unsigned char *)R.d_bwd;
    P.nx = R.nx; P.ny = R.ny; P.nz = R.nz; P.accumulate = 0;
    P.ycap = R.ycap; P.gcap = R.gcap; P.lcap = R.lcap; P.chunk_cells = R.chunk_cells;
    P.steps = reinterpret_cast<const int4 *>(R.d_chunk); P.err = R.d_err;
    P.kind = R.kind; P.zbuf = R.zbuf;
}

int ras1_apply_batch(const BatchApply &B, int grid, int prec, int block, size_t smem, cudaStream_t st) {
    if (grid <= 0 || B.nitems <= 0) return RAS_OK;
    RAS_CK(cudaMemsetAsync(B.qcount, 0, sizeof(int), st));
    auto kern = prec == 64 ? k_ras_apply_batch<64, false>
              : prec == 32 ? (B.polls > 0 ? k_ras_apply_batch<32, true> : k_ras_apply_batch<32, false>)
                           : (B.polls > 0 ? k_ras_apply_batch<16, true> : k_ras_apply_batch<16, false>);
    kern<<<grid, block, smem, st>>>(B);
    RAS_LAUNCHED();
    return RAS_OK;
}

int ras1_batch_grid(int prec, int block, size_t smem, int nitems, int *grid) {
    int dev = 0, sms = 0, per = 0;
    RAS_CK(cudaGetDevice(&dev));
    RAS_CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    if (prec == 64) RAS_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_ras_apply_batch<64, false>, block, smem));
    else if (prec == 32) RAS_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_ras_apply_batch<32, false>, block, smem));
    else RAS_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_ras_apply_batch<16, false>, block, smem));
    if (per < 1) return RAS_EINVAL;
    *grid = std::min(nitems, sms * per);
    return RAS_OK;
}

int ras1_apply(Ras1 &R, const double *r, double *z, int accumulate, cudaStream_t st) {
    ApplyParams P;
    ras1_apply_params(R, P);
    P.r = r; P.z = z; P.accumulate = accumulate;
    P.polls = ras1_polls();
    if (P.polls > 0) RAS_TRY(ras1_limit_ready(R.prec));
    auto kern = R.prec == 64 ? k_ras_apply<64, false>
              : R.prec == 32 ? (P.polls > 0 ? k_ras_apply<32, true> : k_ras_apply<32, false>)
                             : (P.polls > 0 ? k_ras_apply<16, true> : k_ras_apply<16, false>);
    kern<<<R.nsub, R.launch, R.smem_apply, st>>>(P);
    RAS_LAUNCHED();
    if (R.kind != 1) {
        SumParams Q;
        Q.subs = R.d_subs; Q.shapes = R.d_shapes;
        for (int a = 0; a < 3; ++a) { Q.clo[a] = R.d_clo[a]; Q.chi[a] = R.d_chi[a]; Q.parts[a] = R.parts[a]; }
        Q.nx = R.nx; Q.ny = R.ny; Q.nz = R.nz;
        Q.zbuf = R.zbuf; Q.z = z; Q.accumulate = accumulate;
        const int grid = (int)std::min<long long>(((long long)R.N + 255) / 256, 152LL * 16);
        k_ras_sum<<<grid, 256, 0, st>>>(Q);
        RAS_LAUNCHED();
    }
    return RAS_OK;
}

// Algorithmic bytes of one apply: the ILU(0) factors once (7 values per
// overlapped cell: 3 lower, 3 upper off-diagonals and the inverse pivot, at the
// storage precision), r read once and z written once in FP64. (The kernel's
// records carry the inverse pivot twice and r is re-read over the overlap;
// those bytes are not counted.)
double ras1_bytes(const Ras1 &R) {
    const double val = R.prec == 64 ? 8.0 : (R.prec == 32 ? 4.0 : 2.0);
    return 7.0 * val * (double)R.ncell_total + 16.0 * (double)R.N;
}

}  // namespace ras

using namespace ras;

extern "C" int ras_apply_steps(int nx, int ny, int nz, const ras_opts *o, int chunk_cells, int *tab, int cap, int *len) {
    if (!o || !len || nx < 1 || ny < 1 || nz < 1 || chunk_cells < 0 || o->ilu_k != 0) return RAS_EINVAL;
    if (o->factor_prec != 32 && o->factor_prec != 16) return RAS_EINVAL;
    Ras1 R;
    std::vector<int> cuts[3], cidx_tab, steps;
    RAS_TRY(ras1_geometry(R, nx, ny, nz, o->px, o->py, o->pz, o->overlap, o->factor_prec, o->ras_type, cuts, cidx_tab));
    RAS_TRY(schedule_tables(R, chunk_cells, 0, steps));
    std::vector<int> t{(int)R.ring_bytes, R.rec_bytes, R.nshape};
    for (const ShapeInfo &sh : R.shapes) {
        t.insert(t.end(), {sh.bx, sh.by, sh.bz, sh.nchunk});
        t.insert(t.end(), steps.begin() + 4 * sh.chunk_off, steps.begin() + 4 * (sh.chunk_off + sh.nchunk + 1));
    }
    *len = (int)t.size();
    if (!tab || cap < *len) return RAS_EINVAL;
    std::copy(t.begin(), t.end(), tab);
    return RAS_OK;
}
