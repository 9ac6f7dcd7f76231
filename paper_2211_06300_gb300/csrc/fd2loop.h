// 2D time loops with the wave states held on chip.
//
// The per-step kernel (fd2d.cu) reads u_n, u_{n-1} and c and writes u_{n+1} through L2 / HBM at
// every step and pays a launch and a grid-wide dependency per step.  Here one cooperative launch
// runs a whole run of steps: each CTA (one per SM) owns a tile of one shot and keeps u_n and
// u_{n-1} of the tile, with a 4-cell halo, in shared memory for all of them (u_{n+1} overwrites
// u_{n-1} in place).  What crosses the chip per step is the 4-cell rim of each tile and the
// streams the step itself is about (the extended source, CG vectors, stashes, outputs).
//
// Tiles.  A shot's plane is cut into 4 x 4 cell blocks (the halo is 4 cells, so a tile's rim is
// whole blocks); gx x gz tiles per shot are near-equal ranges of block columns and block rows.
// The stencil is a star: a tile exchanges with at most four neighbours and needs no corners.
//
// Exchange.  A thread that computes a rim cell stores it, with the step's tag, into the inbox of
// the neighbour as 8-byte (value, tag) packets (FP64: two packets per value); the neighbour's
// communication warps poll the packets themselves.  An 8-byte access is single-copy atomic, so a
// packet whose tag matches carries its value, and no fence, flag or second round trip is needed:
// 0.6-0.8 us per step over 152 CTAs against 2.0-2.8 us for data + fence + flag + acquire (both
// measured with 0.25-4 KB per neighbour).  Inboxes alternate with the step's parity; a tile
// writes parity p again only after it has its neighbour's packets of the step between, which the
// neighbour sent after it had read parity p.  Tags continue over launches from an epoch word
// that the last CTA of a launch advances, so nothing has to be cleared between launches and a
// replayed CUDA graph is safe.  Rim items come first in every step, so that with more than one
// item per thread the packets travel while the interior is computed.
//
// Every CTA waits on others, so the launch is cooperative (all CTAs resident) and every wait is
// bounded: a wait that runs out sets the device error word and ends the CTA.
//
// Arithmetic: operation for operation that of fd2_step_kernel, so both give the same bits.
#pragma once

#include <type_traits>

#include "esi_internal.h"
#include "pairs.h"

namespace esi {
namespace loop2 {

constexpr double W0 = -205.0 / 72.0, W1 = 8.0 / 5.0, W2 = -1.0 / 5.0, W3 = 8.0 / 315.0,
                 W4 = -1.0 / 560.0;
constexpr int SMP_T = 32;     // of the communication threads: those that sample the receivers
constexpr int INJ_U = 4;      // trace values a thread has in flight for the point sources
constexpr int PF_AHEAD = 2;   // steps by which the streams' L2 prefetch runs ahead

// The cells of one thread along x: four FP32 as two pairs in the arithmetic of the step kernels
// (pairs.h; each lane rounds as the scalar instruction does), or one FP64.
template <typename T>
struct Row4;
template <>
struct __align__(16) Row4<float> {
    static constexpr int CW = 4;
    unsigned long long p[2];
};
template <>
struct Row4<double> {
    static constexpr int CW = 1;
    double p[1];
};

using PF = Pk<float>;
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
    const float v[2] = {x, y};
    return PF::pack(v);
}
__device__ __forceinline__ float lo2(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi2(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }

using RF = Row4<float>;
using RD = Row4<double>;
__device__ __forceinline__ RF add(const RF &a, const RF &b) { return {{PF::add(a.p[0], b.p[0]), PF::add(a.p[1], b.p[1])}}; }
__device__ __forceinline__ RF sub(const RF &a, const RF &b) { return {{PF::sub(a.p[0], b.p[0]), PF::sub(a.p[1], b.p[1])}}; }
__device__ __forceinline__ RF mul(const RF &a, const RF &b) { return {{PF::mul(a.p[0], b.p[0]), PF::mul(a.p[1], b.p[1])}}; }
__device__ __forceinline__ RF fma(const RF &a, const RF &b, const RF &c) {
    return {{PF::fma(a.p[0], b.p[0], c.p[0]), PF::fma(a.p[1], b.p[1], c.p[1])}};
}
__device__ __forceinline__ RF splat(float v) { return {{pack2(v, v), pack2(v, v)}}; }
__device__ __forceinline__ float at(const RF &a, int i) { return (i & 1) ? hi2(a.p[i >> 1]) : lo2(a.p[i >> 1]); }
__device__ __forceinline__ void put(RF &a, int i, float v) {
    a.p[i >> 1] = (i & 1) ? pack2(lo2(a.p[i >> 1]), v) : pack2(v, hi2(a.p[i >> 1]));
}
__device__ __forceinline__ RF ldr(const float *p) {
    const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(p);
    return {{q.x, q.y}};
}
__device__ __forceinline__ void str(float *p, const RF &a) {
    *reinterpret_cast<ulonglong2 *>(p) = make_ulonglong2(a.p[0], a.p[1]);
}
__device__ __forceinline__ RD add(const RD &a, const RD &b) { return {{__dadd_rn(a.p[0], b.p[0])}}; }
__device__ __forceinline__ RD sub(const RD &a, const RD &b) { return {{__dsub_rn(a.p[0], b.p[0])}}; }
__device__ __forceinline__ RD mul(const RD &a, const RD &b) { return {{__dmul_rn(a.p[0], b.p[0])}}; }
__device__ __forceinline__ RD fma(const RD &a, const RD &b, const RD &c) { return {{__fma_rn(a.p[0], b.p[0], c.p[0])}}; }
__device__ __forceinline__ RD splat(double v) { return {{v}}; }
__device__ __forceinline__ double at(const RD &a, int) { return a.p[0]; }
__device__ __forceinline__ void put(RD &a, int, double v) { a.p[0] = v; }
__device__ __forceinline__ RD ldr(const double *p) { return {{*p}}; }
__device__ __forceinline__ void str(double *p, const RD &a) { *p = a.p[0]; }

// The x neighbours of a thread's cells: what they need besides the cells themselves, and the
// sum of the two at distance D (pairs that straddle the packing are added as scalars).
template <typename T>
struct Side;
template <>
struct Side<float> {
    RF l, r;
    __device__ __forceinline__ Side(const float *p) : l(ldr(p - 4)), r(ldr(p + 4)) {}
    template <int D>
    __device__ __forceinline__ RF sum(const RF &c) const {
        if constexpr (D == 4) return add(l, r);
        if constexpr (D == 2) return {{PF::add(l.p[1], c.p[1]), PF::add(c.p[0], r.p[0])}};
        if constexpr (D == 1)
            return {{pack2(hi2(l.p[1]) + hi2(c.p[0]), lo2(c.p[0]) + lo2(c.p[1])),
                     pack2(hi2(c.p[0]) + hi2(c.p[1]), lo2(c.p[1]) + lo2(r.p[0]))}};
        return {{pack2(hi2(l.p[0]) + hi2(c.p[1]), lo2(l.p[1]) + lo2(r.p[0])),
                 pack2(hi2(l.p[1]) + hi2(r.p[0]), lo2(c.p[0]) + lo2(r.p[1]))}};
    }
};
template <>
struct Side<double> {
    double l[4], r[4];
    __device__ __forceinline__ Side(const double *p) {
#pragma unroll
        for (int i = 0; i < 4; ++i) l[i] = p[-1 - i], r[i] = p[1 + i];
    }
    template <int D>
    __device__ __forceinline__ RD sum(const RD &) const {
        return {{__dadd_rn(l[D - 1], r[D - 1])}};
    }
};

__device__ __forceinline__ void st_packets(ulonglong2 *p, unsigned long long x,
                                           unsigned long long y) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}
__device__ __forceinline__ ulonglong2 ld_packets(const ulonglong2 *p) {
    ulonglong2 r;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(r.x), "=l"(r.y) : "l"(p) : "memory");
    return r;
}
// the 16-byte entries of one tile edge cell group: FP32 two cells, FP64 one cell
__device__ __forceinline__ void send(ulonglong2 *p, unsigned tag, float a, float b) {
    const unsigned long long t = (unsigned long long)tag << 32;
    st_packets(p, t | __float_as_uint(a), t | __float_as_uint(b));
}
__device__ __forceinline__ void send(ulonglong2 *p, unsigned tag, double a) {
    const unsigned long long t = (unsigned long long)tag << 32, v = __double_as_longlong(a);
    st_packets(p, t | (v & 0xffffffffull), t | (v >> 32));
}
__device__ __forceinline__ bool tagged(const ulonglong2 &e, unsigned tag) {
    return (unsigned)(e.x >> 32) == tag && (unsigned)(e.y >> 32) == tag;
}
__device__ __forceinline__ void unpack(const ulonglong2 &e, float *dst) {
    *reinterpret_cast<float2 *>(dst) =
        make_float2(__uint_as_float((unsigned)e.x), __uint_as_float((unsigned)e.y));
}
__device__ __forceinline__ void unpack(const ulonglong2 &e, double *dst) {
    *dst = __longlong_as_double((long long)((e.x & 0xffffffffull) | (e.y << 32)));
}

// gamma of the sponge coefficient kappa
template <typename T>
__device__ __forceinline__ T gamma_of(T kap) {
    const T al = T(1) / (T(1) + kap);
    return (T(1) - kap) * al;
}

__device__ __forceinline__ void prefetch_l2(const void *p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Threads: g.nc compute threads, then g.nm communication threads, of which the last SMP_T
// sample.  A compute thread owns a column of cells (Row4<T>::CW wide) in every nseg-th row of the
// tile, counted from the bottom rim on, so that both rims along z are sent first; lanes run along
// x in groups of g.lanes, so that a group's shared-memory accesses are one conflict-free
// wavefront.  The row's global inputs (alpha c and the step's streams) are fetched a row, or a
// step, ahead of their use.
//
// What bounds it: with one or two rows per thread a step is the exchange (0.6-0.8 us), one row's
// dependence chain and two block barriers' worth of waiting, 1.3-1.9 us in FP32 against 3.1 us
// for a launch per step (one shot of 101 x 101 .. 801 x 241); in FP64 the two lanes per clock of
// an SM's FP64 units (101 x 101: 2.0 us against 22.4 us on the eight SMs that its eight 64 x 32
// tiles occupy).  With more rows per thread in FP32 the 14 16-byte shared-memory accesses per row
// (56 cycles per warp) and the chains of too few warps cost more than L2 does in the per-step
// kernel (16 shots of 801 x 241: 10 us against 9.8, 7.0 in two chains); registers are what a
// wider window or more warps would take, and a spill there goes to L2 (the tiles leave no L1),
// which measured worse.
template <typename T, unsigned F>
__global__ void __launch_bounds__(LOOP_THREADS, 1)
    fd2_loop_kernel(const __grid_constant__ StepArgs<T> a, const __grid_constant__ LoopArgs<T> g) {
    using V = Row4<T>;
    constexpr int CW = V::CW;
    constexpr int EPR = sizeof(T) == 4 ? 2 : 4;    // inbox entries per 4-cell row segment
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ double red[LOOP_THREADS / 32];
    __shared__ long long boxes[4];   // the neighbours' inboxes: above, below, left, right
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int tiles = g.gx * g.gz;
    const int sl = blockIdx.x / tiles, tile = blockIdx.x - sl * tiles;
    const int s = g.s0 + sl;
    const int tz = tile / g.gx, tx = tile - tz * g.gx;
    const int q0 = loop_part(tx, g.gx, g.qx), nbx = loop_part(tx + 1, g.gx, g.qx) - q0;
    const int r0 = loop_part(tz, g.gz, g.gr), nbz = loop_part(tz + 1, g.gz, g.gr) - r0;
    const int X0 = 4 * q0, Z0 = 4 * r0, cols = 4 * nbx, rows = 4 * nbz;
    const int P = cols + 8, H = rows + 8;
    const int hr = min(rows, a.nz - Z0);   // rows inside the grid
    const unsigned tag0 = *reinterpret_cast<volatile unsigned *>(g.sync);
    T *buf0 = reinterpret_cast<T *>(smraw), *buf1 = buf0 + (size_t)P * H;
    T *sgx = buf1 + (size_t)P * H, *sgz = sgx + cols;   // gamma by column and by row
    // sponge rows at the top / bottom of the tile, sponge columns (whole blocks) at its sides
    const int nzt = min(max(g.nbz0 - Z0, 0), hr), nzb = min(max(Z0 + hr - g.nbz1, 0), hr - nzt);
    const int nxl = min(max((g.nbx0 - X0 + 3) / 4 * 4, 0), cols);
    const int nxr = min(max(X0 + cols - g.nbx1 / 4 * 4, 0), cols - nxl);
    const int ncs = nxl + nxr;
    T *corner = sgz + rows;                              // gamma where both apply [nzt + nzb][ncs]
    T *patch = corner + (nzt + nzb) * ncs;
    double dot = 0.0;
    if (!a.active || a.active[s]) {
        const bool hasT = tz > 0, hasB = tz + 1 < g.gz, hasL = tx > 0, hasR = tx + 1 < g.gx;
        int np = 0, c0 = 0, nci = 0, pb = 0;
        if constexpr ((F & F_PT) != 0) {
            const int gt = s * tiles + tile;
            pb = g.patch_ptr[gt];
            np = g.patch_ptr[gt + 1] - pb;
            c0 = g.inj_ptr[gt];
            nci = g.inj_ptr[gt + 1] - c0;
        }
        LoopInj<T> *inj = reinterpret_cast<LoopInj<T> *>(patch + 32 * np);   // [nci]
        unsigned short *map = reinterpret_cast<unsigned short *>(inj + nci);  // [nbx * nbz]
        T *st0 = const_cast<T *>(a.cur) + (long long)s * a.sst, *st1 = a.po + (long long)s * a.sst;

        // ---- prologue: states (tile and halo), sponge profiles, injection tables
        {
            const int nq = nbx + 2;
            for (int i = tid; i < nq * H; i += nthr) {
                const int r = i / nq, q = i - r * nq;
                const int gz = Z0 + r - 4, gx = X0 + 4 * (q - 1);
                T *d0 = buf0 + r * P + 4 * q, *d1 = buf1 + r * P + 4 * q;
                if (gz >= 0 && gz < a.nz && gx >= 0 && gx < a.nx) {
                    const long long gi = (long long)gz * a.px + gx;
#pragma unroll
                    for (int h = 0; h < 4; h += 16 / (int)sizeof(T)) {
                        *reinterpret_cast<uint4 *>(d0 + h) = *reinterpret_cast<const uint4 *>(st0 + gi + h);
                        *reinterpret_cast<uint4 *>(d1 + h) = *reinterpret_cast<const uint4 *>(st1 + gi + h);
                    }
                } else {
#pragma unroll
                    for (int h = 0; h < 4; ++h) d0[h] = d1[h] = T(0);
                }
            }
        }
        for (int i = tid; i < cols; i += nthr) sgx[i] = gamma_of(a.kx[X0 + i]);   // px is a multiple of 32
        for (int i = tid; i < rows; i += nthr) sgz[i] = i < hr ? gamma_of(a.kz[Z0 + i]) : T(1);
        for (int i = tid; i < (nzt + nzb) * ncs; i += nthr) {
            const int r = i / ncs, c = i - r * ncs;
            corner[i] = gamma_of(a.kz[Z0 + (r < nzt ? r : r - nzt + hr - nzb)] +
                                 a.kx[X0 + (c < nxl ? c : c - nxl + cols - nxr)]);
        }
        const int me = blockIdx.x, selfS = nbx * 4 * EPR;
        if (tid == 0) {   // sides of an inbox: [from above][from below][from the left][from the right]
            const int nbl = hasL ? q0 - loop_part(tx - 1, g.gx, g.qx) : 0;
            const int nbr = hasR ? loop_part(tx + 2, g.gx, g.qx) - (q0 + nbx) : 0;
            boxes[0] = (long long)(me - g.gx) * g.istride + selfS;
            boxes[1] = (long long)(me + g.gx) * g.istride;
            boxes[2] = (long long)(me - 1) * g.istride + 2 * nbl * 4 * EPR + rows * EPR;
            boxes[3] = (long long)(me + 1) * g.istride + 2 * nbr * 4 * EPR;
        }
        if constexpr ((F & F_PT) != 0) {
            for (int i = tid; i < 32 * np; i += nthr) patch[i] = T(0);
            for (int i = tid; i < nbx * nbz; i += nthr) map[i] = 0;
            for (int i = tid; i < nci; i += nthr) inj[i] = g.inj[c0 + i];
            __syncthreads();
            for (int i = tid; i < np; i += nthr) map[g.patch_blk[pb + i]] = (unsigned short)(i + 1);
        }
        __syncthreads();
        // The point-source cells at trace time t into the patch set p, by the `n` threads that call
        // this as me = 0 .. n - 1.  A cell's contributions are added in list order.  An entry is the
        // latency of L2 or HBM, so a thread's loads go out together.  Short lists (a cell a thread,
        // up to INJ_U contributions each) go straight to the cells.  Of long ones, which can hold
        // thousands of entries a tile, all threads load entries, INJ_U at a time each; where a cell
        // has several contributions, a thread per cell then adds them up from shared memory.  (2000
        // receivers on a line, back-propagation, us per step, with one load at a time by the cell's
        // thread and so: one shot of 101 x 101 33 and 2.9, 20 shots of 97 x 130 68 and 4.7; the
        // per-step kernel 7.7 and 8.1.)
        const bool several = nci > 0 && inj[nci - 1].pos == LOOP_NONE;
        auto end_of = [&](int i) {
            return i + 1 < nci && inj[i + 1].pos != LOOP_NONE ? (int)inj[i + 1].first : nci;
        };
        bool longer = nci > g.nm - SMP_T && inj[g.nm - SMP_T].pos != LOOP_NONE;
        if (several) {
            bool chain = false;
            for (int i = tid; i < nci && inj[i].pos != LOOP_NONE; i += nthr)
                chain |= end_of(i) - inj[i].first > INJ_U;
            longer |= __syncthreads_or(chain) != 0;
        }
        auto load = [&](int c, int t) { return a.inj_trace[inj[c].off + (long long)t * inj[c].stride]; };
        auto inject = [&](T *p, int t, int me, int n, auto &&sync) {
            if (!longer) {
                if (me >= nci || inj[me].pos == LOOP_NONE) return;
                const int c = several ? inj[me].first : me;
                T v[INJ_U], sum = T(0);
                v[0] = load(c, t);
                if (several) {
                    const int end = end_of(me);
#pragma unroll
                    for (int u = 1; u < INJ_U; ++u) v[u] = c + u < end ? load(c + u, t) : T(0);
                    sum += inj[c].w * v[0];
#pragma unroll
                    for (int u = 1; u < INJ_U; ++u)
                        if (c + u < end) sum += inj[c + u].w * v[u];
                } else {
                    sum += inj[c].w * v[0];
                }
                p[inj[me].pos] = sum;
                return;
            }
            for (int c0 = me; c0 < nci; c0 += INJ_U * n) {
                T v[INJ_U];
#pragma unroll
                for (int u = 0; u < INJ_U; ++u) v[u] = c0 + u * n < nci ? load(c0 + u * n, t) : T(0);
#pragma unroll
                for (int u = 0; u < INJ_U; ++u) {
                    const int c = c0 + u * n;
                    if (c >= nci) break;
                    T sum = T(0);
                    sum += inj[c].w * v[u];
                    if (several) inj[c].v = v[u];
                    else p[inj[c].pos] = sum;
                }
            }
            if (!several) return;
            sync();
            for (int i = me; i < nci && inj[i].pos != LOOP_NONE; i += n) {
                const int end = end_of(i);
                T sum = T(0);
#pragma unroll 4
                for (int c = inj[i].first; c < end; ++c) sum += inj[c].w * inj[c].v;
                p[inj[i].pos] = sum;
            }
        };
        if constexpr ((F & F_PT) != 0) {
            inject(patch, a.tin, tid, nthr, [] { __syncthreads(); });
            __syncthreads();
        }

        ulonglong2 *const in0 = g.inbox, *const in1 = g.inbox + (long long)gridDim.x * g.istride;
        const long long fb = (long long)s * a.fstp, fd = (long long)s * a.fst;

        bool late = false;   // a wait of this CTA ran out
        if (tid < g.nc) {
            // ===================================================== compute threads
            const int gi = tid / g.lanes;
            const int ngx = (cols / CW + g.lanes - 1) / g.lanes;
            const int seg = gi / ngx, nseg = g.nc / (g.lanes * ngx);
            const int lc = ((gi - seg * ngx) * g.lanes + tid % g.lanes) * CW;
            // rows seg, seg + nseg, ... of the tile, counted from its bottom rim on
            const int rot = hasB ? rows - 4 : 0;
            const int nrow = lc < cols && seg < nseg ? (hr - seg + nseg - 1) / nseg : 0;
            const int sb = 4 * P + lc + 4, gb = Z0 * a.px + X0 + lc, gx0 = X0 + lc;
            const bool spx = lc < nxl || lc >= cols - nxr;               // sponge columns
            const bool edge = gx0 + CW > a.nx;                           // cells past the grid
            const bool rimx = (hasL && lc < 4) || (hasR && lc >= cols - 4);
            T cgb = T(0);
            if constexpr ((F & F_CGP) != 0) {
                if (!a.cg_first) cgb = T(a.cg_beta[s]);
            }
            (void)cgb;
            auto row_of = [&](int j) {
                const int lr = seg + j * nseg + rot;
                return lr >= hr ? lr - hr : lr;
            };
            // the global inputs of a row
            struct In {
                V ac, x, y, m;
            };
            In in;
            auto fetch = [&](int kk, int lr, bool with_c) {
                const int dk = kk * g.dn, off = gb + lr * a.px;
                if (with_c) in.ac = ldr(g.ac + off);
                if constexpr ((F & F_EXT) != 0) {
                    const T *e = a.ext + fd + (long long)(a.n + dk) * a.N + ((Z0 + lr) * a.nx + gx0);
                    if (!edge) {
#pragma unroll
                        for (int j = 0; j < CW; ++j) put(in.x, j, e[j]);
                    } else {
#pragma unroll
                        for (int j = 0; j < CW; ++j) put(in.x, j, gx0 + j < a.nx ? e[j] : T(0));
                    }
                }
                if constexpr ((F & F_CGP) != 0) {
                    const long long pl = fb + (long long)(a.n + dk) * a.sst;
                    in.x = ldr(a.cg_r + pl + off);
                    if (!a.cg_first) in.y = ldr(a.cg_p + pl + off);
                    if (a.cg_pc > T(0)) in.m = ldr(a.ipb2 + (long long)s * a.sst + off);
                }
                if constexpr ((F & F_AP) != 0) {
                    in.y = ldr(a.ap_p + fb + (long long)(a.nout + dk) * a.sst + off);
                    in.m = ldr(a.pb2 + (long long)s * a.sst + off);
                }
                if constexpr ((F & F_GRD) != 0)
                    in.y = ldr(a.stash_r + ((long long)(a.slot_r + dk) * a.ns + s) * a.sst + off);
                if constexpr ((F & (F_GRD | F_SAD)) != 0) in.m = ldr(a.grad + (long long)s * a.sst + off);
            };
            in.x = in.y = in.m = in.ac = splat(T(0));
            if (nrow > 0) fetch(0, row_of(0), true);
            for (int k = 0; k < g.steps; ++k) {
                const int dk = k * g.dn;
                const T *A = ((k & 1) ? buf1 : buf0) + sb;
                T *B = ((k & 1) ? buf0 : buf1) + sb;
                (void)dk;
#pragma unroll 1
                for (int j = 0; j < nrow; ++j) {
                    const int lr = row_of(j);
                    const int off = gb + lr * a.px;
                    const T *pA = A + lr * P;
                    T *pB = B + lr * P;
                    // L = 2 w0 u + sum_d w_d (the four neighbours at distance d)
                    const V u = ldr(pA);
                    V L;
                    {
                        const Side<T> sd(pA);
                        L = mul(splat(T(W1)), add(sd.template sum<1>(u), add(ldr(pA - P), ldr(pA + P))));
                        L = fma(splat(T(2.0 * W0)), u, L);
                        L = fma(splat(T(W2)), add(sd.template sum<2>(u), add(ldr(pA - 2 * P), ldr(pA + 2 * P))), L);
                        L = fma(splat(T(W3)), add(sd.template sum<3>(u), add(ldr(pA - 3 * P), ldr(pA + 3 * P))), L);
                        L = fma(splat(T(W4)), add(sd.template sum<4>(u), add(ldr(pA - 4 * P), ldr(pA + 4 * P))), L);
                    }
                    V q = splat(T(0));
                    if constexpr ((F & F_EXT) != 0) q = in.x;
                    if constexpr ((F & F_CGP) != 0) {
                        q = in.x;
                        if (a.cg_pc > T(0)) {   // z = r / (pen B^2)
                            q = mul(q, in.m);
                            if (a.pc_y) {   // + theta x the learned coarse correction
                                const float *yr = a.pc_y +
                                    (((long long)s * a.pc_ng * 16 + a.n + dk) * a.pc_hc + (Z0 + lr) / 2) * a.pc_wc;
                                const T th = T(a.pc_theta[s]);
#pragma unroll
                                for (int c = 0; c < CW; ++c)
                                    if (gx0 + c < a.nx) put(q, c, at(q, c) + th * T(yr[(gx0 + c) / 2]));
                            }
                        }
                        if (!a.cg_first) q = fma(splat(cgb), in.y, q);
                        str(a.cg_p + fb + (long long)(a.n + dk) * a.sst + off, q);
                    }
                    if constexpr ((F & (F_EXT | F_CGP)) != 0) L = fma(splat(a.dx2), q, L);   // S from here on
                    if constexpr ((F & F_PT) != 0) {
                        if (np > 0) {
                            const int pid = map[(lr >> 2) * nbx + (lc >> 2)];
                            if (pid) {
                                const T *pp = patch + (k & 1) * 16 * np + (pid - 1) * 16 + (lr & 3) * 4 + (lc & 3);
#pragma unroll
                                for (int c = 0; c < CW; ++c) put(L, c, at(L, c) + pp[c]);
                            }
                        }
                    }
                    // the update: alpha c comes ready from the context; gamma is 1 inside, a function
                    // of the row or of the column alone in the sponge but for its corners
                    V ga = splat(sgz[lr]);
                    if (spx) {
                        const int zr = lr < nzt ? lr : lr - hr + nzb + nzt;
                        ga = lr < nzt || lr >= hr - nzb ? ldr(corner + zr * ncs + (lc < nxl ? lc : lc - cols + ncs))
                                                        : ldr(sgx + lc);
                    }
                    V nw = fma(in.ac, L, fma(ga, sub(u, ldr(pB)), u));
                    if (edge) {   // outside the grid: zero
#pragma unroll
                        for (int c = 0; c < CW; ++c)
                            if (gx0 + c >= a.nx) {
                                put(nw, c, T(0));
                                if constexpr ((F & F_STW) != 0) put(L, c, T(0));
                            }
                    }
                    str(pB, nw);
                    if ((rimx || (hasT && lr < 4) || (hasB && lr >= rows - 4)) && k + 1 < g.steps) {
                        // rim cells to the neighbours that read them
                        const unsigned tag = tag0 + (unsigned)(k + 1);
                        ulonglong2 *const inb = (k & 1) ? in1 : in0;
                        auto put_box = [&](ulonglong2 *box, int es) {
                            if constexpr (sizeof(T) == 4) {
                                send(box, tag, at(nw, 0), at(nw, 1));
                                send(box + es, tag, at(nw, 2), at(nw, 3));
                            } else {
                                send(box + (lc & 3) * es, tag, at(nw, 0));
                            }
                        };
                        const int qd = lc >> 2;
                        if (hasL && lc < 4) put_box(inb + boxes[2] + lr, rows);
                        if (hasR && lc >= cols - 4) put_box(inb + boxes[3] + lr, rows);
                        if (hasT && lr < 4) put_box(inb + boxes[0] + lr * EPR * nbx + qd, nbx);
                        if (hasB && lr >= rows - 4) put_box(inb + boxes[1] + (lr - rows + 4) * EPR * nbx + qd, nbx);
                    }
                    // what the step is about
                    if constexpr ((F & F_SAD) != 0) {
                        const T ez = T(Z0 + lr) * a.dx - T(a.src_pos[3 * s + 2]);
                        V gv = in.m;
#pragma unroll
                        for (int c = 0; c < CW; ++c) {
                            const T ex = T(gx0 + c) * a.dx - T(a.src_pos[3 * s + 0]);
                            const T Bd = a.unit_b ? T(1) : sqrt(ex * ex + ez * ez) + a.eps;
                            const T B2 = Bd * Bd;
                            put(gv, c, at(gv, c) + B2 * at(q, c) * at(L, c));
                        }
                        str(a.grad + (long long)s * a.sst + off, gv);
                    }
                    if constexpr ((F & F_AP) != 0) {   // A p = S^T S p + pen B^2 p
                        const V av = fma(in.m, in.y, nw);
                        T psum = T(0);
#pragma unroll
                        for (int c = 0; c < CW; ++c) psum += at(in.y, c) * at(av, c);
                        str(a.ap + fb + (long long)(a.nout + dk) * a.sst + off, av);
                        // four cells in the field precision, then double: the sum depends on the
                        // cut into tiles only within FP64 rounding
                        dot += double(psum);
                    }
                    if constexpr ((F & F_STW) != 0)
                        str(a.stash_w + ((long long)(a.slot_w + dk) * a.ns + s) * a.sst + off, L);
                    if constexpr ((F & F_GRD) != 0) str(a.grad + (long long)s * a.sst + off, fma(nw, in.y, in.m));
                    if constexpr ((F & F_OUT) != 0) {
                        T *f = a.fout + (long long)s * a.ofst + (long long)(a.nout + dk) * a.oplane;
                        if (a.opx == a.px) {
                            str(f + off, nw);
                        } else {
                            f += (Z0 + lr) * a.opx + gx0;
#pragma unroll
                            for (int c = 0; c < CW; ++c)
                                if (gx0 + c < a.nx) f[c] = at(nw, c);
                        }
                    }
                    if constexpr ((F & F_DFT) != 0)   // the DTFT's block stash
                        str(a.stash_w + ((long long)(a.slot_w + dk) * a.ns + s) * a.sst + off, nw);
                    // the next row's inputs (gradient cells after their store)
                    const bool wrap = j + 1 >= nrow;
                    if (!wrap || k + 1 < g.steps) fetch(wrap ? k + 1 : k, row_of(wrap ? 0 : j + 1), nrow > 1);
                }
                late = __syncthreads_or(0);   // uniform: every thread leaves together
                if (late) break;
            }
        } else {
            // ===================================================== communication threads
            const int ct = tid - g.nc, nxt = g.nm - SMP_T;   // exchange threads: nxt
            for (int k = 0; k < g.steps; ++k) {
                const T *A = (k & 1) ? buf1 : buf0;
                T *B = (k & 1) ? buf0 : buf1;
                const int dk = k * g.dn;
                const unsigned tag = tag0 + (unsigned)(k + 1);
                if (ct >= nxt) {
                    if constexpr ((F & F_SMP) != 0) {   // sample R u of the input state
                        const int to = a.tout + dk;
                        if (to >= 0 && to < g.nt) {
                            const int gt = s * tiles + tile;
                            const int e = g.smp_ptr[gt + 1];
                            for (int j = g.smp_ptr[gt] + ct - nxt; j < e; j += SMP_T) {
                                const LoopSmp<T> m = g.smp[j];
                                T v = T(0);
#pragma unroll
                                for (int c = 0; c < 4; ++c) v += m.w[c] * A[m.idx[c]];
                                a.smp_out[m.off + (long long)to * m.stride] = v;
                            }
                        }
                    }
                } else {
                    // L2 prefetch of the streams' tile rows PF_AHEAD steps on
                    if constexpr ((F & (F_EXT | F_CGP | F_AP | F_GRD)) != 0) {
                        if (k + PF_AHEAD < g.steps) {
                            const int d2 = dk + PF_AHEAD * g.dn;
                            for (int r = ct; r < rows; r += nxt) {
                                if (Z0 + r >= a.nz) break;
                                const long long gi = (long long)(Z0 + r) * a.px + X0;
                                const unsigned nb = (unsigned)(cols * sizeof(T));
                                if constexpr ((F & F_EXT) != 0) {
                                    const T *e = a.ext + fd + (long long)(a.n + d2) * a.N +
                                                 (long long)(Z0 + r) * a.nx + X0;
                                    const unsigned long long b0 = reinterpret_cast<unsigned long long>(e) & ~15ull;
                                    const unsigned long long b1 =
                                        (reinterpret_cast<unsigned long long>(e + min(cols, a.nx - X0)) + 15ull) & ~15ull;
                                    prefetch_l2(reinterpret_cast<const void *>(b0), (unsigned)(b1 - b0));
                                }
                                if constexpr ((F & F_CGP) != 0) {
                                    const long long vi = fb + (long long)(a.n + d2) * a.sst + gi;
                                    prefetch_l2(a.cg_r + vi, nb);
                                    if (!a.cg_first) prefetch_l2(a.cg_p + vi, nb);
                                }
                                if constexpr ((F & F_AP) != 0)
                                    prefetch_l2(a.ap_p + fb + (long long)(a.nout + d2) * a.sst + gi, nb);
                                if constexpr ((F & F_GRD) != 0)
                                    prefetch_l2(a.stash_r + ((long long)(a.slot_r + d2) * a.ns + s) * a.sst + gi, nb);
                            }
                        }
                    }
                    if (k + 1 < g.steps) {
                        // the next step's point sources, into the other patch set
                        if constexpr ((F & F_PT) != 0) {
                            inject(patch + ((k + 1) & 1) * 16 * np, a.tin + dk + g.dn, ct, nxt,
                                   [&] { asm volatile("barrier.sync 1, %0;" ::"r"(nxt) : "memory"); });
                        }
                        // the halo of the new state: entries [above][below][left][right]
                        const ulonglong2 *box = ((k & 1) ? in1 : in0) + (long long)me * g.istride;
                        const int eN = hasT ? nbx * 4 * EPR : 0;
                        const int eS = hasB ? nbx * min(4, a.nz - Z0 - rows) * EPR : 0;
                        const int eW = hasL ? hr * EPR : 0, eE = hasR ? hr * EPR : 0;
                        const int total = eN + eS + eW + eE;
                        constexpr int CPE = 4 / EPR;   // cells per entry
                        auto place = [&](int e, int &src) {   // inbox entry and the offset of its halo cells
                            if (e < eN + eS) {
                                const bool up = e < eN;
                                const int j = up ? e : e - eN;
                                src = up ? j : selfS + j;
                                const int sg = j / nbx, b = j - sg * nbx;   // sg = row * EPR + part
                                return (up ? sg / EPR : rows + 4 + sg / EPR) * P + 4 + 4 * b + (sg % EPR) * CPE;
                            }
                            const bool lf = e < eN + eS + eW;
                            const int j = e - eN - eS - (lf ? 0 : eW);
                            const int part = j / hr, row = j - part * hr;
                            src = 2 * selfS + (lf ? 0 : rows * EPR) + part * rows + row;
                            return (row + 4) * P + (lf ? 0 : 4 + cols) + part * CPE;
                        };
                        constexpr int U = 6;   // entries in flight per thread
                        for (int e0 = ct; e0 < total && !late; e0 += U * nxt) {
                            int dst[U];
                            int src[U];
                            unsigned open = 0;
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const int e = e0 + u * nxt;
                                dst[u] = 0;
                                src[u] = 0;
                                if (e < total) {
                                    dst[u] = place(e, src[u]);
                                    open |= 1u << u;
                                }
                            }
                            for (int polls = 0; open; ++polls) {
                                ulonglong2 v[U];
#pragma unroll
                                for (int u = 0; u < U; ++u)
                                    if (open & (1u << u)) v[u] = ld_packets(box + src[u]);
#pragma unroll
                                for (int u = 0; u < U; ++u)
                                    if ((open & (1u << u)) && tagged(v[u], tag)) {
                                        unpack(v[u], B + dst[u]);
                                        open &= ~(1u << u);
                                    }
                                if (polls >= g.polls) {
                                    atomicExch(a.dev_err, DEV_ERR_LOOP_TIMEOUT);
                                    late = true;
                                    break;
                                }
                            }
                        }
                    }
                }
                late = __syncthreads_or(late);
                if (late) break;
            }
        }
        // ---- epilogue: both states back to the caller's arrays
        if (!late) {
            for (int i = tid; i < nbx * rows; i += nthr) {
                const int r = i / nbx, q = i - r * nbx;
                if (Z0 + r >= a.nz) break;
                const long long gi = (long long)(Z0 + r) * a.px + X0 + 4 * q;
                const T *d0 = buf0 + (r + 4) * P + 4 * (q + 1), *d1 = buf1 + (r + 4) * P + 4 * (q + 1);
#pragma unroll
                for (int h = 0; h < 4; h += 16 / (int)sizeof(T)) {
                    *reinterpret_cast<uint4 *>(st0 + gi + h) = *reinterpret_cast<const uint4 *>(d0 + h);
                    *reinterpret_cast<uint4 *>(st1 + gi + h) = *reinterpret_cast<const uint4 *>(d1 + h);
                }
            }
        }
        if constexpr ((F & F_AP) != 0) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
            if ((tid & 31) == 0) red[tid >> 5] = dot;
            __syncthreads();
            if (tid == 0) {
                double t = 0.0;
                for (int w = 0; w < nthr / 32; ++w) t += red[w];
                a.dot_part[(long long)s * g.dot_stride + tile] += t;
            }
        }
    }
    // the last CTA to finish moves the epoch past every tag of this launch
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(g.sync + 1, 1u) == gridDim.x - 1) {
            g.sync[1] = 0;
            g.sync[0] = tag0 + (unsigned)g.steps + 1u;
        }
    }
}

template <typename T, unsigned F>
cudaError_t go(const StepArgs<T> &a, const LoopArgs<T> &g, int nblk, int threads, size_t smem,
               cudaStream_t st) {
    static PerDevice attr;
    int set = 0;
    cudaError_t e = per_device(attr, &set, [](int *v) {
        *v = 1;
        return cudaFuncSetAttribute(fd2_loop_kernel<T, F>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, LOOP_SMEM);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nblk);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fd2_loop_kernel<T, F>, a, g);
}

template <typename T>
cudaError_t dispatch(unsigned flags, const StepArgs<T> &a, const LoopArgs<T> &g, int nblk,
                     int threads, size_t smem, cudaStream_t st) {
#define ESI_CASE(FL) \
    case (FL):       \
        return go<T, (FL)>(a, g, nblk, threads, smem, st);
    switch (flags) {   // the variants of launch_step2
        ESI_CASE(F_PT | F_SMP)
        ESI_CASE(F_EXT | F_SMP)
        ESI_CASE(F_EXT | F_PT | F_SMP)
        ESI_CASE(F_PT | F_SMP | F_DFT)
        ESI_CASE(F_EXT | F_SMP | F_DFT)
        ESI_CASE(F_EXT | F_PT | F_SMP | F_DFT)
        ESI_CASE(F_CGP | F_SMP)
        ESI_CASE(F_PT | F_STW)
        ESI_CASE(F_EXT | F_STW)
        ESI_CASE(F_EXT | F_PT | F_STW)
        ESI_CASE(F_EXT | F_SAD)
        ESI_CASE(F_EXT | F_PT | F_SAD)
        ESI_CASE(F_EXT | F_SMP | F_SAD)
        ESI_CASE(F_EXT | F_PT | F_SMP | F_SAD)
        ESI_CASE(F_PT)
        ESI_CASE(F_PT | F_OUT)
        ESI_CASE(F_PT | F_OUT | F_SMP)
        ESI_CASE(F_PT | F_AP)
        ESI_CASE(F_PT | F_GRD)
        default:
            return cudaErrorInvalidValue;
    }
#undef ESI_CASE
}

}  // namespace loop2
}  // namespace esi
