// On-chip step kernel: the whole time loop of a grid that fits in the SMs'
// shared memory (FP32 and Q5.27 car grids, theta periodic).
//
// One cooperative launch runs all the steps.  Each CTA owns a block of bx x by
// grid columns (a column: the v x theta values of one (x, y), contiguous in
// memory) and keeps their values on chip for the whole launch, so that a step
// moves only the blocks' edge columns through L2 instead of reading every
// value and all its neighbours from there.
//
// Work split: a thread owns one theta quad (4 consecutive headings) of one v
// row, in all by columns of one x, and walks them along y: the columns y - 1,
// y, y + 1 of its quad pass through registers, the x neighbour of the upwind
// side and the two v neighbours are one 16-byte shared-memory load each, the
// theta neighbours outside the quad a warp shuffle (shared memory where the
// row or the warp ends).  V is held twice (before and after the step).  The
// sweep is bound by shared-memory bandwidth and issue (about 31 shared-memory
// wavefronts and 190 instructions per warp and column).  Measured, us per step
// with the L2-resident form and with this one: 31x31x11x16 FP32 3.2 -> 2.4,
// 60x60x20x36 FP32 10.9 -> 5.3, Q5.27 with steering 16.5 -> 8.5, 47x53x17x27
// with steering 6.5 -> 4.0.  What was tried and is slower: V and V0 in registers
// with the columns unrolled (spills, and 240 instructions per column: 9.5 us on
// 60x60x20x36), the paired FP32 instructions (fewer instructions, but each
// takes two turns of the FMA pipe: 39 against 33 clocks per warp and column).
//
// Step: (1) wait until the (up to four) neighbour CTAs have published the
// previous step's edge columns, (2) copy the ones this thread needs (those on
// the upwind side of its quad only) into its own shared-memory slots with
// cp.async through L2, (3) update the quads; edge columns that a neighbour will
// read (and on the last step every column) also go to the global value buffer,
// (4) publish (barrier, one flag per CTA stored with release semantics).  V
// alternates between the two global buffers, and a CTA writes step
// s + 1 only after its neighbours have published step s, that is, after they
// have read what it overwrites.  Only neighbours wait for one another: there
// is no grid-wide barrier.  Every wait is bounded (limit_ns); on timeout the
// CTA records HJ_ERR_TIMEOUT and leaves, and its neighbours, which wait for its
// step since at most a step's time, run out with it.
//
// The per-cell arithmetic is the resident and generic kernels' (cell_value,
// hj_q527_update), in the same order: the results are the same bit for bit.
#pragma once

#include "hj_resident.cuh"

namespace hj_onchip {

struct Params {
    int bx, by;  // columns of a block along x and y
    int gy;      // blocks along y
    int steps, cut, pub_all;
    long long n0;  // steps taken before this launch
    float k3;
};

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ int32_t fi(float x) { return __float_as_int(x); }
__device__ __forceinline__ float fl(int32_t x) { return __int_as_float(x); }

// p where the mask is all ones, m where it is 0 (one logic instruction, no predicate).
__device__ __forceinline__ float bitsel(uint32_t mask, float p, float m)
{
    return fl((int32_t)(((uint32_t)fi(p) & mask) | ((uint32_t)fi(m) & ~mask)));
}
__device__ __forceinline__ float4 pick4(const uint32_t mask[4], const float4 &p, const float4 &m)
{
    return make_float4(bitsel(mask[0], p.x, m.x), bitsel(mask[1], p.y, m.y), bitsel(mask[2], p.z, m.z),
                       bitsel(mask[3], p.w, m.w));
}

// 16 bytes of shared memory if p; otherwise the result is unspecified (the
// caller masks it away), which costs no register moves to define.
__device__ __forceinline__ float4 lds_if(bool p, const float *a)
{
    float4 v;
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %5, 0;\n\t@q ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "r"(smem_u32(a)), "r"((uint32_t)p));
    return v;
}

// Upwind side of one axis for a thread's quad: every lane that carries
// weight has the flow from index + 1 (PLUS), from index - 1 (MINUS), or the
// lanes differ (MIXED, then the sides are in a bit mask).
enum : int { PLUS = 0, MINUS = 1, MIXED = 2 };

__device__ __forceinline__ int side_class(uint32_t plus, uint32_t weighted)
{
    if ((plus & weighted) == weighted) return PLUS;
    return (plus & weighted) == 0u ? MINUS : MIXED;
}

// Waits until *p >= s (bounded; the timer is looked at now and then only,
// reading it costs more than a poll).
__device__ __forceinline__ bool wait_published(const unsigned int *p, unsigned int s, unsigned long long limit_ns)
{
    unsigned int v;
    unsigned long long deadline = 0ull;
    for (unsigned int i = 1;; ++i) {
        v = hj_ld_acquire_u32(p);
        if (v >= s) break;
        if ((i & 255u) == 0u) {
            const unsigned long long t = global_ns();
            if (deadline == 0ull) deadline = t + limit_ns;
            else if (t > deadline) return false;
        }
    }
    return true;
}

// What a thread knows about its quad for the whole launch.
struct Thread {
    float K1[4], K2[4], k3, k4;  // FP32: |xdot_d| / dx_d; Q5.27: weight magnitudes (int32 bits)
    int32_t nsum[4];             // Q5.27: -(sum of the four weights)
    bool wsmall;                 // Q5.27: none below -2^30 in the warp (hj_q527_update_interior32)
    bool edge_warp;              // Q5.27: some quad of the warp has an x or v ghost
    uint32_t mx[4], my[4];
    uint32_t sx;
    int ovm, ovp, lidx, ridx, lreal, cs;
    bool xmix, ymin, gvm, gvp, vedge_warp, left_sm, right_sm, act, gxm, gxp, gy0, gy1, gu;
};

// Where a step's sweep reads and writes.
struct SweepIO {
    const float *row, *pu, *xm, *xp, *ym_h, *yp_h, *z, *zc;
    float *nxt, *vot;
    int bya;
    bool pub, pub0, publ;  // store to global memory: every column; the first; the last
};

// One step of a thread's quads, along y.
template <bool FIXED, bool MIX, bool PADDED, bool ZFLAT>
__device__ __forceinline__ void sweep(const Thread &T, SweepIO io, const float dt)
{
    const int cs = T.cs, lreal = T.lreal;
    float4 ym = *(const float4 *)io.ym_h, c = *(const float4 *)io.row;  // columns y - 1, y before the update
    for (int j = 0; j < io.bya; ++j) {
        // (threads past the block compute on whatever is there and store
        // nothing: the flow is uniform)
        const bool jlast = j == io.bya - 1;
        const float4 yp = *(const float4 *)(jlast ? io.yp_h : io.row + cs);
        // theta neighbours outside the quad
        float tl = __shfl_up_sync(0xffffffffu, c.w, 1), tr = __shfl_down_sync(0xffffffffu, c.x, 1);
        if (T.left_sm) tl = io.row[T.lidx];
        if (T.right_sm) tr = io.row[T.ridx];
        float4 z;
        if (ZFLAT) {
            const float z0 = io.zc[j];
            z = make_float4(z0, z0, z0, z0);
        } else {
            z = __ldg((const float4 *)io.z);
            io.z += cs;
        }
        float4 vm = *(const float4 *)(io.row + T.ovm), vp = *(const float4 *)(io.row + T.ovp);
        float4 ux = *(const float4 *)io.pu;
        float4 out;
        if constexpr (!FIXED) {
            if (T.vedge_warp) {
                if (T.gvm) vm = f4ghost(c, vm);
                if (T.gvp) vp = f4ghost(c, vp);
            }
            float4 uy;
            if (MIX) {
                ux = pick4(T.mx, ux, lds_if(T.xmix, io.xm));
                uy = pick4(T.my, yp, ym);
                io.xm += cs;
            } else {
                uy = T.ymin ? ym : yp;
            }
            // the right neighbours of the lanes (a padded last quad wraps at lane lreal - 1)
            float t0 = c.y, t1 = c.z, t2 = c.w;
            if (PADDED) {
                if (lreal == 1) t0 = tr;
                if (lreal == 2) t1 = tr;
                if (lreal == 3) t2 = tr;
            }
            const float cc[4] = {c.x, c.y, c.z, c.w}, xx[4] = {ux.x, ux.y, ux.z, ux.w},
                        yy[4] = {uy.x, uy.y, uy.z, uy.w},
                        vv[4] = {fmaxf(vp.x, vm.x), fmaxf(vp.y, vm.y), fmaxf(vp.z, vm.z), fmaxf(vp.w, vm.w)},
                        tt[4] = {fmaxf(t0, tl), fmaxf(t1, c.x), fmaxf(t2, c.y), fmaxf(tr, c.z)},
                        zz[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {  // cell_value
                float r = T.K1[e] * (xx[e] - cc[e]);
                r = fmaf(T.K2[e], yy[e] - cc[e], r);
                r = fmaf(T.k3, vv[e] - cc[e], r);
                r = fmaf(T.k4, tt[e] - cc[e], r);
                f4set(out, e, fminf(zz[e], fmaf(dt, r, cc[e])));
            }
        } else {
            // per lane: the grid value to weigh on each axis and whether it stands for an
            // extrapolated ghost 2 V_c - u (then it is weighed by -W, and V_c by +2W)
            const bool gym = j == 0 && T.gy0, gyp = jlast && T.gy1;
            float4 xa = ux, xb = ux, ya = ym, yb = yp;  // index - 1, index + 1
            if (MIX) {
                if (T.xmix) {
                    xa = *(const float4 *)io.xm;
                    xb = *(const float4 *)io.xp;
                }
                io.xm += cs;
                io.xp += cs;
            }
            if (gym) ya = yp;  // the value the ghost is formed from
            if (gyp) yb = ym;
            const int32_t w3 = fi(T.k3), w4 = fi(T.k4);
            int32_t tt[4];  // the larger theta neighbour
            tt[0] = max(fi(PADDED && lreal == 1 ? tr : c.y), fi(tl));
            tt[1] = max(fi(PADDED && lreal == 2 ? tr : c.z), fi(c.x));
            tt[2] = max(fi(PADDED && lreal == 3 ? tr : c.w), fi(c.y));
            tt[3] = max(fi(tr), fi(c.z));
            // every neighbour of the warp's quads is a grid value (a quad without ghosts gives
            // the same codes in both forms, and a warp that splits takes the time of the two)
            if (T.wsmall && !T.edge_warp && !gym && !gyp) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int32_t u1 = fi(MIX ? bitsel(T.mx[e], f4get(xb, e), f4get(xa, e)) : f4get(ux, e));
                    const int32_t u2 = fi(bitsel(T.my[e], f4get(yb, e), f4get(ya, e)));
                    const int32_t u3 = max(fi(f4get(vp, e)), fi(f4get(vm, e)));
                    f4set(out, e,
                          fl(hj_q527_update_interior32(fi(f4get(c, e)), fi(f4get(z, e)), u1, u2, u3, tt[e],
                                                       fi(T.K1[e]), fi(T.K2[e]), w3, w4, T.nsum[e])));
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const bool xpos = (T.sx >> e) & 1u;
                    const int32_t vc = fi(f4get(c, e)), a1 = fi(T.K1[e]), a2 = fi(T.K2[e]);
                    const int32_t u1 = fi(MIX ? bitsel(T.mx[e], f4get(xb, e), f4get(xa, e)) : f4get(ux, e));
                    const int32_t u2 = fi(bitsel(T.my[e], f4get(yb, e), f4get(ya, e)));
                    const int32_t pv = fi(f4get(vp, e)), mv = fi(f4get(vm, e)), u3 = max(pv, mv);
                    const bool hxg = T.xmix ? (xpos ? T.gxp : T.gxm) : T.gu;
                    const bool hyg = T.my[e] ? gyp : gym;
                    // v: at an end both pv and mv hold the one grid neighbour o; the larger of o and
                    // its ghost 2 V_c - o (upper end: the ghost if equal, it is V(v + 1))
                    const bool hv = T.gvp ? vc >= mv : (T.gvm ? pv < vc : false);
                    const int32_t c0 = T.nsum[e] + (hxg ? 2 * a1 : 0) + (hyg ? 2 * a2 : 0) + (hv ? 2 * w3 : 0);
                    f4set(out, e,
                          fl(hj_q527_update_interior(vc, fi(f4get(z, e)), u1, u2, u3, tt[e], hxg ? -a1 : a1,
                                                     hyg ? -a2 : a2, hv ? -w3 : w3, w4, c0)));
                }
            }
        }
        if (PADDED) {  // pad lanes hold 0
            if (lreal <= 1) out.y = 0.f;
            if (lreal <= 2) out.z = 0.f;
            if (lreal <= 3) out.w = 0.f;
        }
        if (T.act) *(float4 *)io.nxt = out;
        if (io.pub || (io.pub0 && j == 0) || (io.publ && jlast)) *(float4 *)io.vot = out;
        ym = c;
        c = yp;
        io.row += cs;
        io.pu += cs;
        io.nxt += cs;
        io.vot += cs;
    }
}

template <bool FIXED, bool MIX, bool PADDED, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
    onchip_kernel(const float *__restrict__ v0, float *buf, const void *__restrict__ coefp,
                  const int32_t *__restrict__ qw, const void *__restrict__ k4tab, const HjLoop *__restrict__ lp,
                  HjFlags *flags, const HjGeom g, const Params P, long long nint, unsigned int *prog,
                  unsigned long long limit_ns)
{
    extern __shared__ __align__(16) float sm[];
    __shared__ int s_ok;
    const int N1 = g.n1, N2 = g.n2, N3 = g.n3, N4 = g.n4, P4 = g.p4, q4 = P4 / 4;
    const int cs = N3 * P4;  // values of a column: the stride along y, in shared and in global memory
    const int tid = threadIdx.x, lane = tid & 31;
    const int q = tid % q4, rr = tid / q4;
    const int cx = (int)blockIdx.x / P.gy, cy = (int)blockIdx.x - cx * P.gy;
    const int x0 = cx * P.bx, y0 = cy * P.by;
    const int bxa = min(P.bx, N1 - x0), bya = min(P.by, N2 - y0);  // this block's columns
    const bool act = rr / N3 < bxa;
    int k = rr % N3, lx = act ? rr / N3 : 0;  // (threads past the block read the first column's, and store nothing)
    if (FIXED && act && N3 > 2) {
        // In fixed point a warp with an end of v takes the longer form: the ends of
        // all the block's columns come first, so that fewer warps have one (us per
        // step, car: 47x53x17x27 6.1 -> 5.6, 80x80x13x16 6.2 -> 5.2, 60x60x20x36
        // 8.7 -> 8.5, 13x13x64x30 the same).
        const int rm = rr - 2 * bxa;
        lx = rm < 0 ? rr / 2 : rm / (N3 - 2);
        k = rm < 0 ? (rr & 1) * (N3 - 1) : 1 + rm % (N3 - 2);
    }
    const int x = x0 + lx;
    const int e0 = k * P4 + 4 * q;
    const int lreal = min(4, N4 - 4 * q);  // lanes of the quad inside the row

    // shared memory: the block's columns twice (V before and after the step),
    // the x halo slots [2][by] and the y halo slots [2][bx] (columns whose
    // quads are private to the thread that reads them), one V0 per column
    const int ncol = P.bx * P.by;
    float *xm_h = sm + 2 * ncol * cs + e0, *xp_h = xm_h + P.by * cs;
    float *ym_h = xm_h + (2 * P.by + lx) * cs, *yp_h = ym_h + P.bx * cs;
    float *zc = sm + (2 * ncol + 2 * P.by + 2 * P.bx) * cs + lx * P.by;
    const int own = lx * P.by * cs + e0;
    const bool gxm = x == 0, gxp = x == N1 - 1, gy0 = y0 == 0, gy1 = y0 + bya == N2;
    const uint32_t goff = (uint32_t)((x * N2 + y0) * N3) * P4 + e0;

    // the quad's coefficients; which side the flow comes from
    Thread T;
    uint32_t sx = 0u, sy = 0u;  // bit e: the flow of lane e comes from index + 1
    int clx = PLUS, cly = PLUS;
    auto load_coefs = [&](int sel) {
        const int32_t *w = FIXED ? qw + (size_t)sel * hj_qw_count(N3, P4) : nullptr;
        T.k3 = FIXED ? fl(w[2 * cs]) : P.k3;
        T.k4 = FIXED ? fl(w[2 * cs + HJ_QW_TAIL + k]) : ((const float2 *)k4tab)[k].x;
        T.wsmall = true;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            T.nsum[e] = 0;
            T.K1[e] = T.K2[e] = 0.f;
            if (e >= lreal) continue;
            if constexpr (FIXED) {
                T.K1[e] = fl(abs(w[e0 + e]));
                T.K2[e] = fl(abs(w[cs + e0 + e]));
                T.nsum[e] = -(fi(T.K1[e]) + fi(T.K2[e]) + fi(T.k3) + fi(T.k4));
                T.wsmall = T.wsmall && T.nsum[e] >= -(1 << 30);
            } else {
                const HjCoef<float> c = ((const HjCoef<float> *)coefp)[k * N4 + 4 * q + e];
                T.K1[e] = fabsf(c.c1);
                T.K2[e] = fabsf(c.c2);
            }
        }
        if (FIXED) T.wsmall = __all_sync(0xffffffffu, T.wsmall || !act);
    };
    // the sides come from the velocities; lanes whose weight is 0 (at each step
    // size this launch takes: the cut step's table is built only for a call
    // that has one) may sit on any side
    {
        uint32_t wx = 0u, wy = 0u;
        for (int e = 0; e < lreal; ++e) {
            const uint32_t bit = 1u << e;
            if constexpr (FIXED) {
                const HjCoef<double> c = ((const HjCoef<double> *)coefp)[k * N4 + 4 * q + e];
                const int32_t *w1 = P.cut ? qw + hj_qw_count(N3, P4) : qw;
                if (c.c1 >= 0.0) sx |= bit;
                if (c.c2 >= 0.0) sy |= bit;
                if (qw[e0 + e] | w1[e0 + e]) wx |= bit;
                if (qw[cs + e0 + e] | w1[cs + e0 + e]) wy |= bit;
            } else {
                const HjCoef<float> c = ((const HjCoef<float> *)coefp)[k * N4 + 4 * q + e];
                if (c.c1 >= 0.f) sx |= bit;
                if (c.c2 >= 0.f) sy |= bit;
                if (c.c1 != 0.f) wx |= bit;
                if (c.c2 != 0.f) wy |= bit;
            }
        }
        clx = side_class(sx, wx);
        cly = side_class(sy, wy);
    }
    load_coefs(P.cut && P.steps == 1 ? 1 : 0);

    // The x neighbours: in the block (an offset from the thread's own column)
    // or in the halo slots.  FP32: past an end of the grid the slot holds the
    // extrapolated ghost; Q5.27: the ghost may not fit in 32 bits, so the grid
    // value it is formed from is loaded instead (gu).
    const bool xm_in = lx > 0, xp_in = lx < bxa - 1;
    const bool gu = FIXED && (clx == PLUS ? gxp : gxm);
    const bool pu_plus = (clx != MINUS) != gu;
    // v neighbours; at an end of the grid the row the ghost is formed from
    const bool gvm = k == 0, gvp = k == N3 - 1;
    const int ovm = gvm ? P4 : -P4, ovp = gvp ? -P4 : P4;
    // per-lane masks of the lanes whose flow comes from index + 1
    T.xmix = MIX && clx == MIXED;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        T.mx[e] = T.xmix && !((sx >> e) & 1u) ? 0u : ~0u;
        T.my[e] = cly == PLUS || (cly == MIXED && ((sy >> e) & 1u)) ? ~0u : 0u;
    }
    T.ymin = cly == MINUS;
    T.gvm = gvm;
    T.gvp = gvp;
    T.vedge_warp = __any_sync(0xffffffffu, gvm || gvp);
    T.ovm = ovm;
    T.ovp = ovp;
    T.lreal = lreal;
    T.act = act;
    T.cs = cs;
    T.sx = sx;
    T.gxm = gxm;
    T.gxp = gxp;
    T.gy0 = gy0;
    T.gy1 = gy1;
    T.gu = gu;
    T.edge_warp = FIXED && __any_sync(0xffffffffu, act && (gvm || gvp || (T.xmix ? gxm || gxp : gu)));
    // halo columns this thread reads
    const bool need_xm = act && !xm_in && !gxm && (clx != PLUS || gxp);
    const bool need_xp = act && !xp_in && !gxp && (clx != MINUS || gxm);
    const bool need_ym = act && !gy0 && (cly != PLUS || (bya == 1 && gy1));
    const bool need_yp = act && !gy1 && (cly != MINUS || (bya == 1 && gy0));
    const bool need_any = need_xm || need_xp || need_ym || need_yp;
    // the neighbour CTA whose flag thread t < 4 polls
    int nb = -1;
    if (tid == 0 && x0 > 0) nb = (int)blockIdx.x - P.gy;
    if (tid == 1 && x0 + bxa < N1) nb = (int)blockIdx.x + P.gy;
    if (tid == 2 && y0 > 0) nb = (int)blockIdx.x - 1;
    if (tid == 3 && y0 + bya < N2) nb = (int)blockIdx.x + 1;
    // theta neighbours: from the adjacent lane, or from the row in shared memory
    T.left_sm = q == 0 || lane == 0;
    T.right_sm = q == q4 - 1 || lane == 31;
    T.lidx = (q == 0 ? N4 - 1 : 4 * q - 1) - 4 * q;
    T.ridx = (q == q4 - 1 ? 0 : 4 * q + 4) - 4 * q;
    // values a neighbour CTA reads (its upwind side): stored to global memory
    // every step.  A block one column wide at an end of the grid forms its ghost
    // from the other side's column, whatever the quad's own side is (P.pub_all).
    const bool pub_x = act && ((!xm_in && !gxm && (clx != MINUS || P.pub_all)) ||
                               (!xp_in && !gxp && (clx != PLUS || P.pub_all)));
    const bool pub_y0 = pub_x || (act && !gy0 && (cly != MINUS || P.pub_all));
    const bool pub_y1 = pub_x || (act && !gy1 && (cly != PLUS || P.pub_all));
    const float dts[2] = {(float)lp->dt[0], (float)lp->dt[1]};

    // V after n0 steps into shared memory; whether V0 has one value per column
    // in this block (it depends on the position only, Eq. init_V)
    bool zflat = true;
    {
        const float *vin = P.n0 == 0 ? v0 : buf + ((P.n0 - 1) & 1) * nint;
        for (int j = 0; act && j < bya; ++j) {
            *(float4 *)(sm + own + j * cs) = *(const float4 *)(vin + goff + j * cs);
            const float4 z = *(const float4 *)(v0 + goff + j * cs);
            const float z0 = v0[goff + j * cs - e0];
            zflat = zflat && fi(z.x) == fi(z0) && (lreal < 2 || fi(z.y) == fi(z0)) &&
                    (lreal < 3 || fi(z.z) == fi(z0)) && (lreal < 4 || fi(z.w) == fi(z0));
            if (e0 == 0) zc[j] = z0;
        }
        if (tid == 0) s_ok = 1;
        zflat = __syncthreads_and(zflat);
    }

    for (int s = 0; s < P.steps; ++s) {
        const bool final_step = s == P.steps - 1;
        const int sel = P.cut && final_step ? 1 : 0;
        if (FIXED && sel == 1 && s > 0) load_coefs(1);  // the cut step's weights
        const float dt = dts[sel];
        const long long n = P.n0 + s;
        const float *vi = n == 0 ? v0 : buf + ((n - 1) & 1) * nint;
        float *vot = buf + (n & 1) * nint + goff;
        const float *cur = sm + (s & 1) * ncol * cs + own;
        float *nxt = sm + ((s & 1) ^ 1) * ncol * cs + own;
        if (s > 0) {
            if (nb >= 0 && !wait_published(prog + nb * HJ_SYNC_STRIDE, (unsigned int)s, limit_ns)) {
                s_ok = 0;
                *(volatile int *)&flags->status = HJ_ERR_TIMEOUT;
            }
            __syncthreads();  // the neighbours have published step s - 1's values
            if (!s_ok) return;
        }
        const float *xm_p = xm_in ? cur - P.by * cs : xm_h, *xp_p = xp_in ? cur + P.by * cs : xp_h;
        // halo quads of this thread, into its own slots
        if (need_any) {
            const float *src = vi + goff;
            if (need_ym) cp_async16(smem_u32(ym_h), src - cs);
            if (need_yp) cp_async16(smem_u32(yp_h), src + bya * cs);
            if (need_xm || need_xp) {
                uint32_t d = smem_u32(need_xm ? xm_h : xp_h);
                const float *hsrc = src + (need_xm ? -(long long)N2 * cs : (long long)N2 * cs);
                for (int j = 0; j < bya; ++j, d += 4 * cs, hsrc += cs) cp_async16(d, hsrc);
            }
            if (need_xm && need_xp)
                for (int j = 0; j < bya; ++j)
                    cp_async16(smem_u32(xp_h + j * cs), src + j * cs + (long long)N2 * cs);
            asm volatile("cp.async.wait_all;" ::: "memory");
        }
        if constexpr (!FIXED) {  // the ghosts past the ends of x and y, into the halo slots
            if (act && (gxm || gxp || gy0 || gy1)) {
                if (gxm)
                    for (int j = 0; j < bya; ++j)
                        *(float4 *)(xm_h + j * cs) =
                            f4ghost(*(const float4 *)(cur + j * cs), *(const float4 *)(xp_p + j * cs));
                if (gxp)
                    for (int j = 0; j < bya; ++j)
                        *(float4 *)(xp_h + j * cs) =
                            f4ghost(*(const float4 *)(cur + j * cs), *(const float4 *)(xm_p + j * cs));
                if (gy0) *(float4 *)ym_h = f4ghost(*(const float4 *)cur, *(const float4 *)(bya > 1 ? cur + cs : yp_h));
                if (gy1)
                    *(float4 *)yp_h = f4ghost(*(const float4 *)(cur + (bya - 1) * cs),
                                             *(const float4 *)(bya > 1 ? cur + (bya - 2) * cs : ym_h));
            }
        }

        asm volatile("" ::: "memory");  // the slots' stores stay before the sweep's loads of them
        SweepIO io;
        io.row = cur;
        io.pu = pu_plus ? xp_p : xm_p;
        io.xm = gxm ? xp_p : xm_p;  // (Q5.27; for FP32 the slots hold the ghosts)
        io.xp = gxp ? xm_p : xp_p;
        if (!FIXED) {
            io.xm = xm_p;
            io.xp = xp_p;
        }
        io.nxt = nxt;
        io.vot = vot;
        io.z = v0 + goff;
        io.zc = zc;
        io.ym_h = ym_h;
        io.yp_h = yp_h;
        io.bya = bya;
        io.pub = (final_step && act) || pub_x;
        io.pub0 = pub_y0;
        io.publ = pub_y1;
        if (zflat) sweep<FIXED, MIX, PADDED, true>(T, io, dt);
        else sweep<FIXED, MIX, PADDED, false>(T, io, dt);
        if (final_step) return;
        __syncthreads();  // every read of step s is done, every edge value is written
        if (tid == 0)
            asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(prog + blockIdx.x * HJ_SYNC_STRIDE), "r"((unsigned int)(s + 1))
                         : "memory");
    }
}

}  // namespace hj_onchip
