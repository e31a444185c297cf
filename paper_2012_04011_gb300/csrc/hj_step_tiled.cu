// Host side of the tiled step kernel (hj_tiled_kernel.cuh): tile shape,
// tensor maps, shared-memory layout, kernel selection and launch.
#include "hj_tiled_kernel.cuh"

using namespace hj_tiled;

namespace {

KernelFn kernel_fn(bool fixed, bool padded, bool usign, bool bcast, bool track, int nconsumer, int rpt)
{
    // the fixed-point variant selects the upwind side per lane (no USIGN form)
    if (fixed) return select_q527(padded, bcast, track, nconsumer);
    return track ? select_f32_track(padded, usign, bcast, nconsumer, rpt)
                 : select_f32(padded, usign, bcast, nconsumer, rpt);
}

// v rows per consumer thread in the broadcast-V0 single-sided FP32 form
// (bound by data movement: several rows a thread let a CTA hold larger tiles,
// whose halo rows cost less L2 traffic per row, and share the per-plane
// ring and address work): four when tv is a multiple of 4 and that still
// leaves at least 8 consumer warps, else two when tv is even; one otherwise
// and in every other variant.  g->tiled_usign must be current
// (hj_tiled_setup sets it before it sizes a tile).
int tiled_rpt(const hj_grid *g, int ty, int tv)
{
    if (!(g->prec == HJ_FP32 && g->v0_bcast && g->tiled_usign && g->p4 == g->n[3])) return 1;
    if (tv % 4 == 0 && (g->p4 / 4) * ty * (tv / 4) >= 256) return 4;
    return tv % 2 == 0 ? 2 : 1;
}

int consumers_of(const hj_grid *g, int ty, int tv)
{
    return ((g->p4 / 4) * ty * (tv / tiled_rpt(g, ty, tv)) + 31) / 32 * 32;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
    }
    return fn;
}

TiledParams make_params(const hj_grid *g, int ty, int tv, int stages, int xc)
{
    TiledParams P;
    memset(&P, 0, sizeof(P));
    P.ty = ty;
    P.tv = tv;
    P.stages = stages;
    P.q4 = g->p4 / 4;
    P.rpt = tiled_rpt(g, ty, tv);
    P.nconsumer = consumers_of(g, ty, tv);
    P.ncol_v = (g->n[2] + tv - 1) / tv;
    P.ncol = ((g->n[1] + ty - 1) / ty) * P.ncol_v;
    P.halo_box = g->p4 * (tv + 2) * (ty + 2);
    P.halo_floats = (P.halo_box + 31) / 32 * 32;
    P.v0_floats = g->v0_bcast ? 0 : g->p4 * tv * ty;
    P.stage_bytes = ((P.halo_floats + P.v0_floats) * 4 + 127) / 128 * 128;
    P.xc = xc < 1 ? g->n[0] : (xc > g->n[0] ? g->n[0] : xc);
    P.nchunk = (g->n[0] + P.xc - 1) / P.xc;
    P.nitems = P.ncol * P.nchunk;
    P.k3 = (float)g->geom.k3;
    P.k4 = (float)g->geom.k4;
    P.mk34 = (float)(-(g->geom.k3 + g->geom.k4));
    return P;
}

// Planes per work item: all CTAs sweep x concurrently, so the time of a step
// is about (rounds of items) x (planes one item loads, halo planes included).
// Pick the chunk length that minimises it.
int best_chunk(const hj_grid *g, int ncol, int slots)
{
    const int n1 = g->n[0];
    int best_xc = n1;
    double best = 1e300;
    for (int nchunk = 1; nchunk <= n1 / 4 || nchunk == 1; ++nchunk) {
        const int xc = (n1 + nchunk - 1) / nchunk;
        const int nch = (n1 + xc - 1) / xc;
        const long long items = (long long)ncol * nch;
        const long long rounds = (items + slots - 1) / slots;
        const double cost = (double)rounds * (xc + (nch > 1 ? 2 : 0));
        if (cost < best - 1e-9) {
            best = cost;
            best_xc = xc;
        }
    }
    return best_xc;
}

// Fixed point: the most planes any of the n CTAs sweeps in a step, in planes of
// an inner tile.  A plane of a tile at an end of v takes 1.7 + 0.5 / tv times as
// long (extrapolated ghosts take the 64-bit form), at an end of y 1.1 times; the
// CTAs take the items in next_item()'s order.  Beyond 16 rounds the CTAs' shares
// are close to the mean, which is used instead.  Above `limit` the value is a
// lower bound: the mean, or what a CTA has by then.
double heaviest_q527(const hj_grid *g, const TiledParams &P, int xc, int nchunk, int n, double limit)
{
    const long long items = (long long)P.ncol * nchunk;
    const bool mean = items > 16LL * n || n > 1024;
    if (n > items) n = (int)items;
    const int ncol_y = P.ncol / P.ncol_v;
    const double end_v = 1.7 + 0.5 / P.tv;
    auto planes_of = [&](int c) {
        const int x0 = c * xc, x1 = x0 + xc < g->n[0] ? x0 + xc : g->n[0];
        return (x1 < g->n[0] ? x1 + 1 : x1) - (x0 > 0 ? x0 - 1 : 0);
    };
    double planes = 0.0;
    const bool alike = mean && nchunk > 4;  // (the inner chunks are)
    for (int c = 0; c < (alike ? 3 : nchunk); ++c) planes += planes_of(c);
    if (alike) planes *= (double)nchunk / 3;
    // columns at an end of v, of those left at an end of y, inner ones
    const int nv = P.ncol_v < 2 ? 1 : 2, ny = ncol_y < 2 ? 1 : 2, inner = P.ncol_v - nv;
    const double share = planes * (ncol_y * nv * end_v + inner * (ny * 1.1 + (ncol_y - ny))) / n;
    if (mean || share > limit) return share;
    double load[1024] = {0.0}, most = 0.0;
    int shift = 0, place = 0;
    for (int c = 0; c < nchunk; ++c) {
        const int np = planes_of(c);
        for (int iy = 0; iy < ncol_y; ++iy) {
            const double wy = np * (iy == 0 || iy == ncol_y - 1 ? 1.1 : 1.0), wv = np * end_v;
            for (int iv = 0; iv < P.ncol_v; ++iv) {
                const int cta = place >= shift ? place - shift : place + n - shift;
                load[cta] += iv == 0 || iv == P.ncol_v - 1 ? wv : wy;
                if (load[cta] > most) {
                    most = load[cta];
                    if (most > limit) return most;
                }
                if (++place == n) {
                    place = 0;
                    if (++shift == n) shift = 0;
                }
            }
        }
    }
    return most;
}

// Estimated time of a step (in us, up to what all shapes of a grid share) for
// the default tile: (rounds of items) x (planes one item loads) x (time of a
// plane).  A plane costs a fixed part (the waits on its stage and the release)
// and a part per consumer warp that depends on the launch-bound class, which
// sets the registers; the forms that read V0 as a field also pay for the bytes
// through shared memory.  Below 8 warps (11 with several rows a thread) an SM
// is latency-bound and a plane takes as long as with that many.  In fixed
// point the tiles' costs differ and the CTA with the heaviest items sets the
// time.  Coefficients: least squares over the 20 to 40 shapes that
// hj_autotune timed on each of 10 grids (2 to 101 M cells; 18 in fixed point):
// the FP32 ones of the present kernels, the fixed-point ones of the kernel
// before a warp took one form of the update.
// Against the best timed shape of each grid the picks take 1.00 to 1.03 times
// as long with a 4D V0 (mean 1.01), 1.00 to 1.11 (1.02; 6 of the 16 grids not
// in the fit) with the field and 1.00 to 1.18 (1.04) in fixed point (1.00 to
// 1.11 with the kernel of the fit; a fit to the present kernel with the 736
// class gained up to 15 % on 7 of the 18 grids and lost up to 14 % on 4); the shape with the fewest halo reads per
// row, the rule before, took 1.00 to 1.33 (1.13), 1.03 to 1.26 (1.16) and 1.00
// to 1.74 (1.22).  Per step, that rule and this one: 80x80x25x40 FP32 18.4 and
// 15.4 us, 128x128x64x96 with the field 156 and 141, 128x128x30x16 with the
// field 20.3 and 17.9.
// A shape that a lower bound (no item order loads fewer planes than ncol n1 /
// slots per CTA, none is cheaper than an inner one) shows to cost more than
// `limit` returns that bound.
double step_cost(const hj_grid *g, const TiledParams &P, int slots, int xc_req, double limit)
{
    static const double F4D[4] = {0.0089, 0.0111, 0.0148, 0.0210}, FXY[4] = {0.0169, 0.0147, 0.0176, 0.0209},
                        Q[4] = {0.0326, 0.0300, 0.0296, 0.0357};
    const bool fixed = g->prec == HJ_Q527;
    int cls = 0;
    while (cls < 3 && P.nconsumer > hj_tiled_variant(fixed, cls)) ++cls;
    const double least = P.rpt > 1 ? 11 : 8, warps = P.nconsumer / 32 > least ? P.nconsumer / 32 : least;
    double plane;  // time of a plane (fixed point: and `planes` times 0.25)
    if (fixed) {
        plane = warps * Q[cls];
    } else if (!g->v0_bcast) {
        plane = warps * F4D[cls] + 0.2875;
    } else {
        const double per_warp = P.rpt == 1 ? FXY[cls] : (P.rpt == 2 ? 2 * 0.0204 : 4 * 0.0152);
        plane = warps * per_warp + 0.00497 * ((P.halo_box + g->p4 * P.ty * P.tv) / 256.0) + 0.1425;
    }
    const double bound = (1.0 - 1e-9) * P.ncol * g->n[0] / slots * (plane + (fixed ? 0.25 : 0.0));
    if (bound > limit) return bound;
    const int xc = xc_req > 0 && xc_req < g->n[0] ? xc_req : (xc_req > 0 ? g->n[0] : best_chunk(g, P.ncol, slots));
    const int nchunk = (g->n[0] + xc - 1) / xc;
    const long long rounds = ((long long)P.ncol * nchunk + slots - 1) / slots;
    const double planes = (double)rounds * (xc + (nchunk > 1 ? 2 : 1));
    if (!fixed) return planes * plane;
    const double rest = planes * 0.25;
    return heaviest_q527(g, P, xc, nchunk, slots, (limit - rest) / plane) * plane + rest;
}

// The shape with the least step_cost() for a request that leaves one extent or
// both (req[0], req[1] <= 0) open.  Large tiles first: they cost least on most
// grids, and the others' bounds then show it (set-up of a Q5.27 grid of
// 128x128x64x96 228 -> 143 us, 131 with the rule before step_cost(); of equal
// shapes the smaller one counts).
void default_shape(const hj_grid *g, int slots, int maxsmem, const int32_t *req, int *ty, int *tv)
{
    const bool fixed = g->prec == HJ_Q527;
    const int cap = hj_tiled_variant(fixed, 2);
    double best = 1e300;
    int bty = 1, btv = 1;
    for (int a = g->n[1] < 16 ? g->n[1] : 16; a >= 1; --a)
        for (int b = g->n[2] < 16 ? g->n[2] : 16; b >= 1; --b) {
            if ((req[0] > 0 && a != req[0]) || (req[1] > 0 && b != req[1])) continue;
            const TiledParams C = make_params(g, a, b, 1, 0);
            // (fixed point: tiles of one or two rows along an axis measured slower
            // than the estimate, 70x90x40x72 69 us at 15 x 2, 61 at 6 x 5; an extent
            // that is requested is taken as it is)
            const bool thin = fixed && ((req[0] <= 0 && a < 3) || (req[1] <= 0 && b < 3));
            const bool fits = !thin && C.nconsumer <= cap && 4 * (size_t)C.stage_bytes + 2048 <= (size_t)maxsmem;
            if (!fits && !(a == 1 && b == 1)) continue;
            const double c = fits ? step_cost(g, C, slots, req[2], best) : 1e299;
            if (c <= best) {
                best = c;
                bty = a;
                btv = b;
            }
        }
    *ty = bty;
    *tv = btv;
}

size_t tiled_smem_bytes(const TiledParams &P)
{
    return (size_t)P.stages * P.stage_bytes + 2 * MAX_STAGES * sizeof(uint64_t) + 32 * sizeof(unsigned long long) +
           32;
}

// Whether every theta quad has one sign of cos and of sin (lanes whose value
// is exactly 0 after hj_flush_trig carry no weight and count as either);
// also writes the quads' dominant signs into tab_sign[4 * q].
bool sign_uniform(const hj_grid *g, float *tab_sign)
{
    const int N4 = g->n[3];
    double cmax = 0, smax = 0;
    for (int l = 0; l < N4; ++l) {
        const double th = g->lo[3] + (double)l * g->h[3];
        cmax = fmax(cmax, fabs(hj_flush_trig(cos(th))));
        smax = fmax(smax, fabs(hj_flush_trig(sin(th))));
    }
    bool ok = true;
    for (int q = 0; q < g->p4 / 4; ++q) {
        double bc = 0, bs = 0;
        int sc = 1, ss = 1;
        for (int e = 0; e < 4 && 4 * q + e < N4; ++e) {
            const double th = g->lo[3] + (double)(4 * q + e) * g->h[3];
            const double c = hj_flush_trig(cos(th)), sn = hj_flush_trig(sin(th));
            if (fabs(c) > bc) bc = fabs(c), sc = c >= 0 ? 1 : -1;
            if (fabs(sn) > bs) bs = fabs(sn), ss = sn >= 0 ? 1 : -1;
        }
        for (int e = 0; e < 4 && 4 * q + e < N4; ++e) {
            const double th = g->lo[3] + (double)(4 * q + e) * g->h[3];
            // lanes whose weight is exactly 0 may sit on either side
            const double c = hj_flush_trig(cos(th)), s = hj_flush_trig(sin(th));
            if (c != 0.0 && (c >= 0 ? 1 : -1) != sc) ok = false;
            if (s != 0.0 && (s >= 0 ? 1 : -1) != ss) ok = false;
        }
        tab_sign[4 * q + 0] = (float)sc;
        tab_sign[4 * q + 1] = (float)ss;
        tab_sign[4 * q + 2] = 0.f;
        tab_sign[4 * q + 3] = 0.f;
    }
    return ok;
}

}  // namespace

int hj_tiled_threads(const hj_grid *g, int ty, int tv)
{
    const int nc = consumers_of(g, ty, tv);
    return nc <= max_consumers(g->prec == HJ_Q527) ? nc + 32 : 0;
}

int hj_tiled_variant(bool fixed, int i) { return fixed ? VARIANTS_Q527[i] : VARIANTS_F32[i]; }

bool hj_tiled_setup(hj_grid *g, char *why, size_t why_len)
{
    ++g->launch_version;  // tile, tensor maps or kernel variant may change: captured step graphs are stale
    auto fail = [&](const char *m) {
        snprintf(why, why_len, "%s", m);
        return false;
    };
    if (g->prec != HJ_FP32 && g->prec != HJ_Q527) return fail("tiled kernel is FP32 or Q5.27 only");
    const bool fixed = g->prec == HJ_Q527;
    if (g->periodic != 0x8u) return fail("tiled kernel needs theta (axis 4) periodic and x, y, v not");
    if (!g->has_dyn || (g->dyn != HJ_DYN_CAR4D && g->dyn != HJ_DYN_CAR4D_STEER))
        return fail("tiled kernel needs the car dynamics");
    if (g->p4 > 256) return fail("theta rows longer than 256 points");
    if (g->nint >= (1LL << 34)) return fail("grid of 2^34 stored values or more (32-bit float4 indices)");
    EncodeTiledFn enc = get_encode_fn();
    if (!enc) return fail("cuTensorMapEncodeTiled unavailable");

    int sms = 0, maxsmem = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device);
    cudaDeviceGetAttribute(&maxsmem, cudaDevAttrMaxSharedMemoryPerBlockOptin, g->device);

    // quad signs: tab_tiled holds v_k [n3], cos/dx1 [p4], sin/dx2 [p4], then
    // the (cos, sin) sign of each quad's dominant lane [p4]
    float *sgn = (float *)calloc((size_t)g->p4, sizeof(float));
    if (!sgn) return fail("host allocation failed");
    // the single-sided (USIGN) form also needs every speed >= 0 (a negative
    // speed flips the upwind side); otherwise the general form runs
    g->sign_uniform = sign_uniform(g, sgn);
    const bool usign = !fixed && g->lo[2] >= 0.0 && g->sign_uniform;
    cudaError_t e = cudaMemcpy(g->tab_tiled + g->n[2] + 2 * g->p4, sgn, sizeof(float) * g->p4, cudaMemcpyHostToDevice);
    free(sgn);
    if (e != cudaSuccess) return fail("sign table upload failed");
    g->tiled_usign = usign;  // a property of the grid's v and theta ranges (read by tiled_rpt)

    // tile shape: one consumer thread per (row, theta quad) (per two or four v
    // rows in the several-row forms), at most the largest launch-bound class
    // (+ the producer warp).  By default the shape with the least step_cost()
    // among those that fit the largest class without spills (640 consumer
    // threads; 608 in fixed point) and leave room for 4 stages, and as many
    // stages as fit; hj_autotune measures the candidates instead.
    const int q4 = g->p4 / 4;
    if (max_consumers(fixed) / q4 < 1) return fail("theta rows too long for one CTA");
    const int32_t *req = g->tile_req[g->v0_bcast];
    int ty = req[0], tv = req[1];
    if (ty <= 0 || tv <= 0) default_shape(g, sms > 0 ? sms : 1, maxsmem, req, &ty, &tv);
    if (tv > g->n[2]) tv = g->n[2];
    if (ty > g->n[1]) ty = g->n[1];
    while (consumers_of(g, ty, tv) > max_consumers(fixed) && ty > 1) --ty;
    while (consumers_of(g, ty, tv) > max_consumers(fixed) && tv > 1) --tv;
    int stages = req[3];
    if (stages <= 0) {  // as many as fit in shared memory, up to MAX_STAGES
        TiledParams P1 = make_params(g, ty, tv, 1, 0);
        stages = (int)((maxsmem - 2048) / P1.stage_bytes);
        if (stages > MAX_STAGES) stages = MAX_STAGES;
    }
    if (stages < 4 || stages > MAX_STAGES) return fail("stage count out of range");
    TiledParams P = make_params(g, ty, tv, stages, 0);
    if (P.nconsumer > max_consumers(fixed)) return fail("tile needs too many threads");
    size_t smem = tiled_smem_bytes(P);
    if ((int)smem > maxsmem) return fail("tile does not fit in shared memory");
    const void *fn = (const void *)kernel_fn(fixed, g->p4 != g->n[3], usign, g->v0_bcast, false, P.nconsumer, P.rpt);
    const void *fn_track =
        (const void *)kernel_fn(fixed, g->p4 != g->n[3], usign, g->v0_bcast, true, P.nconsumer, P.rpt);
    // (the limit belongs to the kernel, not to the grid: always the largest, so that
    // a grid set up later with a smaller ring does not lower it under this one's)
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsmem) != cudaSuccess ||
        cudaFuncSetAttribute(fn_track, cudaFuncAttributeMaxDynamicSharedMemorySize, maxsmem) != cudaSuccess)
        return fail("cannot raise the shared-memory limit");
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, P.nconsumer + 32, smem) != cudaSuccess ||
        per_sm < 1)
        return fail("tile shape does not fit on an SM");
    const int slots = sms * per_sm;
    const int xc = req[2] > 0 ? req[2] : best_chunk(g, P.ncol, slots);
    P = make_params(g, ty, tv, stages, xc);

    // tensor maps, dims (p4, n3, n2, n1): V0 / buffer A / buffer B with the
    // halo box, and V0 with the halo-free box
    cuuint64_t dims[4] = {(cuuint64_t)g->p4, (cuuint64_t)g->n[2], (cuuint64_t)g->n[1], (cuuint64_t)g->n[0]};
    cuuint64_t strides[3] = {(cuuint64_t)g->p4 * 4, (cuuint64_t)g->p4 * g->n[2] * 4,
                             (cuuint64_t)g->p4 * g->n[2] * g->n[1] * 4};
    cuuint32_t box_halo[4] = {(cuuint32_t)g->p4, (cuuint32_t)(tv + 2), (cuuint32_t)(ty + 2), 1};
    cuuint32_t box_tile[4] = {(cuuint32_t)g->p4, (cuuint32_t)tv, (cuuint32_t)ty, 1};
    cuuint32_t estr[4] = {1, 1, 1, 1};
    void *bases[4] = {g->v0, g->buf, (char *)g->buf + (size_t)g->nint * 4, g->v0};
    for (int i = 0; i < 4; ++i) {
        CUresult r = enc(&g->tmap[i], fixed ? CU_TENSOR_MAP_DATA_TYPE_INT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4,
                         bases[i], dims, strides,
                         i < 3 ? box_halo : box_tile, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            snprintf(why, why_len, "cuTensorMapEncodeTiled failed (%d)", (int)r);
            return false;
        }
    }
    g->tile_ty = ty;
    g->tile_tv = tv;
    g->tile_xc = P.xc;
    g->tile_stages = stages;
    g->tiled_ctas = P.nitems < slots ? P.nitems : slots;
    g->tiled_per_sm = per_sm;
    g->tiled_usign = usign;
    return true;
}

cudaError_t hj_launch_step_tiled(hj_grid *g, long long n, int sel)
{
    const TiledParams P = make_params(g, g->tile_ty, g->tile_tv, g->tile_stages, g->tile_xc);
    KernelFn fn =
        kernel_fn(g->prec == HJ_Q527, g->p4 != g->n[3], g->tiled_usign, g->v0_bcast, g->track, P.nconsumer, P.rpt);
    // a programmatic dependent of the previous launch on the stream: the
    // kernel sets up its ring while the previous step drains and waits for
    // that step's completion before it reads anything it wrote
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)g->tiled_ctas);
    cfg.blockDim = dim3((unsigned)(P.nconsumer + 32));
    cfg.dynamicSmemBytes = tiled_smem_bytes(P);
    cfg.stream = g->stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const CUtensorMap &in = n == 0 ? g->tmap[0] : g->tmap[1 + (int)((n - 1) & 1)];
    const int32_t *qw = g->qw ? g->qw + sel * hj_qw_count(g->n[2], g->p4) : nullptr;
    return cudaLaunchKernelEx(&cfg, fn, in, g->tmap[3], (float *)hj_value_ptr(g, n + 1), (const float *)g->tab_tiled,
                              qw, (const float *)g->v0xy, (const void *)g->k4tab, g->loop, sel, g->dflags, g->geom,
                              P);
}
