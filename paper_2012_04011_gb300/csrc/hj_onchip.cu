// Host side of the on-chip step kernel (hj_onchip.cuh): which grids it takes,
// how they are cut into blocks, and its launch.
#include "hj_onchip.cuh"

using namespace hj_onchip;

namespace {

constexpr unsigned long long WAIT_NS = 2000000000ull;  // 2 s per wait for a neighbour

constexpr int MAX_THREADS = 768;

typedef void (*KernelFn)(const float *, float *, const void *, const int32_t *, const void *, const HjLoop *,
                         HjFlags *, const HjGeom, const Params, long long, unsigned int *, unsigned long long);

// [Q5.27][some theta quad has both signs of cos or of sin][padded rows]
const KernelFn KERNELS[2][2][2] = {
    {{onchip_kernel<false, false, false, MAX_THREADS>, onchip_kernel<false, false, true, MAX_THREADS>},
     {onchip_kernel<false, true, false, MAX_THREADS>, onchip_kernel<false, true, true, MAX_THREADS>}},
    {{onchip_kernel<true, false, false, MAX_THREADS>, onchip_kernel<true, false, true, MAX_THREADS>},
     {onchip_kernel<true, true, false, MAX_THREADS>, onchip_kernel<true, true, true, MAX_THREADS>}}};

size_t block_bytes(const hj_grid *g, int bx, int by)
{
    return ((size_t)bx * by * 2 + 2 * bx + 2 * by) * g->n[2] * g->p4 * 4 + (size_t)bx * by * 4;
}

KernelFn kernel_of(const hj_grid *g) { return KERNELS[g->prec == HJ_Q527][!g->sign_uniform][g->p4 != g->n[3]]; }

}  // namespace

// Cuts the grid into blocks of bx x by columns, one per SM at most, or leaves
// oc_bx = 0: the kernel takes FP32 and Q5.27 car grids with periodic theta
// whose blocks fit in shared memory with at most MAX_THREADS theta quads per
// x row of blocks.  Among the cuts that fit, the one with the least
//     by (500 + 32 warps) + 300 bx
// clocks per step, fitted to measured steps: a column of quads costs each
// thread about 500 clocks of latency and each warp 32 of the SM's
// shared-memory and issue bandwidth; rows along y are what the threads copy
// and publish as y halos.  (40x40x16x24: 4 x 3 columns 2.9 us, 3 x 4 3.2, 6 x 2
// 3.3; 50x50x20x30: 4 x 5 4.5, 2 x 9 5.3.)  Two CTAs per SM, half the block
// each, measured the same (40x50x20x32: 3.6 against 3.7 us) and are not used.
void hj_onchip_setup(hj_grid *g)
{
    g->oc_bx = 0;
    if ((g->prec != HJ_FP32 && g->prec != HJ_Q527) || g->periodic != 0x8u || !g->has_dyn ||
        g->geom.mode3 != HJ_AXIS_CONTROL || g->geom.mode4 != HJ_AXIS_CONTROL || g->p4 > 256 ||
        g->nint >= (1LL << 31))
        return;
    int sms = 0, maxsmem = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device);
    cudaDeviceGetAttribute(&maxsmem, cudaDevAttrMaxSharedMemoryPerBlockOptin, g->device);
    if (sms > HJ_SYNC_CTAS) sms = HJ_SYNC_CTAS;
    const int smem_cap = maxsmem - 1024;
    double best = 1e300;
    for (int bx = 1; bx <= g->n[0]; ++bx) {
        const int threads = (bx * g->n[2] * (g->p4 / 4) + 31) / 32 * 32;
        if (threads > MAX_THREADS) break;
        const int gx = (g->n[0] + bx - 1) / bx;
        for (int by = 1; by <= g->n[1] && (long long)block_bytes(g, bx, by) <= smem_cap; ++by) {
            if ((long long)gx * ((g->n[1] + by - 1) / by) > sms) continue;
            const double cost = by * (500.0 + threads) + 300.0 * bx;
            if (cost >= best) continue;
            best = cost;
            g->oc_bx = bx;
            g->oc_by = by;
        }
    }
    if (g->oc_bx > 0 && cudaFuncSetAttribute((const void *)kernel_of(g), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             smem_cap) != cudaSuccess) {
        cudaGetLastError();
        g->oc_bx = 0;
    }
}

cudaError_t hj_launch_onchip(hj_grid *g, long long n, long long k, bool cut)
{
    const int gx = (g->n[0] + g->oc_bx - 1) / g->oc_bx, gy = (g->n[1] + g->oc_by - 1) / g->oc_by;
    const int threads = (g->oc_bx * g->n[2] * (g->p4 / 4) + 31) / 32 * 32;
    Params P;
    P.bx = g->oc_bx;
    P.by = g->oc_by;
    P.gy = gy;
    P.steps = (int)k;
    P.cut = cut ? 1 : 0;
    P.pub_all = (g->n[0] - 1) % P.bx == 0 || (g->n[1] - 1) % P.by == 0;
    P.n0 = n;
    P.k3 = (float)g->geom.k3;
    const float *v0 = (const float *)g->v0;
    float *buf = (float *)g->buf;
    const void *coef = g->coef, *k4 = g->k4tab;
    const int32_t *qw = g->qw;
    const HjLoop *lp = g->loop;
    HjFlags *flags = g->dflags;
    HjGeom geom = g->geom;
    long long nint = g->nint;
    unsigned int *prog = g->rsync->prog;
    unsigned long long limit = WAIT_NS;
    void *args[] = {&v0, &buf, &coef, &qw, &k4, &lp, &flags, &geom, &P, &nint, &prog, &limit};
    return cudaLaunchCooperativeKernel((const void *)kernel_of(g), gx * gy, threads, args,
                                       block_bytes(g, P.bx, P.by), g->stream);
}
