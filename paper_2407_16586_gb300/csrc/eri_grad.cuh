// What the derivative-ERI class kernels share (one template instance per
// angular class (la lb|lc ld) with la >= lb, lc >= ld and bra pair class >= ket
// pair class: the 21 non-redundant classes for l <= 2, Sec. II.C): the Boys
// function of the fp32 route, the per-quartet screen, and the launch of the
// CTA-wide forms.
#pragma once
#include "tg_internal.cuh"

namespace tg {

// Boys function F_m(T), m = 0..M, for the fp32 route.  Below T = 1 everything
// runs in fp64; for 1 <= T < 36 the top order comes from a Taylor step of the
// fp32 table and the downward recursion F_m = (2T F_{m+1} + e^-T)/(2m+1) runs in
// fp64; for T >= 36 the upward recursion is stable and runs in fp32.  Relative
// accuracy ~1e-7 (the fp32 seed).  e^-T comes from the fp64 table instead of
// exp(), which alone cost as many fp64 instructions as the rest: below 1 from
// (2M+1) F_M - 2T F_{M+1}, above from the same identity at the grid point (orders
// 15 and 16) times a six-term series of e^(T0-T), |T0 - T| <= 0.025, good to
// 2e-12 (the difference cancels towards T = 36; exp() was good to 1e-16), far
// below the 6e-8 of the fp32 seed and of the rounded values.
template <int M>
__device__ __forceinline__ void boys_mixed(float T, float (&F)[M + 1], const double *__restrict__ tab)
{
    if (T < 1.0f) {
        const double Td = (double)T;
        const int i = __double2int_rn(Td * (1.0 / BOYS_H));
        const double d = i * BOYS_H - Td;
        const double *row = tab + i * (BOYS_M + 1) + M;
        double hi = row[BOYS_TAYLOR + 1], f = row[BOYS_TAYLOR];
#pragma unroll
        for (int k = BOYS_TAYLOR - 1; k >= 0; --k) {
            const double dk = d * (1.0 / (k + 1));
            hi = row[k + 1] + hi * dk;
            f = row[k] + f * dk;
        }
        const double t2 = 2.0 * Td, et = (2 * M + 1) * f - t2 * hi;
        F[M] = (float)f;
#pragma unroll
        for (int m = M - 1; m >= 0; --m) {
            f = (t2 * f + et) * (1.0 / (2 * m + 1));
            F[m] = (float)f;
        }
        return;
    }
    if (T < (float)BOYS_TMAX) {
        const float *ftab = reinterpret_cast<const float *>(tab + BOYS_TAB);
        const int i = __float2int_rn(T * (float)(1.0 / BOYS_H));
        const float d = (float)i * (float)BOYS_H - T;
        const float *row = ftab + i * (BOYS_M + 1) + M;
        float acc = row[BOYS_TAYLOR];
#pragma unroll
        for (int k = BOYS_TAYLOR - 1; k >= 0; --k) acc = row[k] + acc * d * (1.0f / (k + 1));
        F[M] = acc;
        const double Td = (double)T;
        const double dd = i * BOYS_H - Td;  // T0 - T
        const double *r64 = tab + i * (BOYS_M + 1);
        double et = 1.0 / 720.0;
        et = et * dd + 1.0 / 120.0;
        et = et * dd + 1.0 / 24.0;
        et = et * dd + 1.0 / 6.0;
        et = et * dd + 0.5;
        et = et * dd + 1.0;
        et = et * dd + 1.0;
        et *= (2 * BOYS_M - 1) * r64[BOYS_M - 1] - 2.0 * BOYS_H * i * r64[BOYS_M];
        const double t2 = 2.0 * Td;
        double f = (double)acc;
#pragma unroll
        for (int m = M - 1; m >= 0; --m) {
            f = (t2 * f + et) * (1.0 / (2 * m + 1));
            F[m] = (float)f;
        }
    } else {
        const float it = 1.0f / T;
        F[0] = 0.88622692545275801365f * sqrtf(it);
        const float et = __expf(-T);
        const float h = 0.5f * it;
#pragma unroll
        for (int m = 0; m < M; ++m) F[m + 1] = ((2 * m + 1) * F[m] - et) * h;
    }
}

// Per-quartet screening bound (see tdgrad.h) and shard membership.
__device__ __forceinline__ bool keep_quartet(const ScreenArgs &scr, const PairSet &bra, const PairSet &ket, int bi,
                                             int ki, int sa, int sb, int sc, int sd)
{
    if (scr.nranks > 1) {
        const int key = max(bra.key[bi], ket.key[ki]);
        if (key % scr.nranks != scr.rank) return false;
    }
    if (scr.tau > 0.0) {
        const double S = fmax(bra.Qd[bi] * ket.Q[ki], bra.Q[bi] * ket.Qd[ki]);
        const int ns = scr.nshell;
        const double *M = scr.M;
        double Mq = M[(size_t)sa * ns + sb];
        Mq = fmax(Mq, M[(size_t)sc * ns + sd]);
        Mq = fmax(Mq, M[(size_t)sa * ns + sc]);
        Mq = fmax(Mq, M[(size_t)sa * ns + sd]);
        Mq = fmax(Mq, M[(size_t)sb * ns + sc]);
        Mq = fmax(Mq, M[(size_t)sb * ns + sd]);
        const double bound = scr.scale * S * Mq * Mq;
        if (bound < scr.tau) return false;
    }
    return true;
}

// Dynamic shared memory a CTA of a class kernel may take (227 KB less 4 KB for
// static arrays).  Every launch allows its kernel this much, whatever it needs
// itself: the attribute belongs to the kernel in the whole context, and a value
// of the launch's own would refuse a larger molecule's launch of another thread
// that had set it just before.
constexpr size_t kCtaSmem = 223 * 1024;

template <typename K>
cudaError_t allow_cta_smem(K kern, size_t sm)
{
    if (sm > kCtaSmem) return cudaErrorInvalidValue;
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCtaSmem);
}

// Shared memory of a CTA-wide form: its arrays beside smem, the tile staging
// with, where out.use_smem says so, the gradient of the largest molecule.
// Where the three together pass the limit (the 99 KB of (dd|pp) from 4 747 atoms)
// the gradient stays in the CTA's slab.
inline size_t unit_smem(size_t arrays, size_t smem, OutArgs &out)
{
    if (out.use_smem && arrays + smem > kCtaSmem) {
        out.use_smem = 0;
        smem -= sizeof(double) * 3 * (size_t)out.natom_max;
    }
    return arrays + smem;
}

// Launch of a persistent class kernel over units: the grid is the smaller of
// gcap and the kernel's resident CTAs per SM times the SM count, and each
// tile is cut into nchunk x nsplit units (nchunk only for the cooperative
// kernel, whose CTA holds ngroups quartets at a time) until there are at
// least four units per CTA, so that classes with few tiles still fill the
// GPU.  Dump mode keeps one unit per tile.
template <typename K>
cudaError_t launch_units(K kern, int ngroups, int gcap, size_t sm, cudaStream_t st, const MolDesc *mols,
                         ClassLaunch cl, const OutArgs &out, const double *boys, int block = TILE)
{
    cudaError_t e = allow_cta_smem(kern, sm);
    if (e != cudaSuccess) return e;
    int dev = 0, nsm = 1, per = 1;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, block, sm)) != cudaSuccess) return e;
    long long gmax = (long long)(per > 0 ? per : 1) * nsm;
    if (gmax > gcap) gmax = gcap;
    cl.nchunk = 1;
    cl.nsplit = 1;
    if (!out.dump) {
        const long long want = 4 * gmax;
        if (ngroups > 0)
            while (cl.ntiles * cl.nchunk < want && cl.nchunk * ngroups < TILE) cl.nchunk *= 2;
        while (cl.ntiles * cl.nchunk * cl.nsplit < want && cl.nsplit < 16) ++cl.nsplit;
        if (cl.split_req > 0) cl.nsplit = cl.split_req;
    }
    const long long units = cl.ntiles * cl.nchunk * cl.nsplit;
    const int grid = (int)(units < gmax ? units : gmax);
    kern<<<grid, block, sm, st>>>(mols, cl, out, boys);
    return cudaGetLastError();
}

}  // namespace tg
