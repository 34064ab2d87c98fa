// Learned block router: tile features, MLP inference, and the training loop
// (forward + backward, fixed-order gradient reduction, Adam), all on the GPU.
// The router predicts log10 of a quartet tile's largest gradient
// contribution; it only decides fp32 vs fp64 for a tile and never skips work.
#include "router.cuh"

namespace tg {

__device__ __forceinline__ float lg10(double x) { return (float)log10(x > 1e-300 ? x : 1e-300); }

// 16 features of one quartet tile (TB bra pairs x TK ket pairs of one class).
__global__ void k_tile_features(int ntiles, const TileRef *tiles, FeatureArgs fa, float *feat)
{
    const int it = blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= ntiles) return;
    const TileRef t = tiles[it];
    const PairSet &bra = fa.sets[t.P], &ket = fa.sets[t.Q];
    const int b0 = t.bt * TB, b1 = min(bra.n, b0 + TB), k0 = t.kt * TK, k1 = min(ket.n, k0 + TK);
    double qb = 0, qdb = 0, qk = 0, qdk = 0, mb = 0, mk = 0, mx = 0, ab = 0, cd = 0, pb = 1e300, pk = 1e300;
    double dmin = 1e300;
    const int ns = fa.nshell;
    for (int i = b0; i < b1; ++i) {
        qb = fmax(qb, bra.Q[i]);
        qdb = fmax(qdb, bra.Qd[i]);
        const int a = bra.sa[i], b = bra.sb[i];
        mb = fmax(mb, fa.M[(size_t)a * ns + b]);
        const double *A = fa.xyz + 3 * fa.sh_atom[a], *B = fa.xyz + 3 * fa.sh_atom[b];
        const double r = sqrt((A[0] - B[0]) * (A[0] - B[0]) + (A[1] - B[1]) * (A[1] - B[1]) + (A[2] - B[2]) * (A[2] - B[2]));
        ab = fmax(ab, r);
        for (int k = 0; k < bra.np[i]; ++k) pb = fmin(pb, fa.pp_p[bra.poff[i] + k]);
    }
    for (int j = k0; j < k1; ++j) {
        qk = fmax(qk, ket.Q[j]);
        qdk = fmax(qdk, ket.Qd[j]);
        const int c = ket.sa[j], d = ket.sb[j];
        mk = fmax(mk, fa.M[(size_t)c * ns + d]);
        const double *C = fa.xyz + 3 * fa.sh_atom[c], *D = fa.xyz + 3 * fa.sh_atom[d];
        const double r = sqrt((C[0] - D[0]) * (C[0] - D[0]) + (C[1] - D[1]) * (C[1] - D[1]) + (C[2] - D[2]) * (C[2] - D[2]));
        cd = fmax(cd, r);
        for (int k = 0; k < ket.np[j]; ++k) pk = fmin(pk, fa.pp_p[ket.poff[j] + k]);
    }
    for (int i = b0; i < b1; ++i) {
        const int a = bra.sa[i], b = bra.sb[i];
        const double *A = fa.xyz + 3 * fa.sh_atom[a], *B = fa.xyz + 3 * fa.sh_atom[b];
        for (int j = k0; j < k1; ++j) {
            const int c = ket.sa[j], d = ket.sb[j];
            mx = fmax(mx, fa.M[(size_t)a * ns + c]);
            mx = fmax(mx, fa.M[(size_t)a * ns + d]);
            mx = fmax(mx, fa.M[(size_t)b * ns + c]);
            mx = fmax(mx, fa.M[(size_t)b * ns + d]);
            const double *C = fa.xyz + 3 * fa.sh_atom[c], *D = fa.xyz + 3 * fa.sh_atom[d];
            double dd = 0.0;
            for (int x = 0; x < 3; ++x) {
                const double u = 0.5 * (A[x] + B[x]) - 0.5 * (C[x] + D[x]);
                dd += u * u;
            }
            dmin = fmin(dmin, dd);
        }
    }
    const double Mt = fmax(fmax(mb, mk), mx);
    const double bnd = fa.scale * fmax(qdb * qk, qb * qdk) * Mt * Mt;
    float *f = feat + (size_t)it * NFEAT;
    f[0] = (float)(pc_la(t.P) + pc_lb(t.P) + pc_la(t.Q) + pc_lb(t.Q)) * 0.125f;
    f[1] = lg10(bnd);
    f[2] = lg10(qb);
    f[3] = lg10(qk);
    f[4] = lg10(qdb);
    f[5] = lg10(qdk);
    f[6] = lg10(mx);
    f[7] = lg10(mb);
    f[8] = lg10(mk);
    f[9] = (float)(sqrt(dmin) * 0.1);
    f[10] = (float)(ab * 0.1);
    f[11] = (float)(cd * 0.1);
    f[12] = lg10(pb);
    f[13] = lg10(pk);
    f[14] = log2f((float)bra.np[b0]);
    f[15] = log2f((float)ket.np[k0]);
}

// The same features for the tiles of a device-built list, from tables: what
// belongs to one side of a tile is formed once per bra and ket tile, the 512
// block factors of a tile become 16 reads of its bra tile's row of maxima, and
// pair centres are kept.  The values are those of k_tile_features, bit for bit
// (maxima and the square root commute; the centre differences are formed alike).
// Bound: the fp64 pipe (the 128 centre distances, 6 instructions each).  The plan
// of the 300-atom workload (3.1e7 tiles), of which features took 184 ms, went
// from 231 to 97 ms.
// One pair per thread, bsz (8 or 16) threads a tile: a thread that walks the up to
// 16 x 36 primitive pairs of a tile alone waits 30 us for its loads.
__global__ void k_side_features(int bsz, PairSet ps, FeatureArgs fa, SideFeature *out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, t = i / bsz, lo = t * bsz;
    double q = 0, qd = 0, m = 0, e2 = 0, p = 1e300;
    if (i < ps.n) {
        q = ps.Q[i];
        qd = ps.Qd[i];
        const int a = ps.sa[i], b = ps.sb[i];
        m = fa.M[(size_t)a * fa.nshell + b];
        const double *A = fa.xyz + 3 * fa.sh_atom[a], *B = fa.xyz + 3 * fa.sh_atom[b];
        e2 = (A[0] - B[0]) * (A[0] - B[0]) + (A[1] - B[1]) * (A[1] - B[1]) + (A[2] - B[2]) * (A[2] - B[2]);
        for (int k = 0; k < ps.np[i]; ++k) p = fmin(p, fa.pp_p[ps.poff[i] + k]);
    }
    for (int o = bsz / 2; o > 0; o /= 2) {
        q = fmax(q, __shfl_xor_sync(0xffffffffu, q, o));
        qd = fmax(qd, __shfl_xor_sync(0xffffffffu, qd, o));
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        e2 = fmax(e2, __shfl_xor_sync(0xffffffffu, e2, o));
        p = fmin(p, __shfl_xor_sync(0xffffffffu, p, o));
    }
    if (i != lo || lo >= ps.n) return;
    SideFeature f;
    f.q = q;
    f.qd = qd;
    f.m = m;
    f.lq = lg10(q);
    f.lqd = lg10(qd);
    f.lm = lg10(m);
    f.extent = (float)(sqrt(e2) * 0.1);
    f.lp = lg10(p);
    f.lnp = log2f((float)ps.np[lo]);
    out[t] = f;
}

__global__ void k_pair_centres(PairSet ps, const double *xyz, const int *sh_atom, double *cen)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ps.n) return;
    const double *A = xyz + 3 * sh_atom[ps.sa[i]], *B = xyz + 3 * sh_atom[ps.sb[i]];
    for (int x = 0; x < 3; ++x) cen[(size_t)x * ps.n + i] = 0.5 * (A[x] + B[x]);
}

// mx[bra tile][c] = max of M[x][c] over the shells x of the tile's pairs; one
// block per bra tile
__global__ void k_bra_density_max(PairSet ps, const double *M, int ns, double *mx)
{
    __shared__ int sh[2 * TB];
    const int lo = blockIdx.x * TB, n = min(ps.n, lo + TB) - lo;
    if (threadIdx.x < n) {
        sh[threadIdx.x] = ps.sa[lo + threadIdx.x];
        sh[n + threadIdx.x] = ps.sb[lo + threadIdx.x];
    }
    __syncthreads();
    for (int c = threadIdx.x; c < ns; c += blockDim.x) {
        double m = 0.0;
        for (int k = 0; k < 2 * n; ++k) m = fmax(m, M[(size_t)sh[k] * ns + c]);
        mx[(size_t)blockIdx.x * ns + c] = m;
    }
}

// One tile per thread; neighbours share the bra tile, so its data come by
// broadcast.  Non-negative doubles are compared as integers (no fp64 pipe).
__global__ void __launch_bounds__(128) k_tile_features_tab(long long n, const uint4 *__restrict__ tiles, FeatureArgs fa,
                                                           FeatureTables ft, float *__restrict__ feat)
{
    const long long it = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (it >= n) return;
    const uint4 t = tiles[it];
    const int P = ft.P[t.w], Q = ft.Q[t.w];
    const int nb = fa.sets[P].n, nk = fa.sets[Q].n;
    const int b0 = t.y * TB, b1 = min(nb, b0 + TB), k0 = t.z * TK, kn = min(nk, k0 + TK) - k0;
    const SideFeature sb = ft.bra[P][t.y], sk = ft.ket[Q][t.z];
    const int *sc = fa.sets[Q].sa + k0, *sd = fa.sets[Q].sb + k0;
    const long long *mrow = reinterpret_cast<const long long *>(ft.mx[P] + (size_t)t.y * fa.nshell);
    const double *cb = ft.cen[P], *ck = ft.cen[Q] + k0;
    double kx[TK], ky[TK], kz[TK];
    long long mx = 0;
#pragma unroll
    for (int j = 0; j < TK; ++j) {
        const int k = min(j, kn - 1);  // a ragged tile repeats its last pair
        kx[j] = ck[k];
        ky[j] = ck[(size_t)nk + k];
        kz[j] = ck[2 * (size_t)nk + k];
        mx = max(mx, max(mrow[sc[k]], mrow[sd[k]]));
    }
    long long dmin = __double_as_longlong(1e300);
    for (int i = b0; i < b1; ++i) {
        const double x = cb[i], y = cb[(size_t)nb + i], z = cb[2 * (size_t)nb + i];
#pragma unroll
        for (int j = 0; j < TK; ++j) {
            const double u = x - kx[j], v = y - ky[j], w = z - kz[j];
            dmin = min(dmin, __double_as_longlong(fma(w, w, fma(v, v, u * u))));
        }
    }
    const double dmx = __longlong_as_double(mx);
    const double Mt = fmax(fmax(sb.m, sk.m), dmx);
    const double bnd = fa.scale * fmax(sb.qd * sk.q, sb.q * sk.qd) * Mt * Mt;
    float *f = feat + (size_t)it * NFEAT;
    f[0] = (float)(pc_la(P) + pc_lb(P) + pc_la(Q) + pc_lb(Q)) * 0.125f;
    f[1] = lg10(bnd);
    f[2] = sb.lq;
    f[3] = sk.lq;
    f[4] = sb.lqd;
    f[5] = sk.lqd;
    f[6] = lg10(dmx);
    f[7] = sb.lm;
    f[8] = sk.lm;
    f[9] = (float)(sqrt(__longlong_as_double(dmin)) * 0.1);
    f[10] = sb.extent;
    f[11] = sk.extent;
    f[12] = sb.lp;
    f[13] = sk.lp;
    f[14] = sb.lnp;
    f[15] = sk.lnp;
}

// Feature standardisation statistics (mean, std) in a fixed order.
__global__ void k_feature_stats(int n, const float *X, float *mu, float *sd)
{
    const int j = threadIdx.x;
    if (j >= NFEAT) return;
    double s = 0.0, s2 = 0.0;
    for (int i = 0; i < n; ++i) {
        const double v = X[(size_t)i * NFEAT + j];
        s += v;
        s2 += v * v;
    }
    const double m = n > 0 ? s / n : 0.0;
    const double var = n > 0 ? s2 / n - m * m : 1.0;
    mu[j] = (float)m;
    sd[j] = (float)sqrt(var > 1e-12 ? var : 1.0);
}

__device__ __forceinline__ void mlp_forward(const float *w, const float *x, float *h1, float *h2, float &y)
{
    const float *W1 = w, *b1 = W1 + NH * NFEAT, *W2 = b1 + NH, *b2 = W2 + NH * NH, *w3 = b2 + NH, *b3 = w3 + NH;
    for (int i = 0; i < NH; ++i) {
        float a = b1[i];
        for (int j = 0; j < NFEAT; ++j) a += W1[i * NFEAT + j] * x[j];
        h1[i] = tanhf(a);
    }
    for (int i = 0; i < NH; ++i) {
        float a = b2[i];
        for (int j = 0; j < NH; ++j) a += W2[i * NH + j] * h1[j];
        h2[i] = tanhf(a);
    }
    float a = b3[0];
    for (int j = 0; j < NH; ++j) a += w3[j] * h2[j];
    y = a;
}

__global__ void k_mlp_predict(int n, const float *X, const float *mu, const float *sd, const float *params, float *out)
{
    __shared__ float w[NPARAM];
    for (int k = threadIdx.x; k < NPARAM; k += blockDim.x) w[k] = params[k];
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float x[NFEAT], h1[NH], h2[NH], y;
    for (int j = 0; j < NFEAT; ++j) x[j] = (X[(size_t)i * NFEAT + j] - mu[j]) / sd[j];
    mlp_forward(w, x, h1, h2, y);
    out[i] = y;
}

// Forward + backward of the expectile loss for TRB samples per block; the
// block's parameter gradient (sum over its samples, divided by n) and loss
// go to partial slots, reduced later in a fixed order.
__global__ void __launch_bounds__(TRB) k_mlp_fwd_bwd(int n, const float *X, const float *y, const float *mu,
                                                     const float *sd, const float *params, float q, float *gpart,
                                                     float *lpart)
{
    extern __shared__ float sm[];
    float *w = sm;                          // NPARAM
    float *sx = w + NPARAM;                 // TRB x NFEAT
    float *s1 = sx + TRB * NFEAT;           // TRB x NH  (h1, then da1)
    float *s2 = s1 + TRB * NH;              // TRB x NH  (h2, then da2)
    float *sdy = s2 + TRB * NH;             // TRB
    float *sl = sdy + TRB;                  // TRB
    float *sa1 = sl + TRB;                  // TRB x NH (da1)
    for (int k = threadIdx.x; k < NPARAM; k += blockDim.x) w[k] = params[k];
    __syncthreads();
    const int s = threadIdx.x;
    const int i = blockIdx.x * TRB + s;
    const float *W2 = w + NH * NFEAT + NH, *w3 = W2 + NH * NH + NH;
    if (i < n) {
        float x[NFEAT], h1[NH], h2[NH], yh;
        for (int j = 0; j < NFEAT; ++j) x[j] = (X[(size_t)i * NFEAT + j] - mu[j]) / sd[j];
        mlp_forward(w, x, h1, h2, yh);
        const float r = y[i] - yh;
        const float wt = r > 0.f ? q : 1.f - q;
        sl[s] = wt * r * r / n;
        const float dy = -2.f * wt * r / n;
        sdy[s] = dy;
        float da2[NH];
        for (int k = 0; k < NH; ++k) da2[k] = dy * w3[k] * (1.f - h2[k] * h2[k]);
        for (int j = 0; j < NH; ++j) {
            float a = 0.f;
            for (int k = 0; k < NH; ++k) a += W2[k * NH + j] * da2[k];
            sa1[s * NH + j] = a * (1.f - h1[j] * h1[j]);
        }
        for (int j = 0; j < NFEAT; ++j) sx[s * NFEAT + j] = x[j];
        for (int k = 0; k < NH; ++k) {
            s1[s * NH + k] = h1[k];
            s2[s * NH + k] = h2[k];
        }
        for (int k = 0; k < NH; ++k) s2[s * NH + k] = h2[k];
        // da2 kept in a second pass below through s2 (h2) and sdy
    } else {
        sl[s] = 0.f;
        sdy[s] = 0.f;
        for (int j = 0; j < NFEAT; ++j) sx[s * NFEAT + j] = 0.f;
        for (int k = 0; k < NH; ++k) {
            s1[s * NH + k] = 0.f;
            s2[s * NH + k] = 0.f;
            sa1[s * NH + k] = 0.f;
        }
    }
    __syncthreads();
    const int nvalid = min(TRB, n - blockIdx.x * TRB);
    float *gp = gpart + (size_t)blockIdx.x * NPARAM;
    // each thread owns parameters k = threadIdx.x + m*TRB and sums over the block's samples in order
    for (int k = threadIdx.x; k < NPARAM; k += TRB) {
        float acc = 0.f;
        if (k < NH * NFEAT) {  // W1[i][j] += da1[i] x[j]
            const int ii = k / NFEAT, j = k % NFEAT;
            for (int t = 0; t < nvalid; ++t) acc += sa1[t * NH + ii] * sx[t * NFEAT + j];
        } else if (k < NH * NFEAT + NH) {  // b1
            const int ii = k - NH * NFEAT;
            for (int t = 0; t < nvalid; ++t) acc += sa1[t * NH + ii];
        } else if (k < NH * NFEAT + NH + NH * NH) {  // W2[i][j] += da2[i] h1[j]
            const int kk = k - NH * NFEAT - NH, ii = kk / NH, j = kk % NH;
            for (int t = 0; t < nvalid; ++t) {
                const float h2v = s2[t * NH + ii];
                const float da2 = sdy[t] * w3[ii] * (1.f - h2v * h2v);
                acc += da2 * s1[t * NH + j];
            }
        } else if (k < NH * NFEAT + NH + NH * NH + NH) {  // b2
            const int ii = k - NH * NFEAT - NH - NH * NH;
            for (int t = 0; t < nvalid; ++t) {
                const float h2v = s2[t * NH + ii];
                acc += sdy[t] * w3[ii] * (1.f - h2v * h2v);
            }
        } else if (k < NPARAM - 1) {  // w3
            const int ii = k - NH * NFEAT - NH - NH * NH - NH;
            for (int t = 0; t < nvalid; ++t) acc += sdy[t] * s2[t * NH + ii];
        } else {  // b3
            for (int t = 0; t < nvalid; ++t) acc += sdy[t];
        }
        gp[k] = acc;
    }
    if (threadIdx.x == 0) {
        float L = 0.f;
        for (int t = 0; t < nvalid; ++t) L += sl[t];
        lpart[blockIdx.x] = L;
    }
}

__global__ void k_sum_partials(int nblocks, int width, const float *part, float *out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= width) return;
    double s = 0.0;
    for (int b = 0; b < nblocks; ++b) s += part[(size_t)b * width + k];
    out[k] = (float)s;
}

__global__ void k_adam(int n, float *params, const float *grad, float *m, float *v, float lr, float b1, float b2,
                       float eps, int step)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const float g = grad[k];
    const float mk = b1 * m[k] + (1.f - b1) * g;
    const float vk = b2 * v[k] + (1.f - b2) * g * g;
    m[k] = mk;
    v[k] = vk;
    const float mh = mk / (1.f - powf(b1, (float)step));
    const float vh = vk / (1.f - powf(b2, (float)step));
    params[k] -= lr * mh / (sqrtf(vh) + eps);
}

}  // namespace tg
