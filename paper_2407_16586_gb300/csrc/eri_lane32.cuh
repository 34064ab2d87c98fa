// fp32 derivative-ERI class kernel: one warp per contracted quartet, one
// primitive quartet per lane.
//
// Algebra (McMurchie-Davidson, both operators s = 1/r and erf(w r)/r), for a bra
// primitive pair p and a ket primitive pair q:
//   F_s[cd][h1] = sum_ab Gamma_s[ab][cd] E^{ab}_{h1}(p)                       (per p, on the warp)
//   y[ab][h1]   = sum_h2 (-1)^|h2| [sum_cd Gamma_s[ab][cd] E^{cd}_{h2}(q)] R_s[h1+h2]
//   z[cd][h2]   = (-1)^|h2| sum_h1 F_s[cd][h1] R_s[h1+h2]
// d/dA and d/dA + d/dB are short dot products with y (eq. deriv, the R-tensor
// shift), d/dC with z; d/dB and d/dD follow from translational invariance
// (eq. ti).  The scaled Hermite basis R'_h = R_h / s^{|h|}, s = sqrt(2 rho),
// keeps every intermediate within fp32 range for any exponent; the factors
// s^{|h|} move onto the short Hermite vectors.  Every primitive quartet's
// contribution is added in fp64, so the result does not depend on how primitive
// quartets are dealt to lanes, up to fp64 rounding.
//
// Why lanes: one thread per contracted quartet kept its Gamma and F rows (15.6 KB
// for (dp|dp)) in local memory and walked up to 36 x 36 primitive quartets one
// after the other; the warp shares them in shared memory (2.6 KB, and 2.9 KB a bra
// primitive pair), and a list of a few hundred contracted quartets fills the GPU
// (fp32 lists of the 6-atom workload on the learned route: 114.5 -> 16.8 ms; of a
// 1/8 shard of the 32-atom workload: 178.6 -> 127.8 ms).  Bound: instruction
// supply -- the unrolled y and z loops of a warp are 16 KB of code, walked by each
// warp on its own ((dp|pp): 6.5 of 9.6 cycles per instruction wait for it, FMA pipe
// 13 %) -- and in the classes up to (pp|ps) the fp64 pipe of the Boys recursion.
#pragma once
#include "eri_herm.cuh"

namespace tg {

template <int LA, int LB, int LC, int LD>
struct Lane32Lay {
    static constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
    static constexpr int NAB = NA * NB, NCD = NC * ND, L1 = LA + LB, L2 = LC + LD, L = L1 + L2;
    static constexpr int NH1 = nherm(L1), E1 = L1 + 2, EBN = (LA + 2) * (LB + 1) * E1;
    static constexpr int RS = 33;
    static constexpr int NP1 = 6;                                  // p, K, P - A (3), 2 zeta_a
    static constexpr int PER_P = 2 * NCD * NH1 + 3 * EBN + NP1;    // floats of one bra primitive pair
    static constexpr int PB_RAW = 2400 / PER_P;                    // bra primitive pairs of a block, 1 to 16
    static constexpr int PB = PB_RAW < 1 ? 1 : (PB_RAW > 16 ? 16 : PB_RAW);
    static constexpr int o_gam = 0;                                // floats: [2][NAB][NCD]
    static constexpr int o_P = o_gam + 2 * NAB * NCD;              // [PB][PER_P]: F [2][NCD][NH1], E tables, scalars
    static constexpr int FLOATS = o_P + PB * PER_P;
    static constexpr int o_X = (FLOATS + 1) / 2;                   // doubles: the closing sums
    static constexpr int TOTAL = (o_X + 9 * RS + 1) & ~1;          // doubles
    static constexpr size_t BYTES = sizeof(double) * (size_t)TOTAL;
};

// Contribution of one primitive quartet: bra primitive pair pf, Kab, PA, za2
// with its F rows and 1-D tables Eb, ket primitive pair kp.
template <int LA, int LB, int LC, int LD>
__device__ __forceinline__ void prim_fp32(const float *gam, const float *Fr, const float *Eb, float pf, float Kab,
                                          float PAx, float PAy, float PAz, float za2, const PrimPairs &pp, int kp,
                                          float ACx, float ACy, float ACz, int nops, float om2f, bool ominf,
                                          const double *boys, float (&qA)[3], float (&qC)[3], float (&qT)[3])
{
    using Lay = Lane32Lay<LA, LB, LC, LD>;
    constexpr int NB = Lay::NB, ND = Lay::ND, NAB = Lay::NAB, NCD = Lay::NCD;
    constexpr int L1 = Lay::L1, L2 = Lay::L2, L = Lay::L;
    constexpr int NH1 = Lay::NH1, NH1P = nherm(L1 + 1), NH2 = nherm(L2), NH2P = nherm(L2 + 1);
    constexpr int NR = nherm(L + 1), E1 = Lay::E1, E2 = L2 + 2;
    const long long nr = pp.n;
    const float qf = pp.fp[kp], Kcd = pp.fK[kp];
    const float QCx = pp.fPA[kp], QCy = pp.fPA[nr + kp], QCz = pp.fPA[2 * nr + kp];
    const float zc2 = 2.0f * pp.fza[kp];
    float Ek[3][LC + 2][LD + 1][L2 + 2];
    etab<LC + 1, LD>(Ek[0], QCx, pp.fPB[kp], 0.5f / qf);
    etab<LC + 1, LD>(Ek[1], QCy, pp.fPB[nr + kp], 0.5f / qf);
    etab<LC + 1, LD>(Ek[2], QCz, pp.fPB[2 * nr + kp], 0.5f / qf);
    const float pq = pf + qf, rho = pf * qf / pq;
    const float Xd = PAx - QCx + ACx, Yd = PAy - QCy + ACy, Zd = PAz - QCz + ACz;
    const float T = rho * (Xd * Xd + Yd * Yd + Zd * Zd);
    const float sc_ = sqrtf(2.0f * rho);
    const float pref = 34.986836655249725f * rsqrtf(pq) / (pf * qf) * Kab * Kcd;
    float spow[L + 3];
    spow[0] = 1.0f;
#pragma unroll
    for (int n = 1; n <= L + 2; ++n) spow[n] = spow[n - 1] * sc_;
    // ket products E^{cd}_{h2} s^{|h2|} (-1)^{|h2|}
    float E3k[NCD][NH2];
    for (int cd = 0; cd < NCD; ++cd) {
        const int mc = cd / ND, md = cd % ND;
        const int cq = (mc == 0) ? 0 : (mc < 3 ? 1 : 2), dq = (md == 0) ? 0 : (md < 3 ? 1 : 2);
        const int cy = cq - (mc - cq * (cq + 1) / 2), cx = LC - cq, cz = LC - cx - cy;
        const int dy = dq - (md - dq * (dq + 1) / 2), dx = LD - dq, dz = LD - dx - dy;
        float kx[E2], ky[E2], kz[E2];
#pragma unroll
        for (int t = 0; t < E2; ++t) {
            kx[t] = t <= cx + dx ? Ek[0][cx][dx][t] : 0.0f;
            ky[t] = t <= cy + dy ? Ek[1][cy][dy][t] : 0.0f;
            kz[t] = t <= cz + dz ? Ek[2][cz][dz][t] : 0.0f;
        }
#pragma unroll
        for (int t = 0; t <= L2; ++t)
#pragma unroll
            for (int u = 0; u <= L2 - t; ++u)
#pragma unroll
                for (int v = 0; v <= L2 - t - u; ++v) {
                    const float w = ((t + u + v) & 1) ? -spow[t + u + v] : spow[t + u + v];
                    E3k[cd][hidx(t, u, v)] = kx[t] * ky[u] * kz[v] * w;
                }
    }
                            for (int o = 0; o < nops; ++o) {
        float R[NR];
        {
            const float th2 = (o == 0) ? 1.0f : (ominf ? 1.0f : om2f / (om2f + rho));
            float Fm[L + 2], base[L + 2];
            boys_mixed<L + 1>(T * th2, Fm, boys);
            float f = pref * sqrtf(th2);
#pragma unroll
            for (int n = 0; n <= L + 1; ++n) {
                base[n] = (n & 1) ? -f * Fm[n] : f * Fm[n];
                f *= th2;
            }
            hermite_R<L + 1>(R, base, Xd * sc_, Yd * sc_, Zd * sc_);
        }
        // ---- bra side: y^{ab} (registers), then d/dA and d/dP
        for (int ab = 0; ab < NAB; ++ab) {
            float gr[NH2];
#pragma unroll
            for (int h = 0; h < NH2; ++h) gr[h] = 0.0f;
            for (int k = 0; k < NCD; ++k) {
                const float gm = gam[(o * NAB + ab) * NCD + k];
#pragma unroll
                for (int h = 0; h < NH2; ++h) gr[h] += gm * E3k[k][h];
            }
            float y[NH1P];
#pragma unroll
            for (int h = 0; h < NH1P; ++h) y[h] = 0.0f;
#pragma unroll
            for (int t2 = 0; t2 <= L2; ++t2)
#pragma unroll
                for (int u2 = 0; u2 <= L2 - t2; ++u2)
#pragma unroll
                    for (int v2 = 0; v2 <= L2 - t2 - u2; ++v2) {
                        const float c0 = gr[hidx(t2, u2, v2)];
#pragma unroll
                        for (int t1 = 0; t1 <= L1 + 1; ++t1)
#pragma unroll
                            for (int u1 = 0; u1 <= L1 + 1 - t1; ++u1)
#pragma unroll
                                for (int v1 = 0; v1 <= L1 + 1 - t1 - u1; ++v1)
                                    y[hidx(t1, u1, v1)] += c0 * R[hidx(t1 + t2, u1 + u2, v1 + v2)];
                    }
            const int ma = ab / NB, mb = ab % NB;
            const int aq = (ma == 0) ? 0 : (ma < 3 ? 1 : 2), bq = (mb == 0) ? 0 : (mb < 3 ? 1 : 2);
            const int ay = aq - (ma - aq * (aq + 1) / 2), ax = LA - aq, az = LA - ax - ay;
            const int by = bq - (mb - bq * (bq + 1) / 2), bx = LB - bq, bz = LB - bx - by;
            // rows: plain E (zero beyond i+j) and derivative DA = 2a E^{i+1} - i E^{i-1}
            float ex[E1], ey[E1], ez[E1], dx[E1], dy[E1], dz[E1];
#pragma unroll
            for (int t = 0; t < E1; ++t) {
                ex[t] = t <= ax + bx ? Eb[((0 * (LA + 2) + ax) * (LB + 1) + bx) * E1 + t] : 0.0f;
                ey[t] = t <= ay + by ? Eb[((1 * (LA + 2) + ay) * (LB + 1) + by) * E1 + t] : 0.0f;
                ez[t] = t <= az + bz ? Eb[((2 * (LA + 2) + az) * (LB + 1) + bz) * E1 + t] : 0.0f;
                dx[t] = za2 * Eb[((0 * (LA + 2) + ax + 1) * (LB + 1) + bx) * E1 + t] - (ax > 0 ? ax * Eb[((0 * (LA + 2) + ax - 1) * (LB + 1) + bx) * E1 + t] : 0.0f);
                dy[t] = za2 * Eb[((1 * (LA + 2) + ay + 1) * (LB + 1) + by) * E1 + t] - (ay > 0 ? ay * Eb[((1 * (LA + 2) + ay - 1) * (LB + 1) + by) * E1 + t] : 0.0f);
                dz[t] = za2 * Eb[((2 * (LA + 2) + az + 1) * (LB + 1) + bz) * E1 + t] - (az > 0 ? az * Eb[((2 * (LA + 2) + az - 1) * (LB + 1) + bz) * E1 + t] : 0.0f);
            }
            // y_{tuv} s^{t+u+v}, contracted: sum_v (e_z, d_z, shifted e_z) then u, then t
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, q0 = 0.f, q1 = 0.f, q2 = 0.f;
#pragma unroll
            for (int t = 0; t <= L1 + 1; ++t) {
                float ux = 0.f, uy = 0.f, uz = 0.f, vy = 0.f, vz = 0.f;
#pragma unroll
                for (int u = 0; u <= L1 + 1 - t; ++u) {
                    float sE = 0.f, sD = 0.f, sS = 0.f;
#pragma unroll
                    for (int v = 0; v <= L1 + 1 - t - u; ++v) {
                        const float yy = y[hidx(t, u, v)] * spow[t + u + v];
                        if (v < E1) {
                            sE += ez[v] * yy;
                            sD += dz[v] * yy;
                        }
                        if (v >= 1) sS += ez[v - 1] * yy;
                    }
                    ux += ey[u] * sE;  // -> d/dA_x (with dx[t]) and d/dP_x (t-1)
                    uy += dy[u] * sE;  // -> d/dA_y
                    uz += ey[u] * sD;  // -> d/dA_z
                    vz += ey[u] * sS;  // -> d/dP_z
                    if (u >= 1) vy += ey[u - 1] * sE;  // -> d/dP_y
                }
                a0 += dx[t] * ux;
                a1 += ex[t] * uy;
                a2 += ex[t] * uz;
                if (t >= 1) q0 += ex[t - 1] * ux;
                q1 += ex[t] * vy;
                q2 += ex[t] * vz;
            }
            qA[0] += a0;
            qA[1] += a1;
            qA[2] += a2;
            qT[0] += q0;
            qT[1] += q1;
            qT[2] += q2;
        }
        // ---- ket side: z^{cd} (registers), then d/dC
        for (int cd = 0; cd < NCD; ++cd) {
            float z[NH2P];
#pragma unroll
            for (int h = 0; h < NH2P; ++h) z[h] = 0.0f;
#pragma unroll
            for (int t1 = 0; t1 <= L1; ++t1)
#pragma unroll
                for (int u1 = 0; u1 <= L1 - t1; ++u1)
#pragma unroll
                    for (int v1 = 0; v1 <= L1 - t1 - u1; ++v1) {
                        const float f0 = Fr[(o * NCD + cd) * NH1 + hidx(t1, u1, v1)] * spow[t1 + u1 + v1];
#pragma unroll
                        for (int t2 = 0; t2 <= L2 + 1; ++t2)
#pragma unroll
                            for (int u2 = 0; u2 <= L2 + 1 - t2; ++u2)
#pragma unroll
                                for (int v2 = 0; v2 <= L2 + 1 - t2 - u2; ++v2)
                                    z[hidx(t2, u2, v2)] += f0 * R[hidx(t1 + t2, u1 + u2, v1 + v2)];
                    }
            const int mc = cd / ND, md = cd % ND;
            const int cq = (mc == 0) ? 0 : (mc < 3 ? 1 : 2), dq = (md == 0) ? 0 : (md < 3 ? 1 : 2);
            const int cy = cq - (mc - cq * (cq + 1) / 2), cx = LC - cq, cz = LC - cx - cy;
            const int dy_ = dq - (md - dq * (dq + 1) / 2), dx_ = LD - dq, dz_ = LD - dx_ - dy_;
            float kx[E2], ky[E2], kz[E2], jx[E2], jy[E2], jz[E2];
#pragma unroll
            for (int t = 0; t < E2; ++t) {
                kx[t] = t <= cx + dx_ ? Ek[0][cx][dx_][t] : 0.0f;
                ky[t] = t <= cy + dy_ ? Ek[1][cy][dy_][t] : 0.0f;
                kz[t] = t <= cz + dz_ ? Ek[2][cz][dz_][t] : 0.0f;
                jx[t] = zc2 * Ek[0][cx + 1][dx_][t] - (cx > 0 ? cx * Ek[0][cx - 1][dx_][t] : 0.0f);
                jy[t] = zc2 * Ek[1][cy + 1][dy_][t] - (cy > 0 ? cy * Ek[1][cy - 1][dy_][t] : 0.0f);
                jz[t] = zc2 * Ek[2][cz + 1][dz_][t] - (cz > 0 ? cz * Ek[2][cz - 1][dz_][t] : 0.0f);
            }
            float c0 = 0.f, c1 = 0.f, c2 = 0.f;
#pragma unroll
            for (int t = 0; t <= L2 + 1; ++t) {
                float ux = 0.f, uy = 0.f, uz = 0.f;
#pragma unroll
                for (int u = 0; u <= L2 + 1 - t; ++u) {
                    float sE = 0.f, sD = 0.f;
#pragma unroll
                    for (int v = 0; v <= L2 + 1 - t - u; ++v) {
                        const int n = t + u + v;
                        const float zz = (n & 1) ? -z[hidx(t, u, v)] * spow[n] : z[hidx(t, u, v)] * spow[n];
                        sE += kz[v] * zz;
                        sD += jz[v] * zz;
                    }
                    ux += ky[u] * sE;
                    uy += jy[u] * sE;
                    uz += ky[u] * sD;
                }
                c0 += jx[t] * ux;
                c1 += kx[t] * uy;
                c2 += kx[t] * uz;
            }
            qC[0] += c0;
            qC[1] += c1;
            qC[2] += c2;
        }
    }
}

template <int LA, int LB, int LC, int LD>
__device__ void quartet_lane32(double *sm, int lane, const GeoArgs &geo, const DensArgs &den, const PrimPairs &pp,
                               int sa, int sb, int sc, int sd, int pb0, int nbp, int ib0, int ibs, int pk0, int nkp,
                               double scale, const double *boys, double (&acc)[9])
{
    using Lay = Lane32Lay<LA, LB, LC, LD>;
    constexpr int NB = Lay::NB, ND = Lay::ND, NAB = Lay::NAB, NCD = Lay::NCD, NH1 = Lay::NH1, E1 = Lay::E1;
    constexpr int EBN = Lay::EBN, PER_P = Lay::PER_P;
    float *gam = reinterpret_cast<float *>(sm) + Lay::o_gam, *P = reinterpret_cast<float *>(sm) + Lay::o_P;
    const int nbf = den.nbf, nops = den.use_lr ? 2 : 1;
    const float om2f = (float)(den.omega * den.omega);
    const bool ominf = isinf(den.omega);
    const double *xa = geo.xyz + 3 * geo.sh_atom[sa], *xc = geo.xyz + 3 * geo.sh_atom[sc];
    const float ACx = (float)(xa[0] - xc[0]), ACy = (float)(xa[1] - xc[1]), ACz = (float)(xa[2] - xc[2]);
    const long long nr = pp.n;
    const int fa = geo.sh_bf[sa], fb = geo.sh_bf[sb], fc = geo.sh_bf[sc], fd = geo.sh_bf[sd];
    // ---- Gamma of both operators
    for (int it = lane; it < NAB * NCD; it += 32) {
        const int ab = it / NCD, cd = it % NCD;
        const size_t m = fa + ab / NB, n = fb + ab % NB, l = fc + cd / ND, s = fd + cd % ND;
        double g0 = 0.0, g1 = 0.0;
        for (int p = 0; p < den.npair; ++p) {
            const double *A = den.A[p], *B = den.B[p];
            const double cj = den.cJ[p] * scale, ck = den.cK[p] * scale, cl = den.cKlr[p] * scale;
            if (cj != 0.0)
                g0 += cj * (den.S[p][m * nbf + n] * den.T[p][l * nbf + s] + den.S[p][l * nbf + s] * den.T[p][m * nbf + n]);
            if (ck != 0.0 || cl != 0.0) {
                const double kk = A[m * nbf + l] * B[n * nbf + s] + A[n * nbf + l] * B[m * nbf + s] +
                                  A[m * nbf + s] * B[n * nbf + l] + A[n * nbf + s] * B[m * nbf + l] +
                                  A[l * nbf + m] * B[s * nbf + n] + A[s * nbf + m] * B[l * nbf + n] +
                                  A[l * nbf + n] * B[s * nbf + m] + A[s * nbf + n] * B[l * nbf + m];
                g0 += ck * kk;
                g1 += cl * kk;
            }
        }
        gam[it] = (float)g0;
        gam[NAB * NCD + it] = (float)g1;
    }
    const int nbra = (nbp - ib0 + ibs - 1) / ibs;
    const int pb = block_pairs(nbra, nkp, Lay::PB);
    double fA[3] = {0.0, 0.0, 0.0}, fC[3] = {0.0, 0.0, 0.0}, fT[3] = {0.0, 0.0, 0.0};
    __syncwarp();
    for (int blk = 0; blk < nbra; blk += pb) {
        const int np = min(pb, nbra - blk);
        // ---- 1-D tables and scalars of the block's bra primitive pairs, then F
        for (int it = lane; it < 3 * np; it += 32) {
            const int pi = it / 3, dir = it % 3;
            const int ip = pb0 + ib0 + (blk + pi) * ibs;
            float *q = P + pi * PER_P + 2 * NCD * NH1;
            const float pf = pp.fp[ip], PA = pp.fPA[dir * nr + ip];
            float E[LA + 2][LB + 1][E1];
            etab<LA + 1, LB>(E, PA, pp.fPB[dir * nr + ip], 0.5f / pf);
#pragma unroll
            for (int i = 0; i <= LA + 1; ++i)
#pragma unroll
                for (int j = 0; j <= LB; ++j)
#pragma unroll
                    for (int t = 0; t < E1; ++t) q[((dir * (LA + 2) + i) * (LB + 1) + j) * E1 + t] = E[i][j][t];
            float *s = q + 3 * EBN;
            s[2 + dir] = PA;
            if (dir == 0) {
                s[0] = pf;
                s[1] = pp.fK[ip];
                s[5] = 2.0f * pp.fza[ip];
            }
        }
        __syncwarp();
        for (int it = lane; it < np * NCD * NH1; it += 32) {
            const int pi = it / (NCD * NH1), r = it % (NCD * NH1), k = r / NH1;
            float *F = P + pi * PER_P;
            const float *Eb = F + 2 * NCD * NH1;
            int t, u, v;
            herm_tuv(r % NH1, t, u, v);
            float s0 = 0.0f, s1 = 0.0f;
            for (int ab = 0; ab < NAB; ++ab) {
                int ax, ay, az, bx, by, bz;
                cart_xyz(LA, ab / NB, ax, ay, az);
                cart_xyz(LB, ab % NB, bx, by, bz);
                float e = 0.0f;
                if (t <= ax + bx && u <= ay + by && v <= az + bz)
                    e = Eb[(ax * (LB + 1) + bx) * E1 + t] * Eb[(((LA + 2) + ay) * (LB + 1) + by) * E1 + u] *
                        Eb[((2 * (LA + 2) + az) * (LB + 1) + bz) * E1 + v];
                s0 += gam[ab * NCD + k] * e;
                s1 += gam[(NAB + ab) * NCD + k] * e;
            }
            F[r] = s0;
            F[NCD * NH1 + r] = s1;
        }
        __syncwarp();
        const int ntot = np * nkp;
        for (int idx = lane; idx < ntot; idx += 32) {
            const int pi = idx / nkp;
            const float *F = P + pi * PER_P, *Eb = F + 2 * NCD * NH1, *s = Eb + 3 * EBN;
            float qA[3] = {0.f, 0.f, 0.f}, qC[3] = {0.f, 0.f, 0.f}, qT[3] = {0.f, 0.f, 0.f};
            prim_fp32<LA, LB, LC, LD>(gam, F, Eb, s[0], s[1], s[2], s[3], s[4], s[5], pp, pk0 + (idx - pi * nkp), ACx,
                                      ACy, ACz, nops, om2f, ominf, boys, qA, qC, qT);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                fA[i] += (double)qA[i];
                fC[i] += (double)qC[i];
                fT[i] += (double)qT[i];
            }
        }
        __syncwarp();  // the block's arrays are rewritten for the next one
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc[i] += fA[i];
        acc[3 + i] += fT[i];
        acc[6 + i] += fC[i];
    }
}

template <int LA, int LB, int LC, int LD>
struct Lane32Op {
    using Lay = Lane32Lay<LA, LB, LC, LD>;
    static constexpr bool FP32 = true;
    static constexpr int L = LA + LB + LC + LD;
    static constexpr int KQ = 1, NW = 1, cta_workers = L <= 3 ? 2 : 1, min_ctas = L == 3 ? 6 : 8;
    static constexpr int group_below = 0;
    static __device__ __forceinline__ void group(double *sm, int lane, int k0, int, const GroupInfo &gi, const MolDesc &md,
                                                 int sa, int sb, int pb0, int nbp, int ib0, int ibs, const double *boys,
                                                 double (&acc)[9])
    {
        quartet_lane32<LA, LB, LC, LD>(sm, lane, md.geo, md.den, md.pp, sa, sb, gi.sc[k0], gi.sd[k0], pb0, nbp, ib0, ibs,
                                       gi.pk0[k0], gi.nk[k0], gi.scale[k0], boys, acc);
    }
};

// The kernel form of a class.  fp64: the Hermite-density kernel.  fp32: the lane
// kernel, but the warp kernel for (dd|pp) and (dd|ds) and the group kernel for
// (dd|dp) and (dd|dd), whose order of fp32 sums differs from the lane kernel's:
// the routed results stay what they were.
template <int LA, int LB, int LC, int LD>
cudaError_t launch_class_kernel(int fp32, int gcap, size_t smem, cudaStream_t st, const MolDesc *mols,
                                const ClassLaunch &cl, const OutArgs &out, const double *boys)
{
    constexpr int nfq = ncart(LA) * ncart(LB) * ncart(LC) * ncart(LD);
    constexpr bool group = nfq >= 648, warp = (LA + LB == 4) && nfq >= 216 && nfq < 648;
    if (!fp32) return launch_lanes<HermOp<LA, LB, LC, LD>>(gcap, st, mols, cl, out, boys);
    if constexpr (warp)
        return launch_warp<LA, LB, LC, LD>(gcap, smem, st, mols, cl, out, boys);
    else if constexpr (group)
        return launch_coop<LA, LB, LC, LD>(gcap, smem, st, mols, cl, out, boys);
    else
        return launch_lanes<Lane32Op<LA, LB, LC, LD>>(gcap, st, mols, cl, out, boys);
}

}  // namespace tg
