// Fock-type build (Sec. II.B, the two-electron part of eqs. G_2e and zfock):
// one warp per canonical shell quartet, one primitive quartet per lane.
//
// The density pairs are combined beforehand (the result is linear in them)
// into S_J = sum_p c_J (B_p + B_p^T), B_K = sum_p c_K B_p and B_lr =
// sum_p c_K_lr B_p.  Per canonical quartet (a b|c d) the integrals
// I_s(m n|l s) of both operators s come from the monomial sums of
// eri_herm.cuh: V_s[m1][m2] = sum_pq s_m1(p) s_m2(q) (-1)^|h2| R_s[h1 + h2]
// over the primitive quartets, and once per contracted quartet
// I_s[ab][cd] = sum_m1m2 c^{ab}_{m1} R^.. V_s[m1][m2] c^{cd}_{m2} S^...  The 8
// permutation images of every integral give
//   Coulomb:  F[m][n], F[n][m] += I_0 S_J[l][s];   F[l][s], F[s][l] += I_0 S_J[m][n]
//   exchange: F[m][l] += I.B[n][s]   F[n][l] += I.B[m][s]   F[m][s] += I.B[n][l]
//             F[n][s] += I.B[m][l]   F[l][m] += I.B[s][n]   F[s][m] += I.B[l][n]
//             F[l][n] += I.B[s][m]   F[s][n] += I.B[l][m]
// with I.B = I_0 B_K + I_1 B_lr, all times 1/|stabiliser| of the quartet.
// Each target block is summed over the quartet on the warp and added to F
// with fp64 atomics.  Bound: the fp64 pipe, as the gradient kernel.
#pragma once
#include "eri_lane32.cuh"

namespace tg {

// One warp's slice of shared memory, in doubles (as HermLay).
template <int LA, int LB, int LC, int LD>
struct FockLay {
    using B = PairMono<LA, LB>;
    using K = PairMono<LC, LD>;
    static constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
    static constexpr int NAB = NA * NB, NCD = NC * ND, L = B::L + K::L;
    static constexpr int NM1 = B::NM, NM2 = K::NM, NS1 = B::NS, NS2 = K::NS, NM2P = NM2 | 1, RS = 33;
    static constexpr int NRH = nherm(L), PB = 16, NP1 = 2;
    static constexpr int NE1 = pair_entries(LA, LB), NE2 = pair_entries(LC, LD);
    static constexpr int NO = (NAB * NCD <= 81) ? 2 : 1;  // operators at a time
    static constexpr int HALF = NE1 + NE2 + NO * NM1 * NCD, ROWS = (NRH + NS2) * RS;
    static constexpr int o_I = 0;                            // [2][NAB][NCD]
    static constexpr int o_V = o_I + 2 * NAB * NCD;          // [NO][NM1][NM2P]
    static constexpr int o_S1 = o_V + NO * NM1 * NM2P;       // [PB][NS1]
    static constexpr int o_P1 = o_S1 + PB * NS1;             // [PB][NP1]: p, 2 pi^(5/2) K / p
    static constexpr int o_pw = o_P1 + PB * NP1;             // [2][3][5] powers of R and S
    static constexpr int o_X = o_pw + 30;
    static constexpr int TOTAL = (o_X + (HALF > ROWS ? HALF : ROWS) + 1) & ~1;
    static constexpr size_t BYTES = sizeof(double) * (size_t)TOTAL;
};

// Per-quartet Fock bound: 8 Q_ab Q_cd M_q (see tg_fock2e in tdgrad.h).
__device__ __forceinline__ bool keep_quartet_fock(const ScreenArgs &scr, const PairSet &bra, const PairSet &ket,
                                                  int bi, int ki, int sa, int sb, int sc, int sd)
{
    if (scr.tau > 0.0) {
        const int ns = scr.nshell;
        const double *M = scr.M;
        double Mq = M[(size_t)sa * ns + sb];
        Mq = fmax(Mq, M[(size_t)sc * ns + sd]);
        Mq = fmax(Mq, M[(size_t)sa * ns + sc]);
        Mq = fmax(Mq, M[(size_t)sa * ns + sd]);
        Mq = fmax(Mq, M[(size_t)sb * ns + sc]);
        Mq = fmax(Mq, M[(size_t)sb * ns + sd]);
        if (scr.scale * bra.Q[bi] * ket.Q[ki] * Mq < scr.tau) return false;
    }
    return true;
}

// Integrals of one canonical quartet (both operators) into I[2][NAB][NCD],
// summed over bra primitive pairs ib0, ib0 + ibs, ...
template <int LA, int LB, int LC, int LD>
__device__ void quartet_fock_ints(double *sm, int lane, const GeoArgs &geo, const PrimPairs &pp, int nops,
                                  double omega, int sa, int sb, int sc, int sd, int pb0, int nbp, int ib0, int ibs,
                                  int pk0, int nkp, const double *boys)
{
    using Lay = FockLay<LA, LB, LC, LD>;
    constexpr int NAB = Lay::NAB, NCD = Lay::NCD, L = Lay::L, NM1 = Lay::NM1, NM2P = Lay::NM2P;
    constexpr int NS1 = Lay::NS1, NS2 = Lay::NS2, RS = Lay::RS, NO = Lay::NO, NP1 = Lay::NP1;
    double *I = sm + Lay::o_I, *V = sm + Lay::o_V, *S1 = sm + Lay::o_S1, *P1 = sm + Lay::o_P1, *pw = sm + Lay::o_pw;
    double *Rr = sm + Lay::o_X, *S2 = Rr + Lay::NRH * RS;
    double *vb = sm + Lay::o_X, *vk = vb + Lay::NE1, *half = vk + Lay::NE2;
    const auto &TBra = pair_tab<LA, LB>();
    const auto &TKet = pair_tab<LC, LD>();
    const bool ominf = isinf(omega);
    const double om = ominf ? 1.0 : omega;
    const double *xa = geo.xyz + 3 * geo.sh_atom[sa], *xb = geo.xyz + 3 * geo.sh_atom[sb];
    const double *xc = geo.xyz + 3 * geo.sh_atom[sc], *xd = geo.xyz + 3 * geo.sh_atom[sd];
    if (lane < 6) {
        const int d = lane % 3;
        const double x = lane < 3 ? xa[d] - xb[d] : xc[d] - xd[d];
        double p = 1.0;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            pw[(lane / 3) * 15 + d * 5 + k] = p;
            p *= x;
        }
    }
    const int nbra = (nbp - ib0 + ibs - 1) / ibs, pb = block_pairs(nbra, nkp, Lay::PB);
    if (nops == 1)
        for (int it = lane; it < NAB * NCD; it += 32) I[NAB * NCD + it] = 0.0;
    for (int o0 = 0; o0 < nops; o0 += NO) {
        for (int it = lane; it < NO * NM1 * NM2P; it += 32) V[it] = 0.0;
        __syncwarp();
        for (int blk = 0; blk < nbra; blk += pb) {
            const int np = min(pb, nbra - blk);
            if (lane < np) {
                const int ip = pb0 + ib0 + (blk + lane) * ibs;
                double s[NS1];
                pair_scalars<LA, LB, false>(pp.oo2[ip], pp.fa[ip], pp.fb[ip], s);
#pragma unroll
                for (int k = 0; k < NS1; ++k) S1[lane * NS1 + k] = s[k];
                P1[lane * NP1] = pp.p[ip];
                P1[lane * NP1 + 1] = pp.kop[ip] * 34.986836655249725;
            }
            __syncwarp();
            const int ntot = np * nkp;
            for (int j0 = 0; j0 < ntot; j0 += 32) {
                const int idx = min(j0 + lane, ntot - 1);
                const int pi = idx / nkp;
                const int ip = pb0 + ib0 + (blk + pi) * ibs, kp = pk0 + (idx - pi * nkp);
                const double p = P1[pi * NP1], q = pp.p[kp];
                const double ir = rsqrt(p + q), rho = p * q * ir * ir;
                const double X = pp.Px[ip] - pp.Px[kp], Y = pp.Py[ip] - pp.Py[kp], Z = pp.Pz[ip] - pp.Pz[kp];
                const double T0 = rho * (X * X + Y * Y + Z * Z);
                const double pref = j0 + lane < ntot ? P1[pi * NP1 + 1] * pp.kop[kp] * ir : 0.0;
                {
                    double s2[NS2];
                    pair_scalars<LC, LD, true>(pp.oo2[kp], pp.fa[kp], pp.fb[kp], s2);
#pragma unroll
                    for (int k = 0; k < NS2; ++k) S2[k * RS + lane] = s2[k];
                }
#pragma unroll 1
                for (int o = 0; o < NO; ++o) {
                    if (o0 + o >= nops) break;
                    double base[L + 1];
                    {
                        double th = 1.0;
                        if (o0 + o == 1 && !ominf) th = om * rsqrt(om * om + rho);
                        double Fm[L + 1];
                        const double th2 = th * th;
                        boys_lane<L>(T0 * th2, Fm, boys);
                        double f = pref * th;
                        const double m2r = -2.0 * rho * th2;
#pragma unroll
                        for (int n = 0; n <= L; ++n) {
                            base[n] = f * Fm[n];
                            f *= m2r;
                        }
                    }
                    double *Rl = Rr + lane;
                    if constexpr (L <= 5) {
                        double R[nherm(L)];
                        hermite_R<L>(R, base, X, Y, Z);
#pragma unroll
                        for (int h = 0; h < nherm(L); ++h) Rl[h * RS] = R[h];
                    } else {
                        Rl[0] = base[L];
                        static_for<L>([&](auto N) {
                            constexpr int n = L - 1 - decltype(N)::value;
                            hermite_level<RS>(Rl, nherm(L - n), X, Y, Z);
                            Rl[0] = base[n];
                        });
                    }
                    __syncwarp();
                    reverse_sums<LA, LB, LC, LD, true>(V + o * NM1 * NM2P, Rr, S2, S1, j0, min(32, ntot - j0), nkp, lane);
                    __syncwarp();
                }
            }
        }
        // ---- V -> I: ket functions, then bra functions
        entry_values<LA, LB>(vb, lane, pw, 1);
        entry_values<LC, LD>(vk, lane, pw + 15, 1);
        __syncwarp();
        for (int it = lane; it < NM1 * NCD; it += 32) {
            const int m1 = it / NCD, cd = it % NCD;
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                double s = 0.0;
                for (int k = TKet.fstart[cd]; k < TKet.fstart[cd + 1]; ++k) {
                    const int e = TKet.fent[k];
                    s += vk[e] * V[(o * NM1 + m1) * NM2P + TKet.own[e]];
                }
                half[(o * NM1 + m1) * NCD + cd] = s;
            }
        }
        __syncwarp();
        for (int it = lane; it < NAB * NCD; it += 32) {
            const int ab = it / NCD, cd = it % NCD;
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                if (o0 + o >= nops) break;
                double s = 0.0;
                for (int k = TBra.fstart[ab]; k < TBra.fstart[ab + 1]; ++k) {
                    const int e = TBra.fent[k];
                    s += vb[e] * half[(o * NM1 + TBra.own[e]) * NCD + cd];
                }
                I[(o0 + o) * NAB * NCD + it] = s;
            }
        }
        __syncwarp();
    }
}

// Contractions of I with the density images and the atomic adds to F.
template <int LA, int LB, int LC, int LD>
__device__ void quartet_fock_scatter(const double *I, int lane, int nops, const double *SJ, const double *BK,
                                     const double *BL, int nbf, int fa, int fb, int fc, int fd, double scale,
                                     double *F)
{
    using Lay = FockLay<LA, LB, LC, LD>;
    constexpr int NA = Lay::NA, NB = Lay::NB, NC = Lay::NC, ND = Lay::ND, NCD = Lay::NCD, NAB = Lay::NAB;
    const double *I1 = I + NAB * NCD;
    auto ix = [&](int ia, int ib, int ic, int id) { return (ia * NB + ib) * NCD + ic * ND + id; };
    // Coulomb: F[m][n], F[n][m] += sum_{ls} I0 S_J[l][s]
    for (int it = lane; it < NAB; it += 32) {
        const int ia = it / NB, ib = it % NB;
        double acc = 0.0;
        for (int ic = 0; ic < NC; ++ic)
            for (int id = 0; id < ND; ++id) acc += I[ix(ia, ib, ic, id)] * SJ[(size_t)(fc + ic) * nbf + fd + id];
        acc *= scale;
        atomicAdd(F + (size_t)(fa + ia) * nbf + fb + ib, acc);
        atomicAdd(F + (size_t)(fb + ib) * nbf + fa + ia, acc);
    }
    // Coulomb: F[l][s], F[s][l] += sum_{mn} I0 S_J[m][n]
    for (int it = lane; it < NCD; it += 32) {
        const int ic = it / ND, id = it % ND;
        double acc = 0.0;
        for (int ia = 0; ia < NA; ++ia)
            for (int ib = 0; ib < NB; ++ib) acc += I[ix(ia, ib, ic, id)] * SJ[(size_t)(fa + ia) * nbf + fb + ib];
        acc *= scale;
        atomicAdd(F + (size_t)(fc + ic) * nbf + fd + id, acc);
        atomicAdd(F + (size_t)(fd + id) * nbf + fc + ic, acc);
    }
    // exchange: eight images, target (row index, column index) and summed
    // indices; shell offsets by position 0..3 = a, b, c, d
    const int off[4] = {fa, fb, fc, fd};
    const int nn[4] = {NA, NB, NC, ND};
    // image k: target F[x][y] += sum I(m n|l s) B[u][v]; positions (x, y, u, v)
    const int img[8][4] = {{0, 2, 1, 3}, {1, 2, 0, 3}, {0, 3, 1, 2}, {1, 3, 0, 2},
                           {2, 0, 3, 1}, {3, 0, 2, 1}, {2, 1, 3, 0}, {3, 1, 2, 0}};
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        const int X = img[k][0], Y = img[k][1], U = img[k][2], V = img[k][3];
        const int nx = nn[X], ny = nn[Y], nu = nn[U], nv = nn[V];
        for (int it = lane; it < nx * ny; it += 32) {
            int pos[4];
            pos[X] = it / ny;
            pos[Y] = it % ny;
            double acc = 0.0;
            for (int u = 0; u < nu; ++u)
                for (int v = 0; v < nv; ++v) {
                    pos[U] = u;
                    pos[V] = v;
                    const int e = ix(pos[0], pos[1], pos[2], pos[3]);
                    const size_t bi = (size_t)(off[U] + u) * nbf + off[V] + v;
                    acc += I[e] * BK[bi];
                    if (nops == 2) acc += I1[e] * BL[bi];
                }
            atomicAdd(F + (size_t)(off[X] + pos[X]) * nbf + off[Y] + pos[Y], acc * scale);
        }
    }
}

// Persistent Fock class kernel over warp units (as k_grad_lanes).  The
// combined matrices are den.A[0] = S_J, den.B[0] = B_K, den.A[1] = B_lr.
template <int LA, int LB, int LC, int LD>
__global__ void __launch_bounds__(32, LA + LB + LC + LD <= 3 ? 16 : 8)
    k_fock_lanes(const MolDesc *__restrict__ mols, ClassLaunch cl, OutArgs out, const double *__restrict__ boys)
{
    using Lay = FockLay<LA, LB, LC, LD>;
    extern __shared__ double smem[];
    const int nw = blockDim.x / 32, grp = threadIdx.x / 32, lane = threadIdx.x % 32;
    double *wsm = smem + (size_t)grp * Lay::TOTAL;
    unsigned long long nq = 0, npq = 0, nbv = 0;
    const int S = cl.nsplit, C = cl.nchunk, QPC = TILE / C;
    const bool same = cl.P == cl.Q;
    const long long units = cl.ntiles * C * S, W = (long long)gridDim.x * nw;
    const long long w0 = (long long)grp * gridDim.x + blockIdx.x;
    for (long long r = 0; r * W < units; ++r) {
        const long long it = r * W + ((r & 1) ? W - 1 - w0 : w0);
        if (it >= units) continue;
        const long long tile = it / (C * S);
        const int chunk = (int)((it / S) % C), split = (int)(it % S);
        const uint4 tl = cl.tiles[tile];
        const MolDesc &md = mols[tl.x];
        const PairSet &bra = md.sets[cl.P], &ket = md.sets[cl.Q];
        for (int qi = chunk * QPC; qi < (chunk + 1) * QPC; ++qi) {
            const int bi = tl.y * TB + qi / TK;
            const int ki = tl.z * TK + qi % TK;
            bool ok = bi < bra.n && ki < ket.n && (!same || bi >= ki);
            if (ok) ok = split < bra.np[bi];
            int sa = 0, sb = 0, sc = 0, sd = 0;
            if (ok) {
                sa = bra.sa[bi];
                sb = bra.sb[bi];
                sc = ket.sa[ki];
                sd = ket.sb[ki];
                ok = keep_quartet_fock(md.scr, bra, ket, bi, ki, sa, sb, sc, sd);
            }
            if (!ok) continue;  // uniform across the warp
            double scale = 1.0;
            if (sa == sb) scale *= 0.5;
            if (sc == sd) scale *= 0.5;
            if (same && bi == ki) scale *= 0.5;
            const int nbp = bra.np[bi], nkp = ket.np[ki];
            if (nkp > 0) {
                const int nops = md.den.use_lr ? 2 : 1;
                quartet_fock_ints<LA, LB, LC, LD>(wsm, lane, md.geo, md.pp, nops, md.den.omega, sa, sb, sc, sd,
                                                  bra.poff[bi], nbp, split, S, ket.poff[ki], nkp, boys);
                const int *bf = md.geo.sh_bf;
                quartet_fock_scatter<LA, LB, LC, LD>(wsm + Lay::o_I, lane, nops, md.den.A[0], md.den.B[0], md.den.A[1],
                                                     md.den.nbf, bf[sa], bf[sb], bf[sc], bf[sd], scale, out.fock);
                __syncwarp();
            }
            if (lane == 0) {
                if (split == 0) nq += 1;
                npq += (unsigned long long)((nbp - split + S - 1) / S) * nkp;
                nbv += (unsigned long long)((nbp - split + S - 1) / S);
            }
        }
    }
    if (lane == 0 && (nq || npq)) {
        atomicAdd(out.counters + 0, nq);
        atomicAdd(out.counters + 1, npq);
        atomicAdd(out.counters + 4, nbv);
    }
}

// CTAs of one warp (see HermOp); F takes atomic adds, so no slab limits the grid.
template <int LA, int LB, int LC, int LD>
cudaError_t launch_fock_class(int, cudaStream_t st, const MolDesc *mols, const ClassLaunch &cl, const OutArgs &out,
                              const double *boys)
{
    constexpr size_t bytes = FockLay<LA, LB, LC, LD>::BYTES;
    static_assert(bytes <= kCtaSmem, "one warp's arrays fit in a CTA");
    return launch_warp_units(k_fock_lanes<LA, LB, LC, LD>, 1, 32, bytes, 1, 1 << 20, st, mols, cl, out, boys);
}

}  // namespace tg
