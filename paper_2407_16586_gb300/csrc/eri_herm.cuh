// fp64 derivative-ERI class kernel: one warp per contracted shell quartet,
// one primitive quartet per lane, the density folded into Hermite densities.
//
// Derivation.  With R = A - B, a^ = zeta_a / p, b^ = zeta_b / p, the expansion
// coefficients of a function pair (eq. cartG) are polynomials in
// P - A = -b^ R and P - B = a^ R:
//   E^{ab}_h(p) = sum_{k,l} c^{ab}_{h,k,l} R^{la+lb-k-l} (-b^)^{la-k} a^^{lb-l} (1/2p)^{(k+l+|h|)/2}
// (integer c; k, l: how much of a and b is expanded about P).  Everything that
// depends on the function pair is in c R^(..), which all primitive pairs
// share; a primitive pair enters through the few scalars
// s_m = (-b^)^(la-k) a^^(lb-l) (1/2p)^((k+l+|h|)/2) only.  So the density of a
// contracted quartet is transformed ONCE to the "monomials" m = (h, k, l),
//   G'[m1][m2] = sum_{ab,cd} Gamma[ab][cd] c^{ab}_{m1} R^.. c^{cd}_{m2} S^..       (S = C - D)
// ((pp|pp): 81 -> 14 x 14, (dd|dd): 1296 -> 76 x 76), and per operator
//   F[h1][m2]   = sum_{m1 of h1} s_m1(p) G'[m1][m2]                 per bra primitive pair
//   X[h]        = sum_{h1+h2=h} (-1)^|h2| s_m2(q) F[h1][m2]         per primitive quartet (lane)
//   E, T_i      = sum_h X[h] R[h], sum_h X[h] R[h + 1_i]            per primitive quartet (lane)
//   U[h1][m2]   = sum_q (-1)^|h2| s_m2(q) R[h1 + h2]                items over lanes, lanes' R from shared memory
//   V[m1][m2]  += s_m1(p) U[h1][m2]                                 per bra primitive pair
// With P = A - b^ R, exp(-mu R^2), and the polynomials in R, eq. deriv becomes
//   d/dA = sum a^ T - 2 mu_ab R E + sum V dG'/dR
//   d/dC = sum -c^ T - 2 mu_cd S E + sum V dG'/dS,   d/dA + d/dB = sum T,
// and d/dB, d/dD follow from translational invariance (eq. ti).  Against
// contracting E tables for every primitive quartet this needs 3 ((pp|pp)) to
// 8 times ((dd|dd)) fewer fp64 operations.
//
// What bounds it: the fp64 pipe.  GB300 retires 2 DFMA per clock and SM, so a
// warp instruction holds it for 16 clocks whether one lane or all 32 are
// active, and everything else (shared-memory traffic, index arithmetic, even
// one warp per scheduler) hides behind it.  Hence full lanes come first:
// primitive quartets of a block of PB bra primitive pairs are flattened over
// the 32 lanes, PB chosen per quartet to waste the fewest; the reverse sums U
// are spread over (h1, m2) items, several lanes per item when there are few.
#pragma once
#include <utility>

#include "eri_warp.cuh"

namespace tg {

// ------------------------------------------------------------ pair tables

// Scalars of order n = |h|: (k, l) with k <= LA, l <= LB, k + l >= n of n's
// parity, k ascending, then l.  nsig: how many; soff / moff: first scalar and
// first monomial of an order.
template <int LA, int LB>
struct PairMono {
    static constexpr int L = LA + LB, NA = ncart(LA), NB = ncart(LB), NAB = NA * NB, NH = nherm(L);
    __host__ __device__ static constexpr int nsig(int n)
    {
        int c = 0;
        for (int k = 0; k <= LA; ++k)
            for (int l = 0; l <= LB; ++l) c += (k + l >= n && ((k + l - n) & 1) == 0) ? 1 : 0;
        return c;
    }
    __host__ __device__ static constexpr int soff(int n)
    {
        int c = 0;
        for (int i = 0; i < n; ++i) c += nsig(i);
        return c;
    }
    __host__ __device__ static constexpr int moff(int n)
    {
        int c = 0;
        for (int i = 0; i < n; ++i) c += nsig(i) * (i + 1) * (i + 2) / 2;
        return c;
    }
    static constexpr int NS = soff(L + 1), NM = moff(L + 1);
    static constexpr int choose2(int n, int k) { return (k == 0 || k == n) ? 1 : 2; }  // n <= 2
    // (x - P)^n in Hermite functions: coefficient of Lambda_t over (1/2p)^((n+t)/2)
    static constexpr int herm_coef(int n, int t)
    {
        int v = 1;
        for (int i = t + 1; i <= n; ++i) v *= i;       // n! / t!
        for (int i = 1; i <= (n - t) / 2; ++i) v /= 2 * i;
        return v;
    }
    static constexpr int monomial(int h, int n, int k, int l)
    {
        int s = 0;
        for (int kk = 0; kk <= LA; ++kk)
            for (int ll = 0; ll <= LB; ++ll) {
                if (kk == k && ll == l) return moff(n) + (h - nherm(n - 1)) * nsig(n) + s;
                s += (kk + ll >= n && ((kk + ll - n) & 1) == 0) ? 1 : 0;
            }
        return -1;
    }
};

// One term c^{ab}_m R_x^px R_y^py R_z^pz: ab | coef << 8 | px << 16 | py << 19 | pz << 22.
constexpr int pair_entries(int la, int lb)
{
    // (ss) 1, (ps) 6, (pp) 39, (ds) 24, (dp) 159, (dd) 648; make_pair_tab counts them again
    return la == 0 ? 1 : (la == 1 ? (lb == 0 ? 6 : 39) : (lb == 0 ? 24 : (lb == 1 ? 159 : 648)));
}

template <int LA, int LB>
struct PairTab {
    using M = PairMono<LA, LB>;
    static constexpr int NE = pair_entries(LA, LB);
    int n;                             // entries found
    unsigned ent[NE];                  // by monomial
    unsigned short own[NE];            // monomial of each entry
    unsigned short start[M::NM + 1];   // entries of monomial m: start[m] .. start[m + 1]
    unsigned short fstart[M::NAB + 1]; // entries of function pair ab: fent[fstart[ab]] .. fent[fstart[ab + 1] - 1]
    unsigned short fent[NE];
    unsigned short hm[M::NH];          // per Hermite index: first monomial | nsig << 8 | first scalar << 12
};

template <int LA, int LB>
constexpr PairTab<LA, LB> make_pair_tab()
{
    using M = PairMono<LA, LB>;
    PairTab<LA, LB> T{};
    int ne = 0;
    for (int n = 0; n <= M::L; ++n)
        for (int t = n; t >= 0; --t)
            for (int u = n - t; u >= 0; --u) {
                const int v = n - t - u, h = hidx(t, u, v);
                T.hm[h] = (unsigned short)((M::moff(n) + (h - nherm(n - 1)) * M::nsig(n)) | (M::nsig(n) << 8) |
                                           (M::soff(n) << 12));
                for (int k = 0; k <= LA; ++k)
                    for (int l = 0; l <= LB; ++l) {
                        if (!(k + l >= n && ((k + l - n) & 1) == 0)) continue;
                        const int m = M::monomial(h, n, k, l);
                        T.start[m] = (unsigned short)ne;
                        for (int ia = 0; ia < M::NA; ++ia)
                            for (int ib = 0; ib < M::NB; ++ib) {
                                const int as = ia == 0 ? 0 : (ia < 3 ? 1 : 2), bs = ib == 0 ? 0 : (ib < 3 ? 1 : 2);
                                const int az = ia - as * (as + 1) / 2, ay = as - az, ax = LA - as;
                                const int bz = ib - bs * (bs + 1) / 2, by = bs - bz, bx = LB - bs;
                                for (int kx = 0; kx <= ax; ++kx)
                                    for (int ky = 0; ky <= ay; ++ky)
                                        for (int lx = 0; lx <= bx; ++lx)
                                            for (int ly = 0; ly <= by; ++ly) {
                                                const int kz = k - kx - ky, lz = l - lx - ly;
                                                if (kz < 0 || kz > az || lz < 0 || lz > bz) continue;
                                                const int nx = kx + lx, ny = ky + ly, nz = kz + lz;
                                                if (nx < t || ny < u || nz < v || ((nx - t) & 1) || ((ny - u) & 1) ||
                                                    ((nz - v) & 1))
                                                    continue;
                                                const int c = M::choose2(ax, kx) * M::choose2(ay, ky) * M::choose2(az, kz) *
                                                              M::choose2(bx, lx) * M::choose2(by, ly) * M::choose2(bz, lz) *
                                                              M::herm_coef(nx, t) * M::herm_coef(ny, u) * M::herm_coef(nz, v);
                                                const int px = ax + bx - nx, py = ay + by - ny, pz = az + bz - nz;
                                                const unsigned w = (unsigned)(ia * M::NB + ib) | ((unsigned)px << 16) |
                                                                   ((unsigned)py << 19) | ((unsigned)pz << 22);
                                                int at = -1;  // terms of the same power add up
                                                for (int e = T.start[m]; e < ne; ++e)
                                                    if ((T.ent[e] & 0xffff00ffu) == w) at = e;
                                                if (at >= 0) {
                                                    T.ent[at] += (unsigned)c << 8;
                                                } else {
                                                    if (ne < PairTab<LA, LB>::NE) {
                                                        T.ent[ne] = w | ((unsigned)c << 8);
                                                        T.own[ne] = (unsigned short)m;
                                                    }
                                                    ++ne;
                                                }
                                            }
                            }
                    }
            }
    T.start[M::NM] = (unsigned short)ne;
    T.n = ne;
    int nf = 0;
    for (int ab = 0; ab < M::NAB; ++ab) {
        T.fstart[ab] = (unsigned short)nf;
        for (int e = 0; e < ne && e < PairTab<LA, LB>::NE; ++e)
            if ((int)(T.ent[e] & 0xff) == ab) T.fent[nf++] = (unsigned short)e;
    }
    T.fstart[M::NAB] = (unsigned short)nf;
    return T;
}

static __device__ const PairTab<0, 0> kPair00 = make_pair_tab<0, 0>();
static __device__ const PairTab<1, 0> kPair10 = make_pair_tab<1, 0>();
static __device__ const PairTab<1, 1> kPair11 = make_pair_tab<1, 1>();
static __device__ const PairTab<2, 0> kPair20 = make_pair_tab<2, 0>();
static __device__ const PairTab<2, 1> kPair21 = make_pair_tab<2, 1>();
static __device__ const PairTab<2, 2> kPair22 = make_pair_tab<2, 2>();

template <int LA, int LB>
__device__ __forceinline__ const PairTab<LA, LB> &pair_tab()
{
    if constexpr (LA == 0) return kPair00;
    else if constexpr (LA == 1 && LB == 0) return kPair10;
    else if constexpr (LA == 1) return kPair11;
    else if constexpr (LB == 0) return kPair20;
    else if constexpr (LB == 1) return kPair21;
    else return kPair22;
}

// ------------------------------------------------------------ layout

// One warp's slice of shared memory, in doubles, for KQ ket pairs at a time.
// Rows that lanes read at different row numbers have an odd stride.  NO
// operators are resident at a time; classes whose arrays are large take the
// operators one after the other (the scalars of a primitive quartet are then
// formed twice, 3 % of the work at (pp|pp)), which keeps at least four warps on
// an SM.
template <int LA, int LB, int LC, int LD, int KQ_>
struct HermLayK {
    using B = PairMono<LA, LB>;
    using K = PairMono<LC, LD>;
    static constexpr int KQ = KQ_;
    static constexpr int NAB = B::NAB, NCD = K::NAB, L1 = B::L, L2 = K::L, L = L1 + L2, LM = L + 1;
    static constexpr int NT1 = B::NH, NM1 = B::NM, NM2 = K::NM, NS1 = B::NS, NS2 = K::NS;
    static constexpr int NABP = NAB | 1, NM2P = NM2 | 1;
    static constexpr int RS = 33;                     // row stride of the per-lane columns
    // The R tensor: in registers up to LM = 5, else in shared-memory rows; X in
    // registers, from L = 5 in passes over ranges of Hermite orders (one a warp),
    // which need R's top order stored too.
    static constexpr bool RREG = LM <= 5, PASSES = !RREG;
    // Warps per quartet: one warp's arrays take 104 ((dd|dp)) or 188 KB ((dd|dd)),
    // so four warps work on one quartet there: transforms, recursion entries and
    // reverse items dealt over them, one range of orders of X each (on a 1/8 shard of
    // the 32-atom workload 22.2 -> 11.3 and 13.9 -> 4.2 ms).  Two at L = 5, 6 (40 to 60
    // KB): 6 to 8 warps an SM instead of 4 or 5 and half the tails (all classes of
    // that shard together 205.9 -> 198.4 ms, 6 atoms 16.0 -> 15.3 ms).
    static constexpr int NW = L >= 7 ? 4 : (PASSES ? 2 : 1);
    // Hermite rows: the reverse sums reach order L - 1 (their items leave out the
    // top order of both sides at once), the recursion in rows needs all
    static constexpr int NRH = nherm(PASSES ? LM : L - 1);
    static constexpr int NO = (NAB * NCD <= 27) ? 2 : 1;
    // bra primitive pairs of a block: a budget of 1200 doubles for F, 1 to 16
    // (700 buys (dp|pp) a sixth warp, but its half-filled passes cost more:
    // 23.4 -> 29.3 ms on a 1/8 shard of the 32-atom workload)
    static constexpr int PB_RAW = 1200 / (NT1 * NM2P * NO * KQ);
    static constexpr int PB = PB_RAW < 1 ? 1 : (PB_RAW > 16 ? 16 : PB_RAW);
    static constexpr int NE1 = pair_entries(LA, LB), NE2 = pair_entries(LC, LD);
    static constexpr int GS = NO * NCD * NABP, MS = NO * NM1 * NM2P, FS = NO * NT1 * NM2P;  // per ket pair
    static constexpr int HS = (NM2 * NABP > NM1 * NCD ? NM2 * NABP : NM1 * NCD) * NO;
    // the transforms' half-way arrays share the space of the R rows
    static constexpr int HALF = NE1 + KQ * (NE2 + HS), ROWS = (NRH + NS2) * RS, RED = 9 * RS * NW;
    static constexpr int SHARED = HALF > ROWS ? (HALF > RED ? HALF : RED) : (ROWS > RED ? ROWS : RED);
    static constexpr int NP1 = 4;                     // per bra primitive pair: a^, mu, 2 pi^(5/2) K / p, p
    static constexpr int o_G = 0;                              // [KQ][NO][NCD][NABP]
    static constexpr int o_Gp = o_G + KQ * GS;                 // [KQ][NO][NM1][NM2P]
    static constexpr int o_V = o_Gp + KQ * MS;                 // [KQ][NO][NM1][NM2P]
    static constexpr int o_F = o_V + KQ * MS;                  // [PB][KQ][NO][NT1][NM2P]
    static constexpr int o_S1 = o_F + PB * KQ * FS;            // [PB][NS1]
    static constexpr int o_P1 = o_S1 + PB * NS1;               // [PB][NP1]
    static constexpr int o_pw = o_P1 + PB * NP1;               // [1 + KQ][3][5] powers of R, then of each S
    static constexpr int o_X = o_pw + (1 + KQ) * 15;           // SHARED
    static constexpr int TOTAL = (o_X + SHARED + 1) & ~1;
    static constexpr size_t BYTES = sizeof(double) * (size_t)TOTAL;
};

// Ket pairs of one bra pair that may be taken together: the most (8, 4, 2, 1)
// with which 16 warps still fit an SM's shared memory, up to L = 2 ((ps|ss):
// 16.7 -> 11.5 ms on a 1/8 shard of the 32-atom workload).  Above, a group costs
// warps and gains nothing ((pp|ps): 23.9 -> 27.6 ms, (dp|pp): 23.4 -> 30.4 ms).
template <int LA, int LB, int LC, int LD>
constexpr int herm_kets()
{
    constexpr size_t cap = (223 * 1024) / 16;
    if (LA + LB + LC + LD > 2) return 1;
    if (HermLayK<LA, LB, LC, LD, 8>::BYTES <= cap) return 8;
    if (HermLayK<LA, LB, LC, LD, 4>::BYTES <= cap) return 4;
    if (HermLayK<LA, LB, LC, LD, 2>::BYTES <= cap) return 2;
    return 1;
}

template <int LA, int LB, int LC, int LD>
using HermLay = HermLayK<LA, LB, LC, LD, herm_kets<LA, LB, LC, LD>()>;

// The valid ket pairs of one bra pair among up to KQ neighbours, in shared
// memory; entries past them have nk = 0 and a valid pk0.  A group is the
// entries k0 .. k0 + kg - 1.
struct GroupInfo {
    static constexpr int CAP = 8;
    int n;                       // valid ket pairs of the whole record
    int sc[8], sd[8];            // shells
    int pk0[8], nk[8];           // primitive pairs
    double scale[8];             // 1/|stabiliser|
};

// (h1, m2) items of the reverse sums: ALL, or those whose V enters a
// derivative, i.e. some monomial of h1 carries a power of R or m2 one of S.
// R row | h1 << 8 | m2 << 14 | scalar of m2 << 21
template <int LA, int LB, int LC, int LD, bool ALL>
constexpr int herm_item_count()
{
    using B = PairMono<LA, LB>;
    using K = PairMono<LC, LD>;
    int n = 0;
    for (int n2 = 0; n2 <= K::L; ++n2)
        for (int k = 0; k <= LC; ++k)
            for (int l = 0; l <= LD; ++l)
                if (k + l >= n2 && ((k + l - n2) & 1) == 0)
                    n += (n2 + 1) * (n2 + 2) / 2 * (ALL || k + l < K::L ? nherm(B::L) : nherm(B::L - 1));
    return n;
}

template <int LA, int LB, int LC, int LD, bool ALL>
struct HermItems {
    static constexpr int N = herm_item_count<LA, LB, LC, LD, ALL>();
    unsigned it[N > 0 ? N : 1];
};

template <int LA, int LB, int LC, int LD, bool ALL>
constexpr HermItems<LA, LB, LC, LD, ALL> make_herm_items()
{
    using B = PairMono<LA, LB>;
    using K = PairMono<LC, LD>;
    HermItems<LA, LB, LC, LD, ALL> T{};
    int n = 0;
    for (int n1 = 0; n1 <= B::L; ++n1)
        for (int t1 = n1; t1 >= 0; --t1)
            for (int u1 = n1 - t1; u1 >= 0; --u1)
                for (int n2 = 0; n2 <= K::L; ++n2)
                    for (int t2 = n2; t2 >= 0; --t2)
                        for (int u2 = n2 - t2; u2 >= 0; --u2) {
                            const int v1 = n1 - t1 - u1, v2 = n2 - t2 - u2;
                            int s = 0;
                            for (int k = 0; k <= LC; ++k)
                                for (int l = 0; l <= LD; ++l) {
                                    if (!(k + l >= n2 && ((k + l - n2) & 1) == 0)) continue;
                                    if (ALL || k + l < K::L || n1 < B::L)
                                        T.it[n++] = (unsigned)hidx(t1 + t2, u1 + u2, v1 + v2) |
                                                    ((unsigned)hidx(t1, u1, v1) << 8) |
                                                    ((unsigned)K::monomial(hidx(t2, u2, v2), n2, k, l) << 14) |
                                                    ((unsigned)(K::soff(n2) + s) << 21);
                                    ++s;
                                }
                        }
    return T;
}

// ------------------------------------------------------------ lane pieces

// F_m(T), m = 0..M, one argument per lane.  T < 64: F_M and F_{M+1} by the
// Taylor step of the table (shared d/k factors), e^-T = (2M+1) F_M - 2T F_{M+1}
// (error below eps (2M+1) F_M, which the next order up divides by 2M-1), then
// downward recursion: no exponential.  T >= 64: upward recursion without e^-T,
// which is under 1e-14 of the smallest order's term there.
template <int M>
__device__ __forceinline__ void boys_lane(double T, double (&F)[M + 1], const double *__restrict__ tab)
{
    if (T < BOYS_TFAR) {
        const int i = __double2int_rn(T * (1.0 / BOYS_H));
        const double d = i * BOYS_H - T;
        const double *row = tab + i * (BOYS_M + 1) + M;
        double hi = row[BOYS_TAYLOR + 1], lo = row[BOYS_TAYLOR];
#pragma unroll
        for (int k = BOYS_TAYLOR - 1; k >= 0; --k) {
            const double dk = d * (1.0 / (k + 1));
            hi = row[k + 1] + hi * dk;
            lo = row[k] + lo * dk;
        }
        const double t2 = 2.0 * T;
        const double et = (2 * M + 1) * lo - t2 * hi;
        F[M] = lo;
#pragma unroll
        for (int m = M - 1; m >= 0; --m) F[m] = (t2 * F[m + 1] + et) * (1.0 / (2 * m + 1));
    } else {
        // 1/2T from the square of 1/sqrt(T), corrected to the last bit: its rounding
        // enters order m m times (F_9: 1.0e-15 rms without, 0.5e-15 with, as by
        // division).  2T by its exponent, capped so that T = inf gives h = 0, not NaN.
        const double is = rsqrt(T), h0 = 0.5 * is * is;
        const double t2 = __hiloint2double(min(__double2hiint(T), 0x7e000000) + 0x100000, __double2loint(T));
        const double h = fma(h0, fma(-t2, h0, 1.0), h0);
        F[0] = 0.88622692545275801365 * is;
#pragma unroll
        for (int m = 0; m < M; ++m) F[m + 1] = (2 * m + 1) * h * F[m];
    }
}

// s_m of one primitive pair: oo2 = 1/2p, a = zeta_a/p, b = zeta_b/p; the ket
// carries the sign (-1)^|h|.
template <int LA, int LB, bool KET>
__device__ __forceinline__ void pair_scalars(double oo2, double a, double b, double (&s)[PairMono<LA, LB>::NS])
{
    double bp[LA + 1], ap[LB + 1], op[LA + LB + 1];
    bp[0] = ap[0] = op[0] = 1.0;
#pragma unroll
    for (int i = 1; i <= LA; ++i) bp[i] = -b * bp[i - 1];
#pragma unroll
    for (int i = 1; i <= LB; ++i) ap[i] = a * ap[i - 1];
#pragma unroll
    for (int i = 1; i <= LA + LB; ++i) op[i] = oo2 * op[i - 1];
    int c = 0;
#pragma unroll
    for (int n = 0; n <= LA + LB; ++n)
#pragma unroll
        for (int k = 0; k <= LA; ++k)
#pragma unroll
            for (int l = 0; l <= LB; ++l)
                if (k + l >= n && ((k + l - n) & 1) == 0) {
                    const double v = bp[LA - k] * ap[LB - l] * op[(k + l + n) / 2];
                    s[c++] = (KET && (n & 1)) ? -v : v;
                }
}

// f(integral_constant<int, 0>), ..., f(integral_constant<int, N - 1>)
template <typename Fn, int... I>
__device__ __forceinline__ void static_for_impl(Fn &&f, std::integer_sequence<int, I...>)
{
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, typename Fn>
__device__ __forceinline__ void static_for(Fn &&f)
{
    static_for_impl(f, std::make_integer_sequence<int, N>{});
}

// Shared-memory load of the unrolled lane phases.  Inline PTX: plain loads
// between this many stores make the compiler's alias analysis take minutes per
// class.  The compiler does not see that it reads memory, so a barrier of the
// warp or CTA stands between it and plain accesses to the same rows.
__device__ __forceinline__ double lds(const double *p)
{
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"((unsigned)__cvta_generic_to_shared(p)));
    return v;
}

// (t, u, v) of a compact Hermite index, at compile time
struct Triple {
    int t, u, v;
};
__host__ __device__ constexpr Triple herm_triple(int h)
{
    for (int n = 0;; ++n)
        if (h < nherm(n)) {
            int r = h - nherm(n - 1);
            for (int t = n;; --t) {
                if (r <= n - t) return Triple{t, n - t - r, r};
                r -= n - t + 1;
            }
        }
}

// One row of the Hermite density: for the bra index h1, X[h1 + h2] gets every
// ket monomial's s_m2 F[h1][m2].
template <int LC, int LD>
struct DensRow {
    using K = PairMono<LC, LD>;
    short h2[K::NM], s[K::NM];
};
template <int LC, int LD>
__host__ __device__ constexpr DensRow<LC, LD> make_dens_row()
{
    using K = PairMono<LC, LD>;
    DensRow<LC, LD> r{};
    for (int h = 0; h < K::NH; ++h) {
        const Triple x = herm_triple(h);
        const int n = x.t + x.u + x.v;
        for (int k = 0; k < K::nsig(n); ++k) {
            const int m = K::moff(n) + (h - nherm(n - 1)) * K::nsig(n) + k;
            r.h2[m] = (short)h;
            r.s[m] = (short)(K::soff(n) + k);
        }
    }
    return r;
}
__host__ __device__ constexpr int herm_sum(int h1, int h2)
{
    const Triple a = herm_triple(h1), b = herm_triple(h2);
    return hidx(a.t + b.t, a.u + b.u, a.v + b.v);
}

// X[h] of one lane for the Hermite orders HLO .. HHI: sum over h1 and the ket
// monomials of s_m2 F[h1][m2] (F: this lane's bra primitive pair).
template <int LA, int LB, int LC, int LD, int HLO, int HHI>
__device__ __forceinline__ void hermite_density(const double *F, const double (&s2)[PairMono<LC, LD>::NS],
                                                double (&X)[nherm(HHI) - nherm(HLO - 1)])
{
    using Lay = HermLay<LA, LB, LC, LD>;
    constexpr int H0 = nherm(HLO - 1), H1 = nherm(HHI);
#pragma unroll
    for (int h = 0; h < H1 - H0; ++h) X[h] = 0.0;
    static_for<Lay::NT1>([&](auto B) {
        static_for<Lay::NM2>([&](auto M2) {
            constexpr int h1 = decltype(B)::value, m2 = decltype(M2)::value;
            constexpr auto row = make_dens_row<LC, LD>();
            constexpr int x = herm_sum(h1, row.h2[m2]), sc = row.s[m2];
            if constexpr (x >= H0 && x < H1) X[x - H0] += s2[sc] * lds(F + h1 * Lay::NM2P + m2);
        });
    });
}

// One pass over a range of orders: E += X[h] R[h], T_i += X[h] R[h + 1_i], R
// from this lane's column.
template <int LA, int LB, int LC, int LD, int HLO, int HHI>
__device__ __forceinline__ void density_pass(const double *F, const double (&s2)[PairMono<LC, LD>::NS],
                                             const double *Rl, double &e, double (&T)[3])
{
    constexpr int RS = HermLay<LA, LB, LC, LD>::RS, H0 = nherm(HLO - 1);
    double X[nherm(HHI) - H0];
    hermite_density<LA, LB, LC, LD, HLO, HHI>(F, s2, X);
    static_for<nherm(HHI) - H0>([&](auto J) {
        constexpr int j = decltype(J)::value;
        constexpr Triple x = herm_triple(H0 + j);
        e += X[j] * lds(Rl + (H0 + j) * RS);
        T[0] += X[j] * lds(Rl + hidx(x.t + 1, x.u, x.v) * RS);
        T[1] += X[j] * lds(Rl + hidx(x.t, x.u + 1, x.v) * RS);
        T[2] += X[j] * lds(Rl + hidx(x.t, x.u, x.v + 1) * RS);
    });
}

// E += X[h] r and T_i += X[h - 1_i] r of Hermite entry h, where X holds the
// orders up to L.
template <int L, int H>
__device__ __forceinline__ void energy_terms(double r, const double (&X)[nherm(L)], double &e, double (&T)[3])
{
    constexpr Triple x = herm_triple(H);
    if constexpr (H < nherm(L)) e += X[H] * r;
    if constexpr (x.t > 0) T[0] += X[hidx(x.t - 1, x.u, x.v)] * r;
    if constexpr (x.u > 0) T[1] += X[hidx(x.t, x.u - 1, x.v)] * r;
    if constexpr (x.v > 0) T[2] += X[hidx(x.t, x.u, x.v - 1)] * r;
}

// How Hermite entry h follows from the level above (hermite_R): direction,
// first and second source, coefficient.  dir | src1 << 2 | src2 << 10 | coef << 18
// (coef 0: no second term, src2 = 0).
struct HermSteps {
    unsigned w[nherm(9)];
};
constexpr HermSteps make_herm_steps()
{
    HermSteps s{};
    for (int h = 1; h < nherm(9); ++h) {
        const Triple x = herm_triple(h);
        const int d = x.t > 0 ? 0 : (x.u > 0 ? 1 : 2), c = d == 0 ? x.t : (d == 1 ? x.u : x.v);
        const int s1 = hidx(x.t - (d == 0), x.u - (d == 1), x.v - (d == 2));
        const int s2 = c > 1 ? hidx(x.t - 2 * (d == 0), x.u - 2 * (d == 1), x.v - 2 * (d == 2)) : 0;
        s.w[h] = (unsigned)d | ((unsigned)s1 << 2) | ((unsigned)s2 << 10) | ((unsigned)(c - 1) << 18);
    }
    return s;
}
static __device__ const HermSteps kHermSteps = make_herm_steps();

// Barrier of the NW warps that share a quartet.
template <int NW>
__device__ __forceinline__ void quartet_sync()
{
    if constexpr (NW == 1) __syncwarp();
    else __syncthreads();
}

// The entries of one level (totals up to top) in the columns of 32 primitive
// quartets by NW warps: total by total from the top, whose entries read the two
// totals below only, so one barrier a total orders reads and writes.
template <int RS, int NW>
__device__ __forceinline__ void hermite_level_warps(double *Rl, int warp, int top, double X, double Y, double Z)
{
#pragma unroll 1
    for (int k = top; k >= 1; --k) {
        const int end = nherm(k);
#pragma unroll 1
        for (int h = nherm(k - 1) + warp; h < end; h += 4 * NW) {
            double v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned w = kHermSteps.w[h + j * NW < end ? h + j * NW : h];
                const unsigned dir = w & 3;
                v[j] = (dir == 0 ? X : (dir == 1 ? Y : Z)) * Rl[((w >> 2) & 0xff) * RS];
                const int c = (int)(w >> 18);
                if (c > 0) v[j] += double(c) * Rl[((w >> 10) & 0xff) * RS];
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (h + j * NW < end) Rl[(h + j * NW) * RS] = v[j];
        }
        quartet_sync<NW>();
    }
}

// Entries 1 .. n - 1 of one level in this lane's column, in place, from high
// to low: every entry reads lower ones, and of four at a time all reads
// precede the writes.
template <int RS>
__device__ __forceinline__ void hermite_level(double *Rl, int n, double X, double Y, double Z)
{
#pragma unroll 1
    for (int h = n - 1; h >= 1; h -= 4) {
        double v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned w = kHermSteps.w[h - k > 0 ? h - k : 1];
            const unsigned dir = w & 3;
            v[k] = (dir == 0 ? X : (dir == 1 ? Y : Z)) * Rl[((w >> 2) & 0xff) * RS];
            const int c = (int)(w >> 18);  // the same for all lanes
            if (c > 0) v[k] += double(c) * Rl[((w >> 10) & 0xff) * RS];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (h - k > 0) Rl[(h - k) * RS] = v[k];
    }
}

// ------------------------------------------------------------ quartet

// Gamma_op of the group's quartets (the 8 permutation images of the pair
// products, times scale), [ket][op][cd][ab], for operators o0 .. o0 + NO - 1.
template <int LA, int LB, int LC, int LD>
__device__ __forceinline__ void herm_gamma(double *G, int tid, int kg, const GroupInfo &gi, int k0, int o0, const DensArgs &den,
                                           const int *sh_bf, int fa, int fb)
{
    using Lay = HermLay<LA, LB, LC, LD>;
    constexpr int NB = ncart(LB), ND = ncart(LD), NFQ = Lay::NAB * Lay::NCD;
    const int nbf = den.nbf;
    for (int x = tid; x < kg * NFQ; x += 32 * Lay::NW) {
        const int kq = x / NFQ, it = x % NFQ, cd = it / Lay::NAB, ab = it % Lay::NAB;
        double *g = G + kq * Lay::GS + cd * Lay::NABP + ab;
        double g0 = 0.0, g1 = 0.0;
        if (k0 + kq < gi.n) {
            const size_t m = fa + ab / NB, n = fb + ab % NB;
            const size_t l = sh_bf[gi.sc[k0 + kq]] + cd / ND, s = sh_bf[gi.sd[k0 + kq]] + cd % ND;
            for (int p = 0; p < den.npair; ++p) {
                const double *A = den.A[p], *B = den.B[p];
                const double cj = den.cJ[p], ck = den.cK[p], cl = den.cKlr[p];
                if (cj != 0.0 && (Lay::NO == 2 || o0 == 0))
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
            g0 *= gi.scale[k0 + kq];
            g1 *= gi.scale[k0 + kq];
        }
        if constexpr (Lay::NO == 2) {
            g[0] = g0;
            g[Lay::NCD * Lay::NABP] = g1;
        } else {
            g[0] = o0 == 0 ? g0 : g1;
        }
    }
}

// c^{ab}_m R^.. of every table entry of a pair class, for n pairs (powers pw,
// 15 apart).
template <int LA, int LB, int NT = 32>
__device__ __forceinline__ void entry_values(double *out, int tid, const double *pw, int n)
{
    const auto &T = pair_tab<LA, LB>();
    constexpr int NE = PairTab<LA, LB>::NE;
    for (int x = tid; x < n * NE; x += NT) {
        const unsigned w = T.ent[x % NE];
        const double *q = pw + x / NE * 15;
        out[x] = double((int)((w >> 8) & 0xff)) * q[(w >> 16) & 7] * q[5 + ((w >> 19) & 7)] * q[10 + ((w >> 22) & 7)];
    }
}

// half[ket][o][m2][ab] = sum_{entries of m2} value Gamma[cd][ab]
template <int LA, int LB, int LC, int LD>
__device__ __forceinline__ void half_ket(double *half, const double *G, const double *vk, int tid, int kg)
{
    using Lay = HermLay<LA, LB, LC, LD>;
    const auto &T = pair_tab<LC, LD>();
    constexpr int N = Lay::NM2 * Lay::NAB;
    for (int x = tid; x < kg * N; x += 32 * Lay::NW) {
        const int kq = x / N, it = x % N, m = it / Lay::NAB, ab = it % Lay::NAB;
        const double *v = vk + kq * Lay::NE2;
#pragma unroll
        for (int o = 0; o < Lay::NO; ++o) {
            const double *g = G + kq * Lay::GS + o * Lay::NCD * Lay::NABP + ab;
            double s = 0.0;
            for (int e = T.start[m]; e < T.start[m + 1]; ++e) s += v[e] * g[(T.ent[e] & 0xff) * Lay::NABP];
            half[kq * Lay::HS + (o * Lay::NM2 + m) * Lay::NABP + ab] = s;
        }
    }
}

// items table of the class a translation unit compiles
template <int LA, int LB, int LC, int LD, bool ALL>
__device__ const HermItems<LA, LB, LC, LD, ALL> kHermItems = make_herm_items<LA, LB, LC, LD, ALL>();

// Reverse sums of one pass (primitive quartets j0 .. j0 + n - 1 of the block, n
// <= 32, lane j - j0's R in column j - j0 of Rr): per bra primitive pair,
// U[h1][m2] = sum_q s_m2 R[h1 + h2], added to V[m1][m2] with its scalars.
template <int LA, int LB, int LC, int LD, bool ALL, int NW = 1>
__device__ __forceinline__ void reverse_sums(double *V, const double *Rr, const double *S2, const double *S1, int j0,
                                             int n, int nkp, int tid)
{
    using B = PairMono<LA, LB>;
    constexpr int NIT = HermItems<LA, LB, LC, LD, ALL>::N, RS = 33, NM2P = PairMono<LC, LD>::NM | 1;
    // lanes per item: as many as fit
    constexpr int SUB = NIT <= 1 ? 16 : (NIT <= 4 ? 8 : (NIT <= 8 ? 4 : (NIT <= 16 ? 2 : 1)));
    constexpr int ITL = 32 / SUB;
    const auto &TBra = pair_tab<LA, LB>();
    const unsigned *items = kHermItems<LA, LB, LC, LD, ALL>.it;
    static_assert(NW == 1 || SUB == 1, "several warps: one lane an item");
    const int pfirst = j0 / nkp, plast = (j0 + n - 1) / nkp, sub = NW == 1 ? tid / ITL : 0;
    for (int i0 = 0; i0 < NIT; i0 += ITL * NW) {
        const int it = i0 + tid % (ITL * NW);
        const unsigned w = items[it < NIT ? it : NIT - 1];
        const double *r = Rr + (w & 0xff) * RS, *s = S2 + (w >> 21) * RS;
        const unsigned hm = TBra.hm[(w >> 8) & 0x3f];
        double *v = V + (hm & 0xff) * NM2P + ((w >> 14) & 0x7f);
        const int ns = (hm >> 8) & 0xf;
        for (int pj = pfirst; pj <= plast; ++pj) {
            const int lo = max(pj * nkp - j0, 0), hi = min((pj + 1) * nkp - j0, n);
            double u = 0.0;
#pragma unroll 4
            for (int j = lo + sub; j < hi; j += SUB) u += s[j] * r[j];
#pragma unroll
            for (int x = ITL; x < 32; x *= 2) u += __shfl_xor_sync(0xffffffffu, u, x);
            if (it < NIT && sub == 0) {
                const double *s1 = S1 + pj * B::NS + (hm >> 12);
                for (int k = 0; k < ns; ++k) v[k * NM2P] += s1[k] * u;
            }
        }
    }
}

// The same for a group of kg > 1 ket pairs, whose lanes are kq LG .. kq LG +
// LG - 1 with the primitive quartets it0 .. it0 + LG - 1 of its own list of np
// * nks[kq]; V of ket pair kq at V + kq * vs.
template <int LA, int LB, int LC, int LD>
__device__ __forceinline__ void reverse_sums_group(double *V, int vs, const double *Rr, const double *S2,
                                                   const double *S1, int it0, int np, int kg, int LG,
                                                   const int *nks, int lane)
{
    using B = PairMono<LA, LB>;
    constexpr int NIT = HermItems<LA, LB, LC, LD, false>::N, RS = 33, NM2P = PairMono<LC, LD>::NM | 1;
    const auto &TBra = pair_tab<LA, LB>();
    const unsigned *items = kHermItems<LA, LB, LC, LD, false>.it;
    for (int x = lane; x < kg * NIT; x += 32) {
        const int kq = x / NIT, nk = nks[kq];
        const int n = min(LG, np * nk - it0);
        if (n <= 0) continue;
        const unsigned w = items[x % NIT];
        const double *r = Rr + (w & 0xff) * RS + kq * LG, *s = S2 + (w >> 21) * RS + kq * LG;
        const unsigned hm = TBra.hm[(w >> 8) & 0x3f];
        double *v = V + kq * vs + (hm & 0xff) * NM2P + ((w >> 14) & 0x7f);
        const int ns = (hm >> 8) & 0xf;
        int pj = it0 / nk, j = 0;
        while (j < n) {
            const int hi = min((pj + 1) * nk - it0, n);
            double u = 0.0;
#pragma unroll 4
            for (; j < hi; ++j) u += s[j] * r[j];
            const double *s1 = S1 + pj * B::NS + (hm >> 12);
            for (int k = 0; k < ns; ++k) v[k * NM2P] += s1[k] * u;
            ++pj;
        }
    }
}

// Bra primitive pairs taken at a time (1 .. cap, at most nbra): the block of
// pb * nkp primitive quartets that leaves the fewest of its lanes idle.
__device__ __forceinline__ int block_pairs(int nbra, int nkp, int cap, int lanes = 32)
{
    int pb = 1, best = -1;
    for (int c = 1; c <= (nbra < cap ? nbra : cap); ++c) {
        const int n = c * nkp, use = n * 64 / ((n + lanes - 1) / lanes);  // primitive quartets per pass, times 64
        if (use >= best) best = use, pb = c;
    }
    return pb;
}

// A group of kg (1, 2, 4, 8; at most KQ) ket pairs with one bra pair by one
// warp, bra primitive pairs ib0, ib0 + ibs, ...  Lanes kq LG .. kq LG + LG - 1
// (LG = 32 / kg) take the primitive quartets of ket pair kq: the density
// transform, its loads and the closing sums, which a few lanes of a single
// quartet would leave half empty in the small classes, run over all ket pairs
// at once.  acc[0..2] += d/dA, acc[3..5] += d/dA + d/dB, acc[6..8] += d/dC
// (this lane's share; d/dA of all ket pairs may sit on any lane, the others on
// their ket pair's lanes).
template <int LA, int LB, int LC, int LD>
__device__ void group_herm(double *sm, int tid, int k0, int kg, const GroupInfo &gi, const GeoArgs &geo, const DensArgs &den,
                           const PrimPairs &pp, int sa, int sb, int pb0, int nbp, int ib0, int ibs, const double *boys,
                           double (&acc)[9])
{
    using Lay = HermLay<LA, LB, LC, LD>;
    constexpr int NCD = Lay::NCD, L = Lay::L, LM = Lay::LM, NT1 = Lay::NT1;
    constexpr int NM1 = Lay::NM1, NM2 = Lay::NM2, NM2P = Lay::NM2P, NS1 = Lay::NS1, NS2 = Lay::NS2, RS = Lay::RS;
    constexpr int NO = Lay::NO, NP1 = Lay::NP1, NABP = Lay::NABP, KQ = Lay::KQ;
    constexpr int NW = Lay::NW, NT = 32 * NW;  // warps and threads that share the group
    const int lane = tid % 32, warp = tid / 32;
    constexpr int NIT = HermItems<LA, LB, LC, LD, false>::N;
    double *G = sm + Lay::o_G, *Gp = sm + Lay::o_Gp, *V = sm + Lay::o_V, *F = sm + Lay::o_F;
    double *S1 = sm + Lay::o_S1, *P1 = sm + Lay::o_P1, *pw = sm + Lay::o_pw, *X1 = sm + Lay::o_X;
    double *Rr = X1, *S2 = X1 + Lay::NRH * RS;                                    // main loop
    double *vb = X1, *vk = X1 + Lay::NE1, *half = vk + KQ * Lay::NE2;              // transforms
    const auto &TBra = pair_tab<LA, LB>();
    const auto &TKet = pair_tab<LC, LD>();
    const int nops = den.use_lr ? 2 : 1;
    const bool ominf = isinf(den.omega);
    const double om = ominf ? 1.0 : den.omega;
    if constexpr (KQ == 1) kg = 1;
    const int LG = 32 / kg, kq = lane / LG, sl = lane % LG;
    if (tid < 3 + 3 * kg) {  // powers of R = A - B and of every S = C - D
        const int d = lane % 3, w = lane / 3;
        const int k = min(k0 + w - 1, gi.n - 1);
        const int s0 = w == 0 ? sa : gi.sc[k], s1 = w == 0 ? sb : gi.sd[k];
        const double x = geo.xyz[3 * geo.sh_atom[s0] + d] - geo.xyz[3 * geo.sh_atom[s1] + d];
        double p = 1.0;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            pw[w * 15 + d * 5 + i] = p;
            p *= x;
        }
    }
    int nkmax = gi.nk[k0];
    for (int k = 1; k < kg; ++k) nkmax = max(nkmax, gi.nk[k0 + k]);
    const int nk = gi.nk[k0 + kq], nkd = max(nk, 1), pk0 = gi.pk0[k0 + kq];  // this lane's ket pair
    const int nbra = (nbp - ib0 + ibs - 1) / ibs;                  // bra primitive pairs of this call
    const int pb = block_pairs(nbra, nkmax, Lay::PB, LG);
    // this lane's sums over its primitive quartets: T, a^ T, c^ T, mu_ab E, mu_cd E
    double aT[3] = {0.0, 0.0, 0.0}, aA[3] = {0.0, 0.0, 0.0}, aC[3] = {0.0, 0.0, 0.0}, eA = 0.0, eC = 0.0;
    double gA[3] = {0.0, 0.0, 0.0}, gC[3] = {0.0, 0.0, 0.0};  // polynomial parts
    quartet_sync<NW>();

    for (int o0 = 0; o0 < nops; o0 += NO) {
        // ---- Gamma -> G'[m1][m2]
        herm_gamma<LA, LB, LC, LD>(G, tid, kg, gi, k0, o0, den, geo.sh_bf, geo.sh_bf[sa], geo.sh_bf[sb]);
        entry_values<LA, LB, NT>(vb, tid, pw, 1);
        entry_values<LC, LD, NT>(vk, tid, pw + 15, kg);
        quartet_sync<NW>();
        half_ket<LA, LB, LC, LD>(half, G, vk, tid, kg);
        quartet_sync<NW>();
        for (int x = tid; x < kg * NM1 * NM2; x += NT) {
            const int q = x / (NM1 * NM2), it = x % (NM1 * NM2), m1 = it / NM2, m2 = it % NM2;
#pragma unroll
            for (int o = 0; o < NO; ++o) {
                const double *h = half + q * Lay::HS + (o * NM2 + m2) * NABP;
                double s = 0.0;
                for (int e = TBra.start[m1]; e < TBra.start[m1 + 1]; ++e) s += vb[e] * h[TBra.ent[e] & 0xff];
                Gp[q * Lay::MS + (o * NM1 + m1) * NM2P + m2] = s;
                V[q * Lay::MS + (o * NM1 + m1) * NM2P + m2] = 0.0;
            }
        }
        quartet_sync<NW>();

        for (int blk = 0; blk < nbra; blk += pb) {
            const int np = min(pb, nbra - blk);
            // ---- scalars of the block's bra primitive pairs, then F[p][ket][h1][m2]
            if (tid < np) {
                const int ip = pb0 + ib0 + (blk + tid) * ibs;
                const double a = pp.fa[ip], b = pp.fb[ip];
                double s[NS1];
                pair_scalars<LA, LB, false>(pp.oo2[ip], a, b, s);
#pragma unroll
                for (int k = 0; k < NS1; ++k) S1[tid * NS1 + k] = s[k];
                P1[tid * NP1] = a;
                P1[tid * NP1 + 1] = pp.za[ip] * b;
                P1[tid * NP1 + 2] = pp.kop[ip] * 34.986836655249725;  // 2 pi^(5/2) K / p
                P1[tid * NP1 + 3] = pp.p[ip];
            }
            quartet_sync<NW>();
            for (int x = tid; x < np * kg * NT1 * NM2; x += NT) {
                const int pq = x / (NT1 * NM2), r = x % (NT1 * NM2), h = r / NM2, m2 = r % NM2;
                const int pi = pq / kg, q = pq % kg;
                const unsigned hm = TBra.hm[h];
                const double *g = Gp + q * Lay::MS + (hm & 0xff) * NM2P + m2, *s = S1 + pi * NS1 + (hm >> 12);
                const int ns = (hm >> 8) & 0xf;
#pragma unroll
                for (int o = 0; o < NO; ++o) {
                    double f = 0.0;
                    for (int k = 0; k < ns; ++k) f += s[k] * g[(o * NM1 + k) * NM2P];
                    F[(pi * KQ + q) * Lay::FS + (o * NT1 + h) * NM2P + m2] = f;
                }
            }
            quartet_sync<NW>();
            const int ntot = np * nk, nmax = np * nkmax;
            for (int it0 = 0; it0 < nmax; it0 += LG) {
                // ---- this lane's primitive quartet
                const int idx = max(min(it0 + sl, ntot - 1), 0);
                const int pi = idx / nkd;
                const int ip = pb0 + ib0 + (blk + pi) * ibs, kp = pk0 + (idx - pi * nkd);
                const double p = P1[pi * NP1 + 3], q = pp.p[kp], c = pp.fa[kp], d = pp.fb[kp];
                const double ir = rsqrt(p + q);
                const double rho = p * q * ir * ir;
                const double X = pp.Px[ip] - pp.Px[kp], Y = pp.Py[ip] - pp.Py[kp], Z = pp.Pz[ip] - pp.Pz[kp];
                const double T0 = rho * (X * X + Y * Y + Z * Z);
                // lanes past the end repeat a quartet with weight zero
                const double pref = it0 + sl < ntot ? P1[pi * NP1 + 2] * pp.kop[kp] * ir : 0.0;
                double s2[NS2];
                pair_scalars<LC, LD, true>(pp.oo2[kp], c, d, s2);
                if (NIT > 0 && warp == 0)
#pragma unroll
                    for (int k = 0; k < NS2; ++k) S2[k * RS + lane] = s2[k];
                double e = 0.0, T[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
                for (int o = 0; o < NO; ++o) {
                    if (o0 + o >= nops) break;
                    double base[LM + 1];
                    {
                        double th = 1.0;
                        if (o0 + o == 1 && !ominf) th = om * rsqrt(om * om + rho);
                        double Fm[LM + 1];
                        const double th2 = th * th;
                        boys_lane<LM>(T0 * th2, Fm, boys);
                        double f = pref * th;
                        const double m2r = -2.0 * rho * th2;
#pragma unroll
                        for (int n = 0; n <= LM; ++n) {
                            base[n] = f * Fm[n];
                            f *= m2r;
                        }
                    }
                    const double *Fl = F + (pi * KQ + kq) * Lay::FS + o * NT1 * NM2P;
                    double *Rl = Rr + lane;
                    if constexpr (Lay::RREG) {
                        double Xd[nherm(L)];
                        hermite_density<LA, LB, LC, LD, 0, L>(Fl, s2, Xd);
                        double R[nherm(LM)];
                        hermite_R<LM>(R, base, X, Y, Z);
                        static_for<nherm(LM)>([&](auto H) {
                            energy_terms<L, decltype(H)::value>(R[decltype(H)::value], Xd, e, T);
                        });
                        if constexpr (NIT > 0)
#pragma unroll
                            for (int h = 0; h < Lay::NRH; ++h) Rl[h * RS] = R[h];
                    } else {
                        // every warp forms the scalars; then (0,0,0) of a level is written after
                        // its entries, which read the level above
                        if (warp == 0) Rl[0] = base[LM];
                        quartet_sync<NW>();
                        static_for<LM>([&](auto I) {
                            constexpr int n = LM - 1 - decltype(I)::value;
                            hermite_level_warps<RS, NW>(Rl, warp, LM - n, X, Y, Z);
                            if (warp == 0) Rl[0] = base[n];
                            quartet_sync<NW>();
                        });
                        // a quarter of the density's products each ((dd|dd): 750, 585, 650, 675) or
                        // a half ((dp|dp): 400 and 280 with more sums to close)
                        if constexpr (NW == 2) {
                            if (warp == 0) density_pass<LA, LB, LC, LD, 0, L - 2>(Fl, s2, Rl, e, T);
                            else density_pass<LA, LB, LC, LD, L - 1, L>(Fl, s2, Rl, e, T);
                        } else if (warp == 0) density_pass<LA, LB, LC, LD, 0, 4>(Fl, s2, Rl, e, T);
                        else if (warp == 1) density_pass<LA, LB, LC, LD, 5, 5>(Fl, s2, Rl, e, T);
                        else if (warp == 2) density_pass<LA, LB, LC, LD, 6, 6>(Fl, s2, Rl, e, T);
                        else density_pass<LA, LB, LC, LD, 7, L>(Fl, s2, Rl, e, T);
                    }
                    quartet_sync<NW>();
                    // ---- reverse sums U[h1][m2], added to V with the bra scalars
                    if constexpr (NIT > 0) {
                        if (kg == 1)
                            reverse_sums<LA, LB, LC, LD, false, NW>(V + o * NM1 * NM2P, Rr, S2, S1, it0,
                                                                    min(32, ntot - it0), nkd, tid);
                        else if constexpr (KQ > 1)
                            reverse_sums_group<LA, LB, LC, LD>(V + o * NM1 * NM2P, Lay::MS, Rr, S2, S1, it0, np, kg, LG,
                                                               gi.nk + k0, lane);
                        quartet_sync<NW>();
                    }
                }
                const double a = P1[pi * NP1];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    aT[i] += T[i];
                    aA[i] += a * T[i];
                    aC[i] += c * T[i];
                }
                eA += P1[pi * NP1 + 1] * e;
                eC += pp.za[kp] * d * e;
            }
            quartet_sync<NW>();  // S1, P1 and F are rewritten for the next block
        }
        // ---- polynomial parts: V with dG'/dR (ket half again) and dG'/dS (bra half)
        if constexpr (NIT > 0) {
            entry_values<LA, LB, NT>(vb, tid, pw, 1);
            if constexpr (Lay::L1 > 0) entry_values<LC, LD, NT>(vk, tid, pw + 15, kg);
            quartet_sync<NW>();
            if constexpr (Lay::L1 > 0) {
                half_ket<LA, LB, LC, LD>(half, G, vk, tid, kg);
                quartet_sync<NW>();
                for (int x = tid; x < kg * Lay::NE1; x += NT) {
                    const int q = x / Lay::NE1, it = x % Lay::NE1;
                    const unsigned w = TBra.ent[it];
                    const int px = (w >> 16) & 7, py = (w >> 19) & 7, pz = (w >> 22) & 7;
                    if (px + py + pz == 0) continue;
                    const int m1 = TBra.own[it], ab = w & 0xff;
                    double s = 0.0;
#pragma unroll
                    for (int o = 0; o < NO; ++o) {
                        const double *h = half + q * Lay::HS + o * NM2 * NABP + ab;
                        const double *v = V + q * Lay::MS + (o * NM1 + m1) * NM2P;
                        for (int m2 = 0; m2 < NM2; ++m2) s += h[m2 * NABP] * v[m2];
                    }
                    s *= double((int)((w >> 8) & 0xff));
                    const double qx = pw[px], qy = pw[5 + py], qz = pw[10 + pz];
                    if (px) gA[0] += s * double(px) * pw[px - 1] * qy * qz;
                    if (py) gA[1] += s * double(py) * qx * pw[5 + py - 1] * qz;
                    if (pz) gA[2] += s * double(pz) * qx * qy * pw[10 + pz - 1];
                }
                quartet_sync<NW>();
            }
            if constexpr (Lay::L2 > 0) {
                // bra half [ket][o][m1][cd]
                for (int x = tid; x < kg * NM1 * NCD; x += NT) {
                    const int q = x / (NM1 * NCD), it = x % (NM1 * NCD), m1 = it / NCD, cd = it % NCD;
#pragma unroll
                    for (int o = 0; o < NO; ++o) {
                        const double *g = G + q * Lay::GS + (o * NCD + cd) * NABP;
                        double s = 0.0;
                        for (int k = TBra.start[m1]; k < TBra.start[m1 + 1]; ++k) s += vb[k] * g[TBra.ent[k] & 0xff];
                        half[q * Lay::HS + (o * NM1 + m1) * NCD + cd] = s;
                    }
                }
                quartet_sync<NW>();
                const double *pk = pw + (1 + kq) * 15;
                for (int it = sl + 32 * warp; it < Lay::NE2; it += LG * NW) {
                    const unsigned w = TKet.ent[it];
                    const int px = (w >> 16) & 7, py = (w >> 19) & 7, pz = (w >> 22) & 7;
                    if (px + py + pz == 0) continue;
                    const int m2 = TKet.own[it], cd = w & 0xff;
                    double s = 0.0;
#pragma unroll
                    for (int o = 0; o < NO; ++o) {
                        const double *h = half + kq * Lay::HS + o * NM1 * NCD + cd;
                        const double *v = V + kq * Lay::MS + o * NM1 * NM2P + m2;
                        for (int m1 = 0; m1 < NM1; ++m1) s += h[m1 * NCD] * v[m1 * NM2P];
                    }
                    s *= double((int)((w >> 8) & 0xff));
                    const double qx = pk[px], qy = pk[5 + py], qz = pk[10 + pz];
                    if (px) gC[0] += s * double(px) * pk[px - 1] * qy * qz;
                    if (py) gC[1] += s * double(py) * qx * pk[5 + py - 1] * qz;
                    if (pz) gC[2] += s * double(pz) * qx * qy * pk[10 + pz - 1];
                }
            }
        }
        quartet_sync<NW>();
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        acc[i] += aA[i] - 2.0 * pw[i * 5 + 1] * eA + gA[i];
        acc[3 + i] += aT[i];
        acc[6 + i] += -aC[i] - 2.0 * pw[(1 + kq) * 15 + i * 5 + 1] * eC + gC[i];
    }
}

// Warps of a CTA, and CTAs an SM that the registers are limited to: 16 warps at
// 128 registers up to L = 2, 12 at 168 for L = 3, 8 at 255 above (12 at 168 for
// (dd|dp), of whose three CTAs shared memory holds two).  One warp per scheduler
// already covers most of the fp64 pipe; the others fill the gaps left by the
// transforms' loads and by dependent steps.  1/8 of the 32-atom workload in fp64,
// classes one after the other and as one call: 220 and 199 ms; with 12 warps up to
// L = 2, 8 for L = 3 and 6 for L = 4: 220 and 195 ms; with 20, 16 and 12: 225 and
// 231 ms.  CTAs are small (one or two warps) because a CTA gives its shared memory
// back only when its last warp ends: with 8 to 16 warps a single long quartet kept
// a whole SM from the next class's launch.
template <int LA, int LB, int LC, int LD>
struct HermOp {
    using Lay = HermLay<LA, LB, LC, LD>;
    static constexpr bool FP32 = false;
    static constexpr int L = LA + LB + LC + LD, KQ = Lay::KQ;
    static constexpr int NW = Lay::NW;  // warps per worker (a worker takes units alone)
    static constexpr int cta_workers = L <= 3 ? 2 : 1, min_ctas = L == 3 ? 6 : (NW == 1 ? 8 : (NW == 2 ? 4 : 10 - L));
    // primitive quartets of a contracted one up to which ket pairs are grouped
    // (kg times it stays below): the smaller the class, the more of a quartet's
    // work is the density transform that a group shares.  On that shard (ps|ss) takes
    // 10.4 ms (9.6 at twice these bounds, 11.8 at half, 16.2 ungrouped), (pp|ss) 7.5
    // (7.2, 8.0, 9.0), (ss|ss) 2.2 (2.2, 2.3, 3.3; 2.6 always grouped)
    static constexpr int group_below = L == 0 ? 512 : (L == 1 ? 256 : (L == 2 ? 128 : 64));
    static __device__ __forceinline__ void group(double *sm, int tid, int k0, int kg, const GroupInfo &gi,
                                                 const MolDesc &md, int sa, int sb, int pb0, int nbp, int ib0, int ibs, const double *boys,
                                                 double (&acc)[9])
    {
        group_herm<LA, LB, LC, LD>(sm, tid, k0, kg, gi, md.geo, md.den, md.pp, sa, sb, pb0, nbp, ib0, ibs, boys, acc);
    }
};

// Persistent class kernel; every warp works alone.  Warp w of W takes the
// units (tile, chunk of cl.nchunk per tile, split) w, 2W - 1 - w, 2W + w, ...:
// a molecule's tiles are in decreasing cost, so the alternating order evens the
// sums out (in a batch the order starts again with every molecule, and two of
// 21 and 26 atoms take 638 ms against 599 ms one after the other).  A unit's quartets are taken in groups of up to KQ ket pairs of one
// bra pair.  Their components are added to the warp's own gradient (shared
// memory, or with out.use_smem = 0 the warp's slab), so the schedule and the
// order of all sums are fixed and results are bitwise reproducible.
template <class Op>
__global__ void __launch_bounds__(32 * Op::NW * Op::cta_workers, Op::min_ctas)
    k_grad_lanes(const MolDesc *__restrict__ mols, ClassLaunch cl, OutArgs out, const double *__restrict__ boys)
{
    using Lay = typename Op::Lay;
    constexpr int RS = Lay::RS, KQ = Op::KQ, NW = Op::NW, NT = 32 * NW;
    extern __shared__ double smem[];
    __shared__ GroupInfo ginfo[Op::cta_workers];
    // nw workers of NW warps each; every warp of a worker walks the same units
    const int nw = blockDim.x / NT, grp = threadIdx.x / NT, tid = threadIdx.x % NT, lane = tid % 32;
    const int n3 = out.natom_total * 3;
    double *wsm = smem + (size_t)grp * Lay::TOTAL;
    GroupInfo &gi = ginfo[grp];
    double *grad = out.use_smem ? smem + (size_t)nw * Lay::TOTAL + (size_t)grp * n3
                                : out.partials + (size_t)(blockIdx.x * nw + grp) * n3;
    if (out.use_smem) {
        for (int k = tid; k < n3; k += NT) grad[k] = 0.0;
        quartet_sync<NW>();
    }
    unsigned long long nq = 0, npq = 0, nbv = 0;  // of this lane's ket pair
    const int S = cl.nsplit, C = cl.nchunk, QPC = TILE / C;
    const int KG = out.dump ? 1 : (QPC < KQ ? QPC : KQ);
    const bool same = cl.P == cl.Q;
    const long long units = cl.ntiles * C * S, W = (long long)gridDim.x * nw;
    // neighbouring warps sit on different CTAs, so a short list spreads over the SMs
    const long long w0 = (long long)grp * gridDim.x + blockIdx.x;
    for (long long r = 0; r * W < units; ++r) {
        const long long it = r * W + ((r & 1) ? W - 1 - w0 : w0);
        if (it >= units) continue;
        const long long tile = it / (C * S);
        const int chunk = (int)((it / S) % C), split = (int)(it % S);
        const uint4 tl = cl.tiles[tile];
        const MolDesc &md = mols[tl.x];
        const PairSet &bra = md.sets[cl.P], &ket = md.sets[cl.Q];
        for (int qi = chunk * QPC; qi < (chunk + 1) * QPC; qi += KG) {
            const int bi = tl.y * TB + qi / TK;
            // lane k < KG: ket pair k of the group
            const int ki = tl.z * TK + qi % TK + lane;
            bool ok = lane < KG && bi < bra.n && ki < ket.n && (!same || bi >= ki);
            if (ok) ok = split < bra.np[bi];
            int sa = 0, sb = 0, sc = 0, sd = 0;
            if (ok) {
                sa = bra.sa[bi];
                sb = bra.sb[bi];
                sc = ket.sa[ki];
                sd = ket.sb[ki];
                ok = keep_quartet(md.scr, bra, ket, bi, ki, sa, sb, sc, sd);
            }
            if (ok) {
                const int nbs = (bra.np[bi] - split + S - 1) / S;
                if (split == 0) nq += 1;  // (only a worker's first warp reports)
                npq += (unsigned long long)nbs * ket.np[ki];
                nbv += (unsigned long long)nbs;
                ok = ket.np[ki] > 0;  // all screened: counted, nothing to add
            }
            const unsigned mask = __ballot_sync(0xffffffffu, ok);
            double g = 0.0;
            if (mask) {
                const int n = __popc(mask), first = __ffs(mask) - 1;
                sa = __shfl_sync(0xffffffffu, sa, first);
                sb = __shfl_sync(0xffffffffu, sb, first);
                const int nbp = bra.np[bi], nbs = (nbp - split + S - 1) / S;
                if (ok && tid < 32) {
                    const int k = __popc(mask & ((1u << lane) - 1));
                    double scale = 1.0;
                    if (sa == sb) scale *= 0.5;
                    if (sc == sd) scale *= 0.5;
                    if (same && bi == ki) scale *= 0.5;
                    gi.sc[k] = sc;
                    gi.sd[k] = sd;
                    gi.pk0[k] = ket.poff[ki];
                    gi.nk[k] = ket.np[ki];
                    gi.scale[k] = scale;
                    if (k == 0) {
                        gi.n = n;
                        for (int j = n; j < GroupInfo::CAP; ++j) gi.nk[j] = 0, gi.pk0[j] = ket.poff[ki];
                    }
                }
                quartet_sync<NW>();
                int kg = 1;
                if (KQ > 1) {
                    int nkmax = gi.nk[0];
                    for (int k = 1; k < n; ++k) nkmax = max(nkmax, gi.nk[k]);
                    while (kg < n && 2 * kg <= KQ && 2 * kg * nbs * nkmax <= Op::group_below) kg *= 2;
                }
                for (int k0 = 0; k0 < n; k0 += kg) {
                    double acc[9];
#pragma unroll
                    for (int k = 0; k < 9; ++k) acc[k] = 0.0;
                    Op::group(wsm, tid, k0, kg, gi, md, sa, sb, bra.poff[bi], nbp, split, S, boys, acc);
                    // the nine sums of every ket pair over its 32 / kg lanes, through shared memory
                    double *red = wsm + Lay::o_X;
                    quartet_sync<NW>();
#pragma unroll
                    for (int k = 0; k < 9; ++k) red[(tid / 32 * 9 + k) * RS + lane] = acc[k];
                    quartet_sync<NW>();
                    if (kg == 1) {  // three lanes a sum
                        double s = 0.0;
                        const int k = lane / 3 < 9 ? lane / 3 : 8, part = lane % 3;
#pragma unroll
                        for (int w = 0; w < NW; ++w)
                            for (int j = part; j < 32; j += 3) s += red[(w * 9 + k) * RS + j];
                        const double s1 = __shfl_down_sync(0xffffffffu, s, 1), s2 = __shfl_down_sync(0xffffffffu, s, 2);
                        if (NW > 1) quartet_sync<NW>();  // all have read
                        if (part == 0 && lane < 27 && tid < 32) red[k * RS] = s + s1 + s2;
                    } else {
                        const int lg = 32 / kg;
                        for (int x = lane; x < 9 * kg; x += 32) {
                            double *p = red + (x % 9) * RS + x / 9 * lg;
                            double s = p[0];
                            for (int j = 1; j < lg; ++j) s += p[j];
                            p[0] = s;
                        }
                    }
                    quartet_sync<NW>();
                    const int i = lane % 3, lg = 32 / kg;
                    if (out.dump) {  // one ket pair; lanes 0..11: output component X * 3 + i
                        const int X = lane / 3;
                        const double dA = red[i * RS], dT = red[(3 + i) * RS], dC = red[(6 + i) * RS];
                        g = X == 0 ? dA : (X == 1 ? dT - dA : (X == 2 ? dC : -dT - dC));
                    } else if (tid < 3) {  // lane i owns component i of every atom
                        const int *at = md.geo.sh_atom;
                        double *gr = grad + md.atom_off * 3 + i;
                        double dA = 0.0, dT = 0.0;
                        for (int k = 0; k < kg && k0 + k < n; ++k) {
                            const double t = red[(3 + i) * RS + k * lg], c = red[(6 + i) * RS + k * lg];
                            gr[at[gi.sc[k0 + k]] * 3] += c;
                            gr[at[gi.sd[k0 + k]] * 3] += -t - c;
                            dT += t;
                        }
                        for (int k = 0; k < kg; ++k) dA += red[i * RS + k * lg];
                        gr[at[sa] * 3] += dA;
                        gr[at[sb] * 3] += dT - dA;
                    }
                    quartet_sync<NW>();
                }
                quartet_sync<NW>();
            }
            if (out.dump && tid < 12) out.dump[((size_t)tile * TILE + qi) * 12 + lane] = g;
        }
    }
    if (out.use_smem && !out.dump) {
        __syncthreads();
        double *slab = out.partials + (size_t)blockIdx.x * n3;
        const double *all = smem + (size_t)nw * Lay::TOTAL;
        for (int k = threadIdx.x; k < n3; k += blockDim.x) {
            double s = 0.0;
            for (int w = 0; w < nw; ++w) s += all[(size_t)w * n3 + k];
            slab[k] += s;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        nq += __shfl_xor_sync(0xffffffffu, nq, o);
        npq += __shfl_xor_sync(0xffffffffu, npq, o);
        nbv += __shfl_xor_sync(0xffffffffu, nbv, o);
    }
    if (tid == 0 && (nq || npq)) {  // a split unit may hold primitives only
        atomicAdd(out.counters + 0, nq);
        atomicAdd(out.counters + (Op::FP32 ? 3 : 1), npq);
        atomicAdd(out.counters + (Op::FP32 ? 5 : 4), nbv);
        if (Op::FP32) atomicAdd(out.counters + 2, nq);
    }
}

// Launch of a kernel over warp units (tile, chunk, split) with at most gmax
// CTAs of nw workers (warps, or teams of threads / 32 warps), which take groups of
// up to kets ket pairs.  Tiles are
// cut into chunks of whole groups until every warp has 32 units (with 4, the
// heaviest units left (pp|pp) SMs idle 57 % of the time on a 1/16 shard of the
// 32-atom workload; 8 instead of 32 cost the fp32 lists of a 1/8 shard 7 %),
// into smaller ones while it has fewer than 4, down to single quartets, and
// then along the bra primitive pairs (which repeats the density transform).
template <typename K>
cudaError_t launch_warp_units(K kern, int nw, int threads, size_t per_warp, int kets, long long gmax, cudaStream_t st,
                              const MolDesc *mols, ClassLaunch cl, const OutArgs &out, const double *boys)
{
    int dev = 0, nsm = 1, per = 1;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    const size_t sm = per_warp * nw;
    if ((e = allow_cta_smem(kern, sm)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads * nw, sm)) != cudaSuccess) return e;
    if (gmax > (long long)(per > 0 ? per : 1) * nsm) gmax = (long long)(per > 0 ? per : 1) * nsm;
    cl.nchunk = 1;
    cl.nsplit = 1;
    const long long warps = gmax * nw;
    while (cl.ntiles * cl.nchunk < 32 * warps && cl.nchunk * kets < TILE) cl.nchunk *= 2;
    while (cl.ntiles * cl.nchunk < 4 * warps && cl.nchunk < TILE) cl.nchunk *= 2;
    if (!out.dump) {
        while (cl.ntiles * cl.nchunk * cl.nsplit < 4 * warps && cl.nsplit < 32) ++cl.nsplit;
        if (cl.split_req > 0) cl.nsplit = cl.split_req;
    }
    const long long units = cl.ntiles * cl.nchunk * cl.nsplit;
    const int grid = (int)(units < gmax ? units : gmax);
    if (units < grid * (long long)nw) nw = (int)((units + grid - 1) / grid);
    kern<<<grid, threads * nw, per_warp * nw, st>>>(mols, cl, out, boys);
    return cudaGetLastError();
}

// Launch of a gradient kernel with at most gcap slabs (8 an SM) of partial
// gradients.  Each worker's gradient lies beside its arrays while that leaves an SM
// three quarters of the workers that fit without it (or of the 8 there are slabs
// for), else every worker adds to a slab of its own: 36 KB a warp at 1500 atoms
// left the fp32 kernels 4 of 8 warps.
template <class Op>
cudaError_t launch_lanes(int gcap, cudaStream_t st, const MolDesc *mols, const ClassLaunch &cl, const OutArgs &out,
                         const double *boys)
{
    constexpr size_t bytes = Op::Lay::BYTES;
    static_assert(bytes <= kCtaSmem, "one warp's arrays fit in a CTA");
    OutArgs o = out;
    const size_t grad = sizeof(double) * 3 * (size_t)o.natom_total;
    const int fit = (int)(kCtaSmem / bytes), fit_g = (int)(kCtaSmem / (bytes + grad));
    o.use_smem = 4 * fit_g >= 3 * (fit < 8 ? fit : 8);
    const int have = o.use_smem ? fit_g : fit, nw = have < Op::cta_workers ? have : Op::cta_workers;
    return launch_warp_units(k_grad_lanes<Op>, nw, 32 * Op::NW, bytes + (o.use_smem ? grad : 0), Op::KQ,
                             o.use_smem ? gcap : (gcap > nw ? gcap / nw : 1), st, mols, cl, o, boys);
}

}  // namespace tg
